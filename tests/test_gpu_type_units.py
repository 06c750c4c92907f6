"""Per-type networks where a block runs tiles of several unit types, one after the other: against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2205_05248_b200 import binding, workloads
from referee import RTOL, check_near_ties, near_tie_rows_allowed, referee, row_rel_err, run_gpu_rollout

pytestmark = pytest.mark.gpu


# 148 blocks: several tiles a block and type, a block with tiles of two types, fewer units than blocks
@pytest.mark.parametrize("prec,shape,types", [("fp32", dict(E=21000, n=5, D=8, A=6), [0, 1, 1, 0, 2]),
                                              ("bf16", dict(E=7001, n=3, D=6, A=5), [1, 0, 1]),
                                              ("fp32", dict(E=4999, n=4, D=9, A=5), [0, 1, 1, 0]),
                                              ("bf16", dict(E=4700, n=8, D=16, A=7, H=128), [0, 1, 0, 1, 1, 1, 0, 0]),
                                              ("fp32", dict(E=9, n=4, D=6, A=5), [3, 1, 0, 2])])
def test_tiles_of_all_types_are_dealt_to_the_blocks_together(prec, shape, types):
    cfg = workloads.typed(workloads.small_config(**{**dict(H=64, L=3, T=6, precision=prec), **shape, "C": 2 * shape["E"]}), agent_type=types)
    ws = [workloads.make_weights(cfg, seed=90 + k) for k in range(max(types) + 1)]
    actor, acts, q = run_gpu_rollout(cfg, ws, splits=[1, 2, 3])
    res = referee(cfg, ws, actor, acts, q)
    assert res["envs"] == cfg["E"]
    actor.destroy()


def test_cursors_advance_once_a_step_whatever_type_ends_last():
    """Cursors of a typed actor equal those of a shared network on the same outcomes, call after call, after a reset too."""
    cfg = workloads.typed(workloads.small_config(E=6000, n=4, D=8, A=5, H=64, C=12000, L=3, T=8), agent_type=[0, 1, 2, 0])
    ws = [workloads.make_weights(cfg, seed=5 + k) for k in range(3)]
    typed, shared = binding.Actor(cfg), binding.Actor(cfg)
    typed.set_weights_typed(ws)
    shared.set_weights(ws[0])
    for again in range(2):
        for part in (1, 3, 1, 2):
            for a in (typed, shared):
                a.rollout(cfg["env"], part, 1.0)
            torch.cuda.synchronize()
            s, t = shared.get_state(), typed.get_state()
            for k in ("slot", "pos", "ep_count"):
                assert torch.equal(s[k], t[k]), k
            for k in ("slot_epid", "slot_len", "slot_complete"):
                assert torch.equal(shared.ring_view()[k], typed.ring_view()[k]), k
        assert typed.status() == shared.status()
        for a in (typed, shared):
            a.reset()
    typed.destroy()
    shared.destroy()


@pytest.mark.parametrize("prec,shape,types", [("fp32", dict(E=9001, n=5, D=8, A=6), [0, 1, 1, 0, 2]), ("bf16", dict(E=7001, n=3, D=6, A=5), [1, 0, 1])])
def test_late_outcomes_where_a_block_runs_several_types(prec, shape, types):
    """List steps with late outcomes of per-type networks, several tiles and types a block: against the oracle."""
    cfg = workloads.typed(workloads.small_config(**{**dict(H=64, L=3, T=6, precision=prec, env=dict(done_thresh24=1 << 21)), **shape, "C": 2 * shape["E"]}), agent_type=types)
    ws = [workloads.make_weights(cfg, seed=40 + k) for k in range(max(types) + 1)]
    actor = binding.Actor(cfg)
    actor.set_weights_typed(ws)
    d_in = actor.env_generate(cfg["env"], 0, cfg["T"])
    h_in = [v.cpu().numpy() for v in d_in]
    g_acts, g_q = actor.set_trace(cfg["T"], want_q=True)
    sess = oracle.Session(cfg, ws, np.arange(cfg["E"]))
    rng = np.random.default_rng(5)
    near, greedy = 0, 0
    for t in range(cfg["T"]):
        M = cfg["E"] - 7 * t
        ids = rng.permutation(cfg["E"])[:M].astype(np.int32)
        act = actor.step_lagged(ids, *[v[t, :M].contiguous() for v in d_in], 0.15).cpu().numpy()
        q = g_q[t][torch.as_tensor(ids, device=g_q.device, dtype=torch.long)].cpu().numpy()
        _, tr = sess.step_lagged(ids, *[v[t, :M] for v in h_in], 0.15, adopt=act, trace=("q", "action_free", "explore"))
        assert row_rel_err(q, tr["q"]).max() <= RTOL[prec]
        diff = np.argwhere(tr["action_free"][None] != act[None])
        check_near_ties(diff, tr["q"][None], q[None], tr["action_free"][None], act[None], tr["explore"][None])
        near, greedy = near + len(diff), greedy + int((tr["explore"] == 0).sum())
    assert near <= near_tie_rows_allowed(prec, greedy), (near, greedy)
    st, rv = actor.get_state(), actor.ring_view()
    for k in ("last_action", "slot", "pos", "ep_count"):
        assert np.array_equal(st[k].cpu().numpy(), getattr(sess, k)), k
    assert row_rel_err(st["h"].cpu().numpy(), sess.h).max() <= RTOL[prec]
    for k in ("slot_epid", "slot_len", "slot_complete"):
        assert np.array_equal(rv[k].cpu().numpy(), sess.ring[k]), k
    written = np.arange(cfg["L"])[None, :] < sess.ring["slot_len"][:, None]
    for k in ("obs", "avail", "action", "reward", "done"):
        assert np.array_equal(rv[k].cpu().numpy()[written], sess.ring[k][written]), k
    assert row_rel_err(rv["q"].cpu().numpy()[written], sess.ring["q"][written]).max() <= RTOL[prec]
    assert actor.status()[0] == 0
    actor.destroy()
