"""Launches of a few steps on the pipelined kernel, several tiles a block: the same results as one long launch."""
import numpy as np
import pytest
import torch

from paper_2205_05248_b200 import binding, workloads

pytestmark = pytest.mark.gpu


# tiles of 128 rows on 148 blocks: two and three tiles a block, a ragged last tile; observation rows and availability blocks
# that are no 16-byte multiples; 32 output columns
@pytest.mark.parametrize("shape", [dict(E=5001, n=8, D=80, A=14), dict(E=9008, n=5, D=24, A=11), dict(E=8000, n=5, D=55, A=12),
                                   dict(E=4744, n=4, D=16, A=20)])
def test_short_launches_equal_a_long_one(shape):
    cfg = workloads.small_config(**{**dict(H=64, L=5, T=22, precision="bf16", env=dict(done_thresh24=1 << 21)), **shape, "C": 2 * shape["E"]})
    w = workloads.make_weights(cfg)
    long, short = binding.Actor(cfg), binding.Actor(cfg)
    staged = long.env_generate(cfg["env"], 0, cfg["T"])
    for a in (long, short):
        a.set_weights(w)
    long.rollout_staged(*staged, cfg["T"], 0.2)
    t = 0
    for part in (1, 2, 7, 3, 1, 1, 6, 1):
        short.rollout_staged(*[x[t:t + part] for x in staged], part, 0.2)
        t += part
    assert t == cfg["T"] and long.step_kernel == short.step_kernel == "actor_tcp_kernel"
    torch.cuda.synchronize()
    s, u, rs, ru = long.get_state(), short.get_state(), long.ring_view(), short.ring_view()
    for k in ("h", "last_action", "slot", "pos", "ep_count"):
        assert torch.equal(s[k], u[k]), k
    written = torch.arange(cfg["L"], device=s["h"].device)[None, :] < rs["slot_len"][:, None]
    for k in ("slot_epid", "slot_len", "slot_complete"):
        assert torch.equal(rs[k], ru[k]), k
    for k in ("obs", "avail", "action", "q", "reward", "done"):
        assert torch.equal(rs[k][written], ru[k][written]), k
    assert long.status() == short.status() and long.status()[0] == 0
    long.destroy()
    short.destroy()


def test_lists_of_several_tiles_a_block_equal_full_steps():
    """A shuffled list of every environment gives what the dense step gives, outcomes at once or a call later."""
    cfg = workloads.small_config(E=6004, n=8, D=24, A=10, H=64, C=12008, L=4, T=6, precision="bf16", env=dict(done_thresh24=1 << 21))
    w = workloads.make_weights(cfg)
    actors = [binding.Actor(cfg) for _ in range(3)]
    for a in actors:
        a.set_weights(w)
    dense, listed, late = actors
    obs, avail, rew, done = dense.env_generate(cfg["env"], 0, cfg["T"])
    rng = np.random.default_rng(3)
    for t in range(cfg["T"]):
        ids = rng.permutation(cfg["E"]).astype(np.int32)
        sel = torch.as_tensor(ids, device=obs.device, dtype=torch.long)
        a = dense.step(obs[t], avail[t], rew[t], done[t], 0.2)
        b = listed.step_subset(ids, obs[t][sel], avail[t][sel], rew[t][sel], done[t][sel], 0.2)
        prev = max(t - 1, 0)
        c = late.step_lagged(ids, obs[t][sel], avail[t][sel], rew[prev][sel], done[prev][sel], 0.2)
        assert torch.equal(a[sel], b) and torch.equal(a[sel], c), t
    assert all(x.step_kernel == "actor_tcp_kernel" for x in actors)
    s, u, v = dense.get_state(), listed.get_state(), late.get_state()
    rd, rl, rt = dense.ring_view(), listed.ring_view(), late.ring_view()
    for k in ("h", "last_action", "slot", "pos", "ep_count"):
        assert torch.equal(s[k], u[k]), k
    written = torch.arange(cfg["L"], device=obs.device)[None, :] < rd["slot_len"][:, None]
    for k in ("slot_epid", "slot_len", "slot_complete"):
        assert torch.equal(rd[k], rl[k]), k
    for k in ("obs", "avail", "action", "q", "reward", "done"):
        assert torch.equal(rd[k][written], rl[k][written]), k
    # the late actor: everything but the outcome of its last step, which has not arrived
    going = s["pos"] > 0                                  # (the others' episodes end with that outcome)
    for k in ("h", "last_action", "slot", "pos", "ep_count"):
        assert torch.equal(s[k][going], v[k][going]), k
    assert torch.equal(rd["slot_len"], rt["slot_len"]) and torch.equal(rd["slot_epid"], rt["slot_epid"])
    ends = torch.zeros_like(rd["slot_complete"])
    ends[v["slot"][~going].long()] = 1
    assert torch.equal(rd["slot_complete"], rt["slot_complete"] | ends)
    for k in ("obs", "avail", "action", "q"):
        assert torch.equal(rd[k][written], rt[k][written]), k
    told = written.clone()
    told[v["slot"].long(), v["pos"].long() - 1] = False
    for k in ("reward", "done"):
        assert torch.equal(rd[k][told], rt[k][told]), k
    for a in actors:
        assert a.status()[0] == 0
        a.destroy()


# availability of a step that is no 16-byte multiple: one-step launches run here, longer ones on the one-tile kernel
@pytest.mark.parametrize("shape", [dict(E=3785, n=5, D=24, A=11), dict(E=2999, n=7, D=32, A=17)])
def test_one_step_launches_of_odd_batches_equal_a_long_one(shape):
    """A rollout of a batch that is no 16-byte multiple is the same however it is divided: state and choices bit by bit, Q up to the
    order of its sum."""
    cfg = workloads.small_config(**{**dict(H=64, L=5, T=14, precision="bf16", env=dict(done_thresh24=1 << 21)), **shape, "C": 2 * shape["E"]})
    w = workloads.make_weights(cfg)
    long, short = binding.Actor(cfg), binding.Actor(cfg)
    staged = long.env_generate(cfg["env"], 0, cfg["T"])
    for a in (long, short):
        a.set_weights(w)
    long.rollout_staged(*staged, cfg["T"], 1.0)
    t, kernels = 0, set()
    for part in (1, 1, 4, 1, 3, 1, 2, 1):
        short.rollout_staged(*[x[t:t + part].clone() for x in staged], part, 1.0)
        kernels.add((part == 1, short.step_kernel))
        t += part
    assert t == cfg["T"] and kernels == {(True, "actor_tcp_kernel"), (False, "actor_tc_kernel")} and long.step_kernel == "actor_tc_kernel"
    torch.cuda.synchronize()
    s, u, rs, ru = long.get_state(), short.get_state(), long.ring_view(), short.ring_view()
    for k in ("h", "last_action", "slot", "pos", "ep_count"):
        assert torch.equal(s[k], u[k]), k
    written = torch.arange(cfg["L"], device=s["h"].device)[None, :] < rs["slot_len"][:, None]
    for k in ("slot_epid", "slot_len", "slot_complete"):
        assert torch.equal(rs[k], ru[k]), k
    for k in ("obs", "avail", "action", "reward", "done"):
        assert torch.equal(rs[k][written], ru[k][written]), k
    # two orders of 67 terms: each is off by at most 66 roundings (or cuts, 2^-23) of partial sums that the terms' magnitudes bound
    bound = 2 * 66 * 2.0 ** -23 * float((np.abs(w["W2"]).sum(axis=1) + np.abs(w["b2"])).max())
    assert float((rs["q"][written] - ru["q"][written]).abs().max()) <= bound
    assert long.status() == short.status() and long.status()[0] == 0
    long.destroy()
    short.destroy()
