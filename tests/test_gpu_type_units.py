"""Per-type networks where a block runs tiles of several unit types, one after the other: against the oracle."""
import numpy as np
import pytest
import torch

from paper_2205_05248_b200 import binding, workloads
from referee import referee, run_gpu_rollout

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
