"""Infinite biases and biases beyond the largest finite bf16 value on the bf16 kernels: what the CUDA-core kernel makes of them."""
import numpy as np
import pytest
import torch

from paper_2205_05248_b200 import binding, workloads
from referee import RTOL
from test_gpu_batch_ends import _at

pytestmark = pytest.mark.gpu

MAX = np.finfo(np.float32).max
# 16-byte boundaries: inputs and batches off them on the pipelined kernel (word-by-word rows; 32 output columns; availability
# alone), whole ones there, and a batch that the one-tile kernel takes
SHAPES = {"rows": dict(E=3785, n=5, D=55, A=12), "wide": dict(E=3787, n=5, D=31, A=17), "avail": dict(E=3786, n=5, D=24, A=11),
          "whole": dict(E=40, n=8, D=80, A=14), "one tile": dict(E=41, n=5, D=24, A=11)}
KINDS = [("rows", "step", 1), ("rows", "step", 0), ("rows", "subset", 1), ("rows", "lagged", 0), ("wide", "step", 3), ("wide", "lagged", 1), ("avail", "step", 0),
         ("avail", "subset", 0), ("whole", "step", 0), ("whole", "lagged", 0), ("one tile", "step", 0)]


def _weights(cfg, net):
    w, H = {k: v.copy() for k, v in workloads.make_weights(cfg).items()}, cfg["H"]
    if net == "output":
        w["b2"][[1, 2, 4]] = -np.inf, -MAX, MAX
    elif net == "gates":                       # reset, update, candidate: infinities and largest values on units of their own
        for g in range(3):
            w["b_ih"][g * H + 4 * g:g * H + 4 * g + 4] = np.inf, -np.inf, MAX, -MAX
        w["b_hh"][2 * H + 20:2 * H + 24] = np.inf, -np.inf, MAX, -MAX
    else:                                      # one unit of fc1 infinite (the operand of the largest value is), the rest of them shut
        w["b1"][[3, 5, 6]] = np.inf if net == "fc1" else MAX, -np.inf, -MAX
    return w


@pytest.mark.parametrize("net", ["output", "gates", "fc1", "fc1 largest"])
@pytest.mark.parametrize("shape,kind,offset", KINDS)
def test_infinite_and_largest_biases(shape, kind, offset, net):
    cfg = workloads.small_config(**{**dict(H=64, L=4, T=3, precision="bf16", env=dict(done_thresh24=1 << 21)), **SHAPES[shape], "C": 2 * SHAPES[shape]["E"]})
    E, T = cfg["E"], cfg["T"]
    w = _weights(cfg, net)
    got = {}
    for kernel in ("auto", "ffma"):
        a = binding.Actor(cfg, kernel=kernel)
        a.set_weights(w)
        acts, q = a.set_trace(T, want_q=True)
        inputs = a.env_generate(cfg["env"], 0, T)
        ids = np.random.default_rng(2).permutation(E).astype(np.int32)
        for t in range(T):
            x = [v[t].contiguous() for v in inputs]
            x[0], x[1] = _at(x[0], offset), _at(x[1], offset or (5 if shape == "avail" and kind == "subset" else 0))
            eps = 1.0 if t < T - 1 else 0.0    # (drawn actions keep both on one course; the last step chooses)
            a.step(*x, eps) if kind == "step" else a.step_subset(ids, *x, eps) if kind == "subset" else a.step_lagged(ids, *x, eps)
        assert a.status()[0] == 0
        if kernel == "auto":
            assert a.step_kernel == ("actor_tc_kernel" if shape == "one tile" else "actor_tcp_kernel")
        rv = a.ring_view()
        written = torch.arange(cfg["L"], device=q.device)[None, :] < rv["slot_len"][:, None]
        got[kernel] = [v.cpu() for v in (acts, q, a.get_state()["h"], rv["q"][written], rv["slot_len"])]
        a.destroy()
    (acts, q, h, rq, sl), (acts_f, q_f, h_f, rq_f, sl_f) = got["auto"], got["ffma"]
    assert torch.equal(sl, sl_f)
    for x, y in ((q, q_f), (h, h_f), (rq, rq_f)):
        assert torch.equal(x.isnan(), y.isnan())
        assert torch.equal(x[y.isinf()], y[y.isinf()]) and not x[~y.isinf()].isinf().any()
        x, y = torch.where(y.isfinite(), x, 0.0).double(), torch.where(y.isfinite(), y, 0.0).double()
        big = y.abs() > 1e30
        assert bool(((x - y).abs() <= 1e-5 * y.abs())[big].all())
        x, y = torch.where(big, 0.0, x), torch.where(big, 0.0, y)
        assert bool(((x - y).abs() <= RTOL["bf16"] * y.abs().amax(-1, keepdim=True).clamp(min=1e-3)).all())
    # the choice of the last step: the same, or a near-tie of the two kernels' values
    differ = torch.nonzero(acts[-1] != acts_f[-1])
    for e, i in differ.tolist():
        row, tol = q_f[-1, e, i], RTOL["bf16"] * float(torch.where(q_f[-1, e, i].abs() < 1e30, q_f[-1, e, i], 0.0).abs().max())
        assert abs(float(row[acts[-1, e, i]] - row[acts_f[-1, e, i]])) <= 1e-4 + 2 * tol
    assert torch.equal(acts[:-1], acts_f[:-1])
