"""The split-operand tensor-core kernel (general path: fp32, per-type networks, launches and shapes the bf16 kernels do
not take) at the edges of its tiles, slices and dispatch, against the oracle."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2205_05248_b200 import binding, workloads
from referee import referee, run_gpu_rollout

pytestmark = pytest.mark.gpu


# A tile has 128 rows = n * environments; fc1 goes in K steps of 16 observations and, in bf16, slices of 96; 16 and 17
# actions lie on both sides of the width of the Q product; at hidden 128 the gate slices stream through the ring in fp32
# and stay (nearly) resident in bf16 with few observations.
@pytest.mark.parametrize("prec,H,shape", [
    ("fp32", 64, dict(E=8, n=3, D=30, A=9)),            # one environment per block
    ("fp32", 64, dict(E=300, n=1, D=1, A=1)),
    # 128 environments per tile, a ragged last tile.  (Nine actions: the referee's error is relative to the row's largest
    # |Q|, and with two of them it falls to about 1e-3 in one of 100,000 rows, where the rounding of 64 products of size
    # 0.1 - up to 64 * 0.1 * 2^-24 = 4e-7 - is beyond 1e-5 of it in any order of summation.)
    ("fp32", 64, dict(E=20000, n=1, D=17, A=9, L=4, T=5)),
    ("fp32", 64, dict(E=600, n=32, D=16, A=17, T=6)),   # four environments per tile, the wide Q product
    ("fp32", 64, dict(E=7, n=32, D=63, A=32)),
    ("fp32", 64, dict(E=2500, n=8, D=80, A=16, T=6)),   # full tiles, the largest observation
    ("fp32", 64, dict(E=331, n=5, D=64, A=11, C=662)),
    ("bf16", 64, dict(E=331, n=3, D=30, A=9, C=662)),   # fewer agents than the pipelined kernel takes, unaligned rows
    ("bf16", 64, dict(E=40, n=2, D=255, A=20)),         # three fc1 slices
    ("bf16", 64, dict(E=3000, n=3, D=31, A=16, T=6)),
    ("fp32", 128, dict(E=8, n=3, D=30, A=9)),
    ("fp32", 128, dict(E=2500, n=8, D=80, A=14, T=6)),
    ("fp32", 128, dict(E=40, n=5, D=96, A=16)),
    ("bf16", 128, dict(E=331, n=3, D=30, A=9, C=662)),
    ("bf16", 128, dict(E=1700, n=5, D=55, A=12, T=6)),
    ("bf16", 128, dict(E=40, n=4, D=200, A=20)),        # three fc1 slices, the wide Q product
])
def test_shapes(prec, H, shape):
    cfg = workloads.small_config(**{**dict(H=H, L=6, T=14, C=shape["E"], precision=prec), **shape})
    w = workloads.make_weights(cfg)
    T = cfg["T"]
    actor, acts, q = run_gpu_rollout(cfg, w, splits=[1, T - 1], work_steps=T)
    res = referee(cfg, w, actor, acts, q)
    assert res["kernel"] == "ffma"          # the general path's name
    assert actor.step_kernel == "actor_tcs_kernel"
    actor.destroy()


@pytest.mark.parametrize("H", [64, 128])
def test_precision_is_that_of_the_fma_chain(H):
    """fp32: the largest Q and hidden-state differences to the oracle are those of the CUDA-core kernel.  Both sum the same
    products; bound of one summation order against the other: twice the CUDA-core kernel's own largest difference."""
    cfg = dict(workloads.config(5, E=1024, H=H, precision="fp32"), T=16, C=1024)
    w = workloads.make_weights(cfg)
    err = {}
    for kernel in ("auto", "ffma"):
        actor, acts, q = run_gpu_rollout(cfg, w, kernel=kernel)
        res = referee(cfg, w, actor, acts, q)
        err[kernel] = (res["q_err"], res["h_err"])
        assert actor.step_kernel == {"auto": "actor_tcs_kernel", "ffma": "actor_ffma_kernel"}[kernel]
        actor.destroy()
    print(f"largest row-wise relative differences to the oracle (Q, h): {err}")
    assert err["auto"][0] <= 2 * err["ffma"][0] and err["auto"][1] <= 2 * err["ffma"][1]


@pytest.mark.parametrize("prec,H,shape,kernel", [
    ("fp32", 64, dict(n=3, D=97, A=9), "actor_ffma_kernel"), ("fp32", 64, dict(n=3, D=96, A=17), "actor_ffma_kernel"),
    ("fp32", 64, dict(n=3, D=96, A=16), "actor_tcs_kernel"), ("fp32", 128, dict(n=3, D=16, A=17), "actor_ffma_kernel"),
    ("fp32", 128, dict(n=3, D=97, A=9), "actor_ffma_kernel"), ("bf16", 128, dict(n=3, D=321, A=17), "actor_ffma_kernel"),
    ("bf16", 64, dict(n=3, D=30, A=9), "actor_tcs_kernel"), ("bf16", 64, dict(n=4, D=30, A=8), "actor_tcp_kernel"),
    ("bf16", 128, dict(n=8, D=80, A=14), "actor_tcs_kernel")])
def test_kernel_of_a_step(prec, H, shape, kernel):
    """Which kernel a dense step and a list step run on, at the edges of the shapes that the split-operand kernel takes."""
    cfg = workloads.small_config(H=H, E=8, C=8, L=4, precision=prec, **shape)
    a = binding.Actor(cfg)
    a.set_weights(workloads.make_weights(cfg))
    assert a.step_kernel == ""
    x = [v[0] for v in a.env_generate(cfg["env"], 0, 1)]
    a.step(*x, 0.1)
    assert a.step_kernel == kernel
    a.step_subset(np.arange(3), *[v[:3].contiguous() for v in x], 0.1)
    assert a.step_kernel == ("actor_tcs_kernel" if kernel == "actor_tcp_kernel" else kernel)   # (three environments: no whole chunk)
    a.destroy()


@pytest.mark.parametrize("D", [30, 32])
def test_observations_at_any_float_address(D):
    """Device inputs that start on a 4-byte boundary only give the same results as aligned ones."""
    cfg = workloads.small_config(H=64, E=50, n=3, D=D, A=9, C=50, L=5, precision="fp32")
    w = workloads.make_weights(cfg)
    a, b = (binding.Actor(cfg) for _ in range(2))
    for x in (a, b):
        x.set_weights(w)
    for t in range(7):
        obs, avail, reward, done = (v[0] for v in a.env_generate(cfg["env"], t, 1))
        shifted = torch.empty(obs.numel() + 1, device="cuda")[1:].view_as(obs).copy_(obs)
        av1 = torch.empty(avail.numel() + 1, dtype=torch.uint8, device="cuda")[1:].view_as(avail).copy_(avail)
        assert torch.equal(a.step(obs, avail, reward, done, 0.1), b.step(shifted, av1, reward, done, 0.1))
    assert torch.equal(a.ring_mem, b.ring_mem) and torch.equal(a.get_state()["h"], b.get_state()["h"])
    a.destroy()
    b.destroy()


@pytest.mark.parametrize("H", [64, 128])
def test_types_without_agents_and_one_agent_per_type(H):
    """A unit type that no agent has, and a team of one agent per type: every environment refereed."""
    for n, types in ((3, [0, 0, 2]), (4, [3, 2, 1, 0])):
        cfg = workloads.small_config(H=H, E=1500, n=n, D=13, A=6, C=3000, L=4, T=9, precision="fp32")
        cfg["agent_type"] = types
        ws = [workloads.make_weights(cfg, seed=100 + k) for k in range(max(types) + 1)]
        actor, acts, q = run_gpu_rollout(cfg, ws, splits=[2, 7])
        referee(cfg, ws, actor, acts, q)
        actor.destroy()


@pytest.mark.parametrize("over", [dict(), dict(precision="fp32"), dict(n=3, A=9, D=30), dict(E=2300, D=240, precision="fp32")])
def test_host_step_on_pinned_and_pageable_arrays(over):
    """Pinned arrays are read by the step kernel, pageable ones copied, large observations (here 2300 x 8 x 240 floats, 17.7
    MB) always copied: the same actions, records and state as the step on device arrays."""
    cfg = workloads.small_config(**{**dict(H=64, E=70, n=8, D=80, A=14, L=5, precision="bf16"), **over})
    cfg["C"] = cfg["E"]
    w = workloads.make_weights(cfg)
    dev, pin, page = (binding.Actor(cfg) for _ in range(3))
    for a in (dev, pin, page):
        a.set_weights(w)
    for t in range(7):
        x = [v[0] for v in dev.env_generate(cfg["env"], t, 1)]
        want = dev.step(*x, 0.1).cpu()
        h = [v.cpu() for v in x]
        assert torch.equal(page.step_host(*h, 0.1, torch.empty_like(want)), want)
        out = torch.empty_like(want).pin_memory() if t % 2 else torch.empty_like(want)
        assert torch.equal(pin.step_host(*[v.pin_memory() for v in h], 0.1, out), want)
    for a in (pin, page):
        assert torch.equal(a.ring_mem, dev.ring_mem) and torch.equal(a.get_state()["h"], dev.get_state()["h"])
        assert a.status()[0] == 0
        a.destroy()
    dev.destroy()


@pytest.mark.parametrize("prec,H,T", [("fp32", 64, 240_000), ("bf16", 128, 300_000)])
def test_launch_behind_a_long_one(prec, H, T):
    """A launch that starts beside its predecessor while that still runs for longer than a bounded wait lasts (about a
    second): the wait for the predecessor counts against none of its own waits."""
    cfg = workloads.small_config(H=H, E=1, n=4, D=8, A=4, C=2, L=50, precision=prec, seed=5)
    w = workloads.make_weights(cfg)
    # steps for a first launch of 1.5 s, whatever a step takes: timed over a twelfth of T, the second of two launches
    a = binding.Actor(cfg, work_steps=1)
    a.set_weights(w)
    probe = a.env_generate(cfg["env"], 0, T // 12)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    for e in ev[:2]:
        e.record()
        a.rollout_staged(*probe, T // 12, 0.2)
    ev[2].record()
    torch.cuda.synchronize()
    a.destroy()
    T = max(T, int(1500.0 / ev[1].elapsed_time(ev[2]) * (T // 12)))
    states = []
    for together in (True, False):
        a = binding.Actor(cfg, work_steps=1)
        a.set_weights(w)
        staged = a.env_generate(cfg["env"], 0, T)
        short = a.env_generate(cfg["env"], T, 40)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        ev[0].record()
        a.rollout_staged(*staged, T, 0.2)
        if not together:
            torch.cuda.synchronize()
        a.rollout_staged(*short, 40, 0.2)
        ev[1].record()
        torch.cuda.synchronize()
        assert ev[0].elapsed_time(ev[1]) > 1200.0, "the first launch is too short for what is tested"
        status, counters = a.status()
        assert status == 0 and counters["agent_steps"] == 4 * (T + 40)
        states.append((a.get_state()["h"].clone(), a.ring_mem.clone()))
        a.destroy()
    assert all(torch.equal(x, y) for x, y in zip(*states))


@pytest.mark.parametrize("over,kernel", [(dict(), "auto"), (dict(precision="fp32"), "auto"), (dict(H=128), "auto"),
                                         (dict(n=5, D=55, A=12), "pipelined"), (dict(n=5, D=55, A=12, E=72), "pipelined")])
def test_host_step_on_pinned_arrays_at_any_address(over, kernel):
    """Pinned arrays that start where the kernels could not read them, or read them on another kernel, are copied: the same
    actions, records and state as the step on device arrays, whatever the addresses."""
    cfg = workloads.small_config(**{**dict(H=64, E=70, n=8, D=80, A=14, L=5, precision="bf16"), **over})
    cfg["C"] = cfg["E"]
    w = workloads.make_weights(cfg)
    dev, pin = (binding.Actor(cfg, kernel=kernel) for _ in range(2))
    for a in (dev, pin):
        a.set_weights(w)
    offsets = [(0, 0, 0, 0, 0), (16, 16, 4, 1, 4), (4, 0, 0, 0, 0), (0, 3, 0, 0, 0), (0, 0, 2, 0, 0), (0, 0, 0, 3, 2), (8, 8, 1, 1, 1)]
    for t, off in enumerate(offsets):
        x = [v[0] for v in dev.env_generate(cfg["env"], t, 1)]
        want = dev.step(*x, 0.1).cpu()
        host = [torch.empty(v.numel() * v.element_size() + 32, dtype=torch.uint8).pin_memory() for v in (*x, want)]
        for b, o, v in zip(host, off, x):
            b[o:o + v.numel() * v.element_size()] = v.cpu().contiguous().view(-1).view(torch.uint8)
        at = [C.c_void_p(b.data_ptr() + o) for b, o in zip(host, off)]
        binding._check(pin.lib.marl_actor_step_host(pin.handle, *at[:4], C.c_float(0.1), at[4]))
        got = host[4][off[4]:off[4] + want.numel() * 4].clone().view(torch.int32).view_as(want)
        assert torch.equal(got, want), off
    assert torch.equal(pin.ring_mem, dev.ring_mem) and torch.equal(pin.get_state()["h"], dev.get_state()["h"])
    for a in (pin, dev):
        assert a.status()[0] == 0
        a.destroy()


@pytest.mark.parametrize("shift", ["obs", "avail"])
def test_hidden_128_gates_of_unaligned_inputs_are_the_accurate_ones(shift):
    """bf16 at hidden 128: a dense step on inputs off a 16-byte boundary has the gate functions of the general path.  So it is,
    bit for bit, the step over the list of all environments, which always has them; the aligned dense step is not."""
    cfg = workloads.small_config(H=128, E=200, n=8, D=80, A=14, C=200, L=5, precision="bf16")
    w = workloads.make_weights(cfg)
    h = {}
    for how in ("aligned", "shifted", "list"):
        a = binding.Actor(cfg)
        a.set_weights(w)
        obs, avail, reward, done = (v[0] for v in a.env_generate(cfg["env"], 0, 1))
        if how == "shifted" and shift == "obs":
            obs = torch.empty(obs.numel() + 1, device="cuda")[1:].view_as(obs).copy_(obs)
        elif how == "shifted":
            avail = torch.empty(avail.numel() + 1, dtype=torch.uint8, device="cuda")[1:].view_as(avail).copy_(avail)
        if how == "list":
            a.step_subset(np.arange(200), obs, avail, reward, done, 0.1)
        else:
            a.step(obs, avail, reward, done, 0.1)
        torch.cuda.synchronize()
        h[how] = a.get_state()["h"].clone()
        assert a.status()[0] == 0
        a.destroy()
    assert torch.equal(h["shifted"], h["list"]) and not torch.equal(h["aligned"], h["list"])


@pytest.mark.parametrize("H", [64, 128])
@pytest.mark.parametrize("net", ["mixed", "one sign", "large weights"])
def test_infinite_and_very_large_values_fp32(H, net):
    """fp32: infinities, NaN and values beyond the largest finite bf16 (3.39e38) go through the network as on the CUDA-core
    kernel: the same infinities and NaN, other values to 1e-5, the same actions."""
    cfg = workloads.small_config(H=H, E=16, n=2, D=20, A=4, C=16, L=5, precision="fp32")
    w = {k: v.copy() for k, v in workloads.make_weights(cfg).items()}
    rng = np.random.default_rng(3)
    big = 3.4e38
    if net == "one sign":                      # every unit infinite, every gate's sum of one sign: h stays finite
        w["W1"][:, 0] = 0.3
        w["W_ih"][:H] = np.abs(w["W_ih"][:H]) + 0.01
        w["W_ih"][H:2 * H] = -np.abs(w["W_ih"][H:2 * H]) - 0.01
        w["W_ih"][2 * H:] = np.abs(w["W_ih"][2 * H:]) * rng.choice([-1.0, 1.0], size=(H, 1)).astype(np.float32)
    w["W1"][:, 1] *= 1e-3                      # (large observations: no overflow of a sum, whatever its order)
    if net == "large weights":
        w["W1"][3, 5] = np.inf
        w["W2"][1, 7] = big
        w["W2"][2, 9] = -np.inf
        w["W1"][4, 6] = -big
    got = {}
    for kernel in ("auto", "ffma"):
        a = binding.Actor(cfg, kernel=kernel)
        a.set_weights(w)
        acts, q = a.set_trace(2)
        for t in range(2):
            obs, avail, reward, done = (v[0] for v in a.env_generate(dict(cfg["env"], done_thresh24=0), t, 1))
            if net != "large weights":
                for e, (col, v) in enumerate([(0, np.inf), (0, -np.inf), (1, big), (1, -big), (1, 3.3895e38), (0, np.nan), (0, 1e30)]):
                    obs[e, 0, col] = v
            else:
                obs[:, :, 6] *= 1e-3
                obs[3, 1, 5] = 0.0
            a.step(obs, avail, reward, done, 0.0)
        torch.cuda.synchronize()
        got[kernel] = (acts.cpu(), q.double().cpu(), a.get_state()["h"].double().cpu())
        a.destroy()
    assert torch.equal(got["auto"][0], got["ffma"][0])
    # a Q value is bounded by its row of W2 (|h| <= 1): differences are measured against that
    scale = torch.as_tensor(np.maximum(np.abs(np.where(np.isfinite(w["W2"]), w["W2"], 0)).max(axis=1), 1.0)).double()
    for x, y, sc in ((got["auto"][1], got["ffma"][1], scale), (got["auto"][2], got["ffma"][2], torch.ones(H).double())):
        assert torch.equal(x.isnan(), y.isnan()) and torch.equal(x.isinf(), y.isinf())
        assert torch.equal(x[x.isinf()], y[y.isinf()])
        f = torch.isfinite(y)
        assert f.any()
        assert bool(((x - y).abs() <= 1e-5 * sc)[f].all())
    if net != "mixed":
        assert (~torch.isfinite(got["ffma"][1])).any() == (net == "large weights")
