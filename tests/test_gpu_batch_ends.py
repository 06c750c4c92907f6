"""One-step launches on inputs that start and end inside a 16-byte unit, on the pipelined kernel: against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2205_05248_b200 import binding, workloads
from referee import RTOL, check_near_ties, near_tie_rows_allowed, row_rel_err

pytestmark = pytest.mark.gpu

# Small batches go to the split-operand kernel: these have more rows than 148 tiles of 128, and one a single tile a block.  Rows of 55
# and 31 observations take the word-by-word path (any float is a start), of 24 only the availability may start and end
# anywhere; 17 actions take the 32-column kernel; one to four environments in the last chunk; availability blocks of 24
# bytes.
SHAPES = [dict(E=3785, n=5, D=55, A=12), dict(E=3787, n=5, D=31, A=17), dict(E=3786, n=5, D=24, A=11), dict(E=4811, n=4, D=9, A=6),
          dict(E=1931, n=5, D=55, A=12)]


def _at(v, offset):
    """The same tensor, starting `offset` elements behind a 16-byte boundary, at the very end of its allocation."""
    buf = torch.empty(offset + v.numel(), dtype=v.dtype, device=v.device)
    out = buf[offset:].view(v.shape)
    out.copy_(v)
    return out


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["step", "subset", "lagged"])
def test_inputs_that_start_and_end_anywhere(kind, shape):
    cfg = workloads.small_config(**{**dict(H=64, L=3, T=6, precision="bf16", env=dict(done_thresh24=1 << 21)), **shape, "C": 2 * shape["E"]})
    E, n, A, T = cfg["E"], cfg["n"], cfg["A"], cfg["T"]
    w = workloads.make_weights(cfg)
    actor = binding.Actor(cfg)
    actor.set_weights(w)
    d_in = actor.env_generate(cfg["env"], 0, T)
    h_in = [v.cpu().numpy() for v in d_in]
    g_acts, g_q = actor.set_trace(T, want_q=True)
    sess = oracle.Session(cfg, w, np.arange(E))
    rng = np.random.default_rng(5)
    eps, near, greedy = 0.15, 0, 0
    for t in range(T):
        M = E if kind == "step" else E - t  # lists of every length modulo four
        ids = np.arange(E) if kind == "step" else rng.permutation(E)[:M].astype(np.int32)
        x = [v[t, :M].contiguous() for v in d_in]
        x[0], x[1] = _at(x[0], t % 4 if cfg["D"] % 8 else 0), _at(x[1], (0, 1, 7, 15, 16, 3)[t])
        act = (actor.step(*x, eps) if kind == "step" else actor.step_subset(ids, *x, eps) if kind == "subset" else actor.step_lagged(ids, *x, eps)).cpu().numpy()
        assert actor.step_kernel == "actor_tcp_kernel"
        q = g_q[t][torch.as_tensor(ids, device=g_q.device, dtype=torch.long)].cpu().numpy()
        _, tr = (sess.step_lagged if kind == "lagged" else sess.step_subset)(ids, *[v[t, :M] for v in h_in], eps, adopt=act, trace=("q", "action_free", "explore"))
        err = row_rel_err(q, tr["q"])
        assert err.max() <= RTOL["bf16"]
        diff = np.argwhere(tr["action_free"][None] != act[None])
        check_near_ties(diff, tr["q"][None], q[None], tr["action_free"][None], act[None], tr["explore"][None])
        near, greedy = near + len(diff), greedy + int((tr["explore"] == 0).sum())
    assert near <= near_tie_rows_allowed("bf16", greedy), (near, greedy)
    st, rv = actor.get_state(), actor.ring_view()
    for k in ("last_action", "slot", "pos", "ep_count"):
        assert np.array_equal(st[k].cpu().numpy(), getattr(sess, k)), k
    assert row_rel_err(st["h"].cpu().numpy(), sess.h).max() <= RTOL["bf16"]
    for k in ("slot_epid", "slot_len", "slot_complete"):
        assert np.array_equal(rv[k].cpu().numpy(), sess.ring[k]), k
    written = np.arange(cfg["L"])[None, :] < sess.ring["slot_len"][:, None]
    for k in ("obs", "avail", "action", "reward", "done"):
        assert np.array_equal(rv[k].cpu().numpy()[written], sess.ring[k][written]), k
    assert row_rel_err(rv["q"].cpu().numpy()[written], sess.ring["q"][written]).max() <= RTOL["bf16"]
    assert actor.status()[0] == 0
    actor.destroy()


@pytest.mark.parametrize("kind", ["step", "lagged"])
def test_staging_slots_that_held_the_ends_of_an_array(kind):
    """Four tiles a block: the slots that held an array's first and last bytes, which no bulk copy brings, are filled again by bulk
    copies.  Where the arrays start changes which bytes those are and nothing else."""
    cfg = workloads.small_config(H=64, L=4, T=4, precision="bf16", env=dict(done_thresh24=1 << 21), E=11999, n=5, D=55, A=12, C=11999)
    ids = np.random.default_rng(3).permutation(cfg["E"]).astype(np.int32)
    got = []
    for offset in (1, 2, 3):
        a = binding.Actor(cfg)
        a.set_weights(workloads.make_weights(cfg))
        x = a.env_generate(cfg["env"], 0, cfg["T"])
        for t in range(cfg["T"]):
            inputs = [_at(v[t], o) for v, o in zip(x, (offset, 5 * offset, 0, 0))]
            a.step(*inputs, 0.1) if kind == "step" else a.step_lagged(ids, *inputs, 0.1)
            assert a.step_kernel == "actor_tcp_kernel"
        torch.cuda.synchronize()
        assert a.status()[0] == 0
        got.append((a.get_state()["h"].clone(), a.ring_mem.clone()))
        a.destroy()
    for h, ring in got[1:]:
        assert torch.equal(h, got[0][0]) and torch.equal(ring, got[0][1])


def _pair(shape):
    cfg = workloads.small_config(**{**dict(H=64, L=4, T=7, precision="bf16", env=dict(done_thresh24=1 << 21)), **shape, "C": 2 * shape["E"]})
    actors = [binding.Actor(cfg) for _ in range(2)]
    for a in actors:
        a.set_weights(workloads.make_weights(cfg))
    return cfg, actors, actors[0].env_generate(cfg["env"], 0, cfg["T"])


def _same(one, two):
    torch.cuda.synchronize()
    s, u = one.get_state(), two.get_state()
    for k in ("h", "last_action", "slot", "pos", "ep_count"):
        assert torch.equal(s[k], u[k]), k
    assert torch.equal(one.ring_mem, two.ring_mem)
    for a in (one, two):
        assert a.status()[0] == 0
        a.destroy()


@pytest.mark.parametrize("shape", SHAPES[:3])
def test_pinned_host_arrays_of_a_batch_that_ends_anywhere(shape):
    """A host step that reads the caller's pinned arrays in place: what the step on device arrays gives."""
    cfg, (dev, pin), x = _pair(shape)
    for t in range(cfg["T"]):
        want = dev.step(*[v[t] if v[t].data_ptr() % 16 == 0 else _at(v[t], 0) for v in x], 0.15)
        got = pin.step_host(*[v[t].cpu().pin_memory() for v in x], 0.15, torch.empty_like(want, device="cpu").pin_memory())
        assert torch.equal(got, want.cpu()), t
        assert dev.step_kernel == pin.step_kernel == "actor_tcp_kernel"
    _same(dev, pin)


@pytest.mark.parametrize("kind", ["step", "subset", "lagged"])
def test_captured_steps_on_inputs_that_start_anywhere(kind):
    """Two steps in one graph, replayed: what the same steps give one by one.  (Nothing explores: the draws of a replay are those
    of its capture.)"""
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        cfg, (cap, ref), x = _pair(SHAPES[0])
        E, n = cfg["E"], cfg["n"]
        inputs = [[_at(v[t], o) for v, o in zip(x, (t % 4, t, 0, 0))] for t in range(cfg["T"])]
        lists = [np.random.default_rng(t).permutation(E).astype(np.int32) for t in range(cfg["T"])]
        out = [torch.empty((E, n), dtype=torch.int32, device="cuda") for _ in range(cfg["T"])]
        torch.cuda.synchronize()

        def call(a, t, to=None):
            if kind == "step":
                return a.step(*inputs[t], 0.0, to)
            return a.step_subset(lists[t], *inputs[t], 0.0, lagged=kind == "lagged", actions_out=to)
        call(cap, 0)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            for t in (1, 2):
                call(cap, t, out[t])
            assert cap.step_kernel == "actor_tcp_kernel"
        graph.replay()
        out[3] = call(cap, 3)
        want = [call(ref, t) for t in range(4)]
        torch.cuda.synchronize()
        assert all(torch.equal(out[t], want[t]) for t in (1, 2, 3))
        _same(cap, ref)
    graph.reset()


@pytest.mark.parametrize("kind", ["step", "subset", "lagged"])
def test_a_published_network_on_inputs_that_start_anywhere(kind):
    """A network published for step 3 is the one that steps 3 and later use, as if it had been loaded there."""
    cfg, (pub, ref), x = _pair(SHAPES[1])
    new = workloads.make_weights(cfg, seed=977)
    ids = np.random.default_rng(1).permutation(cfg["E"]).astype(np.int32)
    for t in range(cfg["T"]):
        if t == 1:
            pub.publish_weights(new, version=2, effective_step=3)
        if t == 3:
            ref.set_weights(new, version=2)
        inputs = [_at(v[t], o) for v, o in zip(x, (1 + t % 3, 2 * t + 1, 0, 0))]
        a, b = (m.step(*inputs, 0.15) if kind == "step" else m.step_subset(ids, *inputs, 0.15, lagged=kind == "lagged") for m in (pub, ref))
        assert torch.equal(a, b), t
        assert pub.step_kernel == ref.step_kernel == "actor_tcp_kernel"
    assert pub.weights_version == ref.weights_version == 2
    _same(pub, ref)
