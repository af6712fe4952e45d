"""Calls captured in a caller's own CUDA graph: their launches keep plain
dependencies and a long Yee call gathers from the planes, with the results of
the same calls made directly (overlapping launches, binned gather, sorted)."""
import numpy as np
import pytest

from paper_1409_5574_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1409_5574_gb300 import prad


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    prad.load_library()


def _case(kind):
    if kind.startswith("wave"):
        wl = W.plane_wave(a0=350.0, n=3001, seed=8)
        return wl, 9, 1 if kind == "wave_one_step" else 4, {}, False
    rng = np.random.default_rng(4)
    wl = W.yee2d(n_grid=64, slab=32, n_particles=524_303, seed=4, with_grid=False)
    wl.yee = W.yee_planes(128, 96, 250.0, 2 * np.pi / 32, rng)
    return wl, 8, 8, dict(sort_interval=4) if kind == "yee_sorted" else {}, kind == "yee_sorted"


@pytest.mark.parametrize("kind", ["wave_one_step", "wave_fused", "yee", "yee_sorted"])
def test_captured_call_equals_direct(kind):
    wl, steps, spl, kw, pid = _case(kind)
    got = []
    for captured in (False, True):
        stream = torch.cuda.Stream()
        ctx = prad.Context(wl.problem_kwargs(), photon_capacity=1 << 21, max_particles=wl.n,
                           steps_per_launch=spl, stream=stream, **kw)
        st = ctx.to_device(wl.state, with_pid=pid)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            ctx.push_emit(st, steps)  # (scratch and kernels in place before a capture)
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                ctx.push_emit(st, steps, t0=steps)
            with torch.cuda.stream(stream):
                g.replay()
        else:
            with torch.cuda.stream(stream):
                ctx.push_emit(st, steps, t0=steps)
        torch.cuda.synchronize()
        stats = ctx.energy_budget()[2]
        le, ll = ctx.ledger()
        order = torch.argsort(st["pid"]) if pid else slice(None)
        got.append(({k: v[order].cpu().numpy() for k, v in st.items()}, le.cpu().numpy(),
                    ll.cpu().numpy(), stats))
        ctx.close()
    a, b = got
    for k in a[0]:
        np.testing.assert_array_equal(a[0][k], b[0][k], err_msg=k)
    np.testing.assert_allclose(a[1], b[1], rtol=1e-13, atol=0)
    np.testing.assert_allclose(a[2], b[2], rtol=1e-13, atol=0)
    assert a[3] == b[3] and a[3]["records"] > 100
