"""Scratch of long Yee calls in the caller's order: taking it leaves another
stream's capture intact, it can be taken before a time loop, and a caller can
do without it."""
import numpy as np
import pytest

from paper_1409_5574_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1409_5574_gb300 import prad

N, STEPS = 524_301, 8


@pytest.fixture(scope="module")
def wl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.yee2d(n_grid=64, slab=32, n_particles=2 * N, seed=6, with_grid=False)
    dxn = 2 * np.pi / 32
    rng = np.random.default_rng(6)
    w.yee = W.yee_planes(120, 180, 250.0, dxn, rng)
    w.state["x"] = rng.uniform(0, 120, w.n) * dxn
    w.state["y"] = rng.uniform(0, 180, w.n) * dxn
    return w


def _ctx(wl, **kw):
    ctx = prad.Context(wl.problem_kwargs(), photon_capacity=1 << 22, max_particles=wl.n,
                       steps_per_launch=STEPS, **kw)
    st = ctx.to_device(wl.state)
    torch.cuda.synchronize()
    return ctx, st


def _push(ctx, st, n, t0=0):
    ctx.push_emit({k: v[:n] for k, v in st.items()}, STEPS, t0=t0)


def test_first_long_call_leaves_another_capture_intact(wl):
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    a = torch.zeros(1000, device="cuda")
    ctx, st = _ctx(wl, stream=own)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(other):
        a.add_(1.0)
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=other, capture_error_mode="global"):
        a.add_(1.0)
        _push(ctx, st, N)
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert a.eq(2.0).all()
    assert ctx.energy_budget()[2]["records"] > 100
    ctx.close()


def test_reserved_scratch_and_none(wl):
    _push(*_ctx(wl), N)  # (the kernels are loaded)
    torch.cuda.synchronize()
    got = []
    for on in (True, False):
        ctx, st = _ctx(wl)
        ctx.reserve_binning(True)
        held = torch.cuda.mem_get_info()[0]
        if not on:
            ctx.reserve_binning(False)
            assert torch.cuda.mem_get_info()[0] >= held + 44 * wl.n
            held = torch.cuda.mem_get_info()[0]
        for k, n in enumerate((N, N + 1, N + 77_000, 2 * N)):  # (no call allocates)
            _push(ctx, st, n, t0=k * STEPS)
            assert torch.cuda.mem_get_info()[0] == held
        got.append(({k: v.cpu().numpy() for k, v in st.items()}, ctx.energy_budget()))
        ctx.close()
    for k in got[0][0]:
        np.testing.assert_array_equal(got[0][0][k], got[1][0][k], err_msg=k)
    assert got[0][1][2] == got[1][1][2] and got[0][1][2]["records"] > 100
    np.testing.assert_allclose(got[0][1][:2], got[1][1][:2], rtol=1e-13)


def test_reserving_needs_a_yee_grid(wl):
    ctx = prad.Context(dict(wl.problem_kwargs(), field_kind=prad.PRAD_FIELD_CONST), max_particles=64,
                       photon_capacity=64)
    with pytest.raises(prad.PradError) as e:
        ctx.reserve_binning()
    assert e.value.code == prad.PRAD_ERR_STATE
    ctx.reserve_binning(False)
    ctx.close()
