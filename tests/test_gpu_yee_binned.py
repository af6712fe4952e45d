"""The Yee push of particles in the caller's own order: calls of several steps
gather through tiles and an order of the particles found on the device, calls
of one step gather from global memory.  The two take the same steps: state,
counters and photon records are the same bits, per-particle ledgers the same
up to the grouping of their FP64 adds."""
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


def _problem(nx, ny, n, seed, spread):
    """n electrons over the whole grid and past its seams (spread) or within
    40 x 40 cells of a corner, one of them not finite."""
    rng = np.random.default_rng(seed)
    dxn = 2 * np.pi / 32
    wl = W.yee2d(n_grid=64, slab=32, n_particles=n, seed=seed, with_grid=False)
    wl.yee = W.yee_planes(nx, ny, 250.0, dxn, rng)
    ex, ey = (nx, ny) if spread else (min(nx, 40), min(ny, 40))
    wl.state["x"] = rng.uniform(-0.5, ex + 0.5, n) * dxn
    wl.state["y"] = rng.uniform(-0.5, ey + 0.5, n) * dxn
    wl.state["uy"][n // 3] = np.nan
    return wl


def _run(wl, calls, per_launch, pid, **kw):
    off = 3
    ctx = prad.Context(wl.problem_kwargs(), photon_capacity=1 << 23, max_particles=wl.n + off,
                       steps_per_launch=per_launch, **kw)
    st = ctx.to_device(wl.state)
    if pid:  # ids in another order than the particles'
        st["pid"] = torch.as_tensor(np.random.default_rng(1).permutation(wl.n).astype(np.int32)
                                    + 7).cuda()
    t = 2
    for steps in calls:
        ctx.push_emit(st, steps, t0=t, pid0=7, ledger_offset=off)
        t += steps
    ph = ctx.photons(on_device=False)
    stats = ctx.energy_budget()[2]
    le, ll = ctx.ledger()
    rec = np.stack([ph[k].numpy().view(np.uint32) for k in
                    ("pid", "step", "x", "y", "z", "nx", "ny", "nz", "eps", "weight")], 1)
    out = ({k: v.cpu().numpy() for k, v in st.items()}, rec[np.lexsort(rec.T[::-1])],
           le.cpu().numpy(), ll.cpu().numpy(), {k: v for k, v in stats.items()
                                                if k != "spec_launches"})
    ctx.close()
    return out


@pytest.mark.parametrize("nx,ny,n,spread,steps,per_launch,pid,kw", [
    (130, 100, 524301, True, 8, 8, False, {}),         # tiles cut by the grid's end
    (130, 100, 306001, True, 55, 1, True, {}),         # binned twice, one step per launch
    (40, 300, 480007, True, 9, 4, False, {}),          # narrower than the staged region
    (37, 29, 70001, False, 60, 60, False, {}),         # one launch longer than the interval
    (4129, 4100, 524301, True, 8, 8, True, {}),        # sparse: the plain kernel stands in
    (4129, 4100, 524301, False, 8, 5, False, {}),      # more tiles than shared counters
    (256, 256, 524288, False, 8, 4, False, dict(n_try=2, select_prob=0.5)),
    (256, 250, 524301, False, 8, 8, True, dict(specialize=True)),
])
def test_binned_equals_plain(nx, ny, n, spread, steps, per_launch, pid, kw):
    wl = _problem(nx, ny, n, seed=nx + n, spread=spread)
    assert n * steps >= (1 << 22) and (per_launch >= 4 or n * steps >= (1 << 24))
    a = _run(wl, [1] * steps, 1, pid, **dict(kw, specialize=False))
    b = _run(wl, [steps], per_launch, pid, **kw)
    for k in a[0]:
        np.testing.assert_array_equal(a[0][k], b[0][k], err_msg=k)
    assert 100 < len(a[1]) < 1 << 23
    np.testing.assert_array_equal(a[1], b[1])
    np.testing.assert_allclose(a[2], b[2], rtol=1e-13, atol=0)
    np.testing.assert_allclose(a[3], b[3], rtol=1e-13, atol=0)
    a[4]["nan_frozen"] = b[4]["nan_frozen"] = min(a[4]["nan_frozen"], b[4]["nan_frozen"])
    assert a[4] == b[4] and a[4]["nan_frozen"] >= 1  # (counted per launch)
