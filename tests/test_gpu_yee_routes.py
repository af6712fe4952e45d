"""Long Yee calls by what their particles look like: which kernels run them is
decided by sizes and by counts on the device, and every route gives the steps
of the plain gather (calls of one step)."""
import numpy as np
import pytest

from paper_1409_5574_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1409_5574_gb300 import prad


def _problem(nx, ny, n, ex, ey, order=None, jitter=0.0):
    """n electrons over ex x ey cells in the middle of the grid, the last one not
    finite, in random order or in order of cells (moved by jitter after)."""
    rng = np.random.default_rng(nx + n)
    dxn = 2 * np.pi / 32
    wl = W.yee2d(n_grid=64, slab=32, n_particles=n, seed=n, with_grid=False)
    wl.yee = W.yee_planes(nx, ny, 200.0, dxn, rng)
    x, y = (nx - ex) / 2 + rng.uniform(0, ex, n), (ny - ey) / 2 + rng.uniform(0, ey, n)
    if order:
        by = np.lexsort((x, y.astype(int))) if order == "rows" else np.lexsort(
            (x.astype(int), y.astype(int), x.astype(int) // 32, y.astype(int) // 32))
        x, y = x[by], y[by]
        x += jitter * rng.standard_normal(n)
        y += jitter * rng.standard_normal(n)
    wl.state["x"], wl.state["y"] = x * dxn, y * dxn
    wl.state["ux"][n - 1] = np.inf
    return wl


def _run(wl, calls, per_launch, ids=False, ledger=False, **kw):
    problem = dict(wl.problem_kwargs())
    if ledger:
        problem["rr_mode"] = prad.PRAD_RR_LEDGER
    ctx = prad.Context(problem, photon_capacity=1 << 24, max_particles=wl.n + 5,
                       steps_per_launch=per_launch, **kw)
    st = ctx.to_device(wl.state)
    if ids:  # in another order than the particles
        order = np.random.default_rng(1).permutation(wl.n).astype(np.int32)
        st["pid"] = torch.as_tensor(order + 11).cuda()
    t = 0
    for steps in calls:
        ctx.push_emit(st, steps, t0=t, pid0=11 if ids else 0, ledger_offset=5 if ids else 0)
        t += steps
    ph = ctx.photons(on_device=False)
    rec = np.stack([ph[k].numpy().view(np.uint32) for k in
                    ("pid", "step", "x", "y", "nx", "ny", "nz", "eps", "weight")], 1)
    stats = ctx.energy_budget()[2]
    le, ll = ctx.ledger()
    out = ({k: v.cpu().numpy() for k, v in st.items()}, rec[np.lexsort(rec.T[::-1])],
           le.cpu().numpy(), ll.cpu().numpy(), stats)
    ctx.close()
    return out


CASES = {
    # name: (nx, ny, n, ex, ey, order, jitter, steps, per_launch, kw)
    "more items than blocks": (300, 280, 2_097_152, 300, 280, None, 0.0, 9, 9, {}),
    "sparse, specialised": (4100, 4129, 524_301, 4000, 4000, None, 0.0, 9, 8, dict(specialize=True)),
    "clump, specialised": (4100, 4129, 524_301, 60, 70, None, 0.0, 9, 8, dict(specialize=True)),
    "dense, specialised": (256, 250, 2_097_152, 256, 250, None, 0.0, 9, 9, dict(specialize=True)),
    "rows of cells, one step": (300, 280, 2_097_152, 300, 280, "rows", 0.0, 9, 1, {}),
    "cells, drifted, one step": (300, 280, 2_097_152, 300, 280, "cells", 40.0, 9, 1, {}),
    "cells, specialised": (2050, 2049, 2_097_152, 500, 500, "cells", 0.3, 9, 4, dict(specialize=True)),
    "random, specialised": (500, 490, 2_097_152, 500, 490, None, 0.0, 9, 4, dict(specialize=True)),
    "cells, short": (96, 130, 524_301, 96, 130, "cells", 0.0, 9, 9, {}),
    "dense, control": (300, 280, 2_097_152, 300, 280, None, 0.0, 9, 9,
                       dict(n_try=2, select_prob=0.5)),
    "dense, ledger, ids": (300, 280, 2_097_157, 300, 280, None, 0.0, 9, 8,
                           dict(ledger=True, ids=True)),
    "one step, ledger, ids": (300, 280, 2_097_157, 300, 280, None, 0.0, 9, 1,
                              dict(ledger=True, ids=True)),
    "cells, one step, control": (300, 280, 2_097_157, 300, 280, "cells", 0.0, 9, 1,
                                 dict(n_try=2, select_prob=0.5)),
    "more tiles than work": (8200, 8190, 524_301, 60, 70, None, 0.0, 8, 8, {}),
}


@pytest.mark.parametrize("name", CASES)
def test_route_equals_one_step_calls(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny, n, ex, ey, order, jitter, steps, per_launch, kw = CASES[name]
    wl = _problem(nx, ny, n, ex, ey, order, jitter)
    a = _run(wl, [1] * steps, 1, **{k: v for k, v in kw.items() if k != "specialize"})
    b = _run(wl, [steps], per_launch, **kw)
    for k in a[0]:
        np.testing.assert_array_equal(a[0][k], b[0][k], err_msg=k)
    assert 100 < len(a[1]) < 1 << 24
    np.testing.assert_array_equal(a[1], b[1])
    np.testing.assert_allclose(a[2], b[2], rtol=1e-13, atol=0)
    np.testing.assert_allclose(a[3], b[3], rtol=1e-13, atol=0)
    # the electron that is not finite is counted once per launch, by the kernel
    # that advances the others and by no other
    launches = -(-steps // per_launch)
    assert a[4].pop("nan_frozen") == steps and b[4].pop("nan_frozen") == launches
    assert a[4].pop("spec_launches") == 0
    assert b[4].pop("spec_launches") == (launches if kw.get("specialize") else 0)
    assert a[4] == b[4]
