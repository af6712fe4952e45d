"""The angular spread's kernels of the standard configuration (LL kick, field-form
H_eff, one trial, no other diagnostic), fused, one step per launch and on the
Yee grid (plain, tile-sorted, binned), against the oracle and each other.

Records of the same particle and step have the oracle's direction within 5e-4
of the spread's own angle (the table's interpolation error), twice the
collinear direction's difference and 2e-6 for float32 rounding."""
from collections import Counter

import numpy as np
import pytest

import oracle as O
from paper_1409_5574_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1409_5574_gb300 import prad

SPREAD = 2  # PRAD_DIAG_ANGLE_SPREAD


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    prad.load_library()


def _yee(nx, ny, n, seed):
    rng = np.random.default_rng(seed)
    dxn = 2 * np.pi / 32
    wl = W.yee2d(n_grid=64, slab=32, n_particles=n, seed=seed, with_grid=False)
    wl.yee = W.yee_planes(nx, ny, 300.0, dxn, rng)
    wl.state["x"] = rng.uniform(-0.5, nx + 0.5, n) * dxn
    wl.state["y"] = rng.uniform(-0.5, ny + 0.5, n) * dxn
    return wl


def _records(wl, calls, diagnostics, pid=False, **kw):
    ctx = prad.Context(wl.problem_kwargs(), photon_capacity=1 << 22, max_particles=wl.n,
                       diagnostics=diagnostics, **kw)
    st = ctx.to_device(wl.state, with_pid=pid)
    t = 0
    for steps in calls:
        ctx.push_emit(st, steps, t0=t)
        t += steps
    ph = {k: v.numpy() for k, v in ctx.photons(on_device=False).items() if k != "dropped"}
    ctx.close()
    order = np.lexsort((ph["eps"], ph["step"], ph["pid"]))
    return {k: v[order] for k, v in ph.items()}


def _single(ph):
    keys = list(zip(ph["pid"].tolist(), ph["step"].tolist()))
    count = Counter(keys)
    return {k: i for i, k in enumerate(keys) if count[k] == 1}


def _dirs(ph, idx):
    return np.stack([ph["nx"][idx], ph["ny"][idx], ph["nz"][idx]], 1).astype(np.float64)


@pytest.mark.parametrize("case,per_launch", [("wave", 30), ("wave", 1), ("wave back", 7),
                                             ("const", 40), ("yee", 12), ("yee sorted", 5)])
def test_standard_spread_matches_the_oracle(case, per_launch):
    kw, steps = dict(steps_per_launch=per_launch), 30
    if case.startswith("wave"):
        wl = W.plane_wave(a0=300.0, n=3000 + 7, seed=51)
        if case == "wave back":  # the wave along -x, the other handedness
            wl.direction, wl.hand = -1, -1
            wl.state["ux"] = -wl.state["ux"]
    elif case == "const":
        wl, steps = W.const_b(n=3000 + 7, nsteps=150, seed=52), 150
        wl.rr_mode = prad.PRAD_RR_APPLY
    else:
        wl, steps = _yee(130, 100, 9000 + 13, 53), 12
        if case == "yee sorted":
            kw.update(sort_interval=5, pid=True)
    wl = wl.subset(np.arange(wl.n))
    wl.state = {k: v.astype(np.float32).astype(np.float64) for k, v in wl.state.items()}
    assert wl.rr_mode == prad.PRAD_RR_APPLY
    on, off = _records(wl, [steps], SPREAD, **kw), _records(wl, [steps], 0, **kw)
    problem = wl.problem_kwargs()
    ref_on = O.run(O.Problem(**problem, ang_spread=1), wl.copy_state(), steps, capacity=1 << 20)
    ref_off = O.run(O.Problem(**problem), wl.copy_state(), steps, capacity=1 << 20)
    sets = [on, off, ref_on["photons"], ref_off["photons"]]
    keys = [_single(p) for p in sets]
    common = sorted(set(keys[0]) & set(keys[1]) & set(keys[2]) & set(keys[3]))
    assert len(common) > 500
    assert len(common) >= 0.998 * min(len(k) for k in keys) - 4
    d_on, d_off, r_on, r_off = (_dirs(p, np.array([k[c] for c in common]))
                                for p, k in zip(sets, keys))
    theta = np.arccos(np.clip((r_on * r_off).sum(1), -1.0, 1.0))
    assert np.median(theta) > 1e-5  # (the spread is really there)
    tol = 5e-4 * theta + 2.0 * np.linalg.norm(d_off - r_off, axis=1) + 2e-6
    bad = np.linalg.norm(d_on - r_on, axis=1) > tol
    assert bad.sum() <= 1e-3 * len(common), bad.sum()


@pytest.mark.parametrize("rr", ["apply", "ledger"])
@pytest.mark.parametrize("tiled", ["binned", "sorted"])
def test_tiled_spread_equals_plain(rr, tiled):
    """Standard (apply) and general (ledger) variants: the same records from the
    planes and from staged tiles, directions to the rounding of the turn."""
    wl = _yee(150, 90, 524_301, 54)
    wl.rr_mode = prad.PRAD_RR_APPLY if rr == "apply" else prad.PRAD_RR_LEDGER
    steps = 8
    a = _records(wl, [1] * steps, SPREAD, pid=tiled == "sorted")
    b = _records(wl, [steps], SPREAD, pid=tiled == "sorted", steps_per_launch=steps,
                 sort_interval=4 if tiled == "sorted" else 0)
    assert 1000 < a["pid"].size < 1 << 22
    for k in ("pid", "step", "x", "y", "z", "eps", "weight"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    for k in ("nx", "ny", "nz"):
        np.testing.assert_allclose(a[k], b[k], rtol=0, atol=5e-7, err_msg=k)
