"""FP64 emission against the oracle from rates of a few in a thousand per step
to dN far above 1: the trials that an FP32 estimate rules out are exactly trials
without a record, so records, multiplicities and counters agree one by one."""
import numpy as np
import pytest

import oracle as O
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


@pytest.mark.parametrize("n_try,select", [(1, 1.0), (3, 0.5)])
@pytest.mark.parametrize("case", ["constb", "constb_large_dt", "wave"])
def test_fp64_records_equal_oracle(case, n_try, select):
    n, steps = 2053, 30
    if case == "wave":
        wl = W.plane_wave(a0=500.0, n=n, seed=5)
    else:
        wl = W.const_b(n=n, seed=6)
        wl.dt *= 150.0 if case == "constb_large_dt" else 1.0
    ctx = prad.Context(wl.problem_kwargs(), precision=prad.PRAD_FP64, photon_capacity=1 << 19,
                       max_particles=n, steps_per_launch=7, n_try=n_try, select_prob=select)
    ctx.push_emit(ctx.to_device(wl.state), steps)
    g = {k: v.numpy() for k, v in ctx.photons(on_device=False).items() if k != "dropped"}
    stats = ctx.energy_budget()[2]
    ctx.close()
    r = O.run(O.Problem(**wl.problem_kwargs(), n_try=n_try, select_prob=select),
              wl.copy_state(), steps, capacity=1 << 19)
    p = r["photons"]

    def table(q):
        o = np.lexsort((q["eps"], q["step"], q["pid"]))
        return [q[k][o].astype(np.float64) for k in ("pid", "step", "weight", "eps")]

    a, b = table({k: (v.view(np.uint32) if k in ("pid", "step") else v) for k, v in g.items()}), \
        table(p)
    assert 20 < len(a[0]) < 1 << 19 and len(a[0]) == len(b[0])
    for k in range(2):
        np.testing.assert_array_equal(a[k], b[k])
    np.testing.assert_allclose(a[2], b[2], rtol=1e-6)
    np.testing.assert_allclose(a[3], b[3], rtol=1e-6)
    assert stats["dn_gt1"] == r["stats"]["dn_gt1"]


@pytest.mark.parametrize("rr", [0, 1, 2])
@pytest.mark.parametrize("e_field", [0.0, 1e9])
def test_fp64_state_is_the_same_for_every_launch_shape(rr, e_field):
    """Constant B, with and without E (whose zero terms a pure B field leaves
    out), the LL ledger off, booked and applied: 1/gamma is carried from step
    to step within a launch and formed anew at its start, to the same bits."""
    wl = W.const_b(n=700, seed=3, rr_mode=rr)
    wl.E = (0.0, e_field, 0.0)
    got = []
    for spl in (1, 7, 40):
        ctx = prad.Context(wl.problem_kwargs(), precision=prad.PRAD_FP64, max_particles=wl.n,
                           photon_capacity=1 << 14, steps_per_launch=spl)
        st = ctx.to_device(wl.state)
        ctx.push_emit(st, 40)
        got.append({k: v.cpu().numpy() for k, v in st.items()})
        ctx.close()
    ref = wl.copy_state()
    O.run(O.Problem(**wl.problem_kwargs()), ref, 40)
    for k in ("x", "y", "z", "ux", "uy", "uz"):
        np.testing.assert_array_equal(got[0][k], got[1][k], err_msg=k)
        np.testing.assert_array_equal(got[0][k], got[2][k], err_msg=k)
    u = np.stack([got[0][k] - ref[k] for k in ("ux", "uy", "uz")], 1)
    n = np.linalg.norm(np.stack([ref[k] for k in ("ux", "uy", "uz")], 1), axis=1)
    assert (np.linalg.norm(u, axis=1) <= 1e-12 * n).all()
