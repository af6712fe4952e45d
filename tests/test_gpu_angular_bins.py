"""The angular histogram bins by FP32 angles where those are sure of the bin:
every record lands in the bin that FP64 angles give it, for bins from one to
thousands per axis, along and across the beam, and for the angular-spread
kernels whose records it reads."""
import numpy as np
import pytest

import oracle as O
from paper_1409_5574_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1409_5574_gb300 import prad


@pytest.fixture(scope="module")
def held():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = W.plane_wave(a0=450.0, n=40_000, seed=12)
    ctx = prad.Context(wl.problem_kwargs(), photon_capacity=1 << 21, max_particles=wl.n,
                       steps_per_launch=20, diagnostics=prad.PRAD_DIAG_ANGLE_SPREAD)
    ctx.push_emit(ctx.to_device(wl.state), 60)
    ph = {k: v.numpy() for k, v in ctx.photons(on_device=False).items() if k != "dropped"}
    assert 50_000 < ph["nx"].size < 1 << 21
    yield ctx, ph
    ctx.close()


@pytest.mark.parametrize("nt,nph,tmax", [(1, 1, np.pi), (45, 72, np.pi / 2), (4096, 2, np.pi),
                                         (2, 4096, 1.0), (89, 92, 0.3)])
@pytest.mark.parametrize("axis,ref", [((-1.0, 0.0, 0.0), (0.0, 1.0, 0.0)),
                                      ((0.0, 0.0, 1.0), (1.0, 0.0, 0.0)),
                                      ((-3.0, 1.0, 2.0), (0.0, 0.2, -1.0))])
def test_bins_equal_fp64_bins(held, nt, nph, tmax, axis, ref):
    ctx, ph = held
    got = ctx.angular_histogram(axis=axis, ref=ref, ntheta=nt, nphi=nph, theta_max=tmax)
    want = O.angular_histogram(ph["nx"], ph["ny"], ph["nz"], ph["eps"], ph["weight"], axis, ref,
                               nt, nph, tmax)
    # (a direction within FP64 rounding of an edge could go either way: none here)
    np.testing.assert_array_equal(got != 0.0, want != 0.0)
    np.testing.assert_allclose(got, want, rtol=1e-11, atol=0)
