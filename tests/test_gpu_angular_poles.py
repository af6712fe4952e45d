"""Records of a collimated beam, within a few mrad of the histogram's axis or of
its opposite, where the FP32 cosine of the angle rounds beyond +-1: each lands
in the bin that FP64 angles give it, or in none."""
import math

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1409_5574_gb300 import prad

W_REF = 2.0 * math.pi * 299792458.0 / 0.8e-6
M_E, Q_E = 9.1093837015e-31, 1.602176634e-19
BEAMS = [(-1.0, 0.0, 0.0), (3.0, -1.0, -2.0)]


@pytest.fixture(scope="module", params=BEAMS, ids=["along -x", "oblique"])
def beam(request):
    """One step of gamma = 1e5 electrons, off the beam's axis by 1e-5 to 3e-3
    rad, in a constant field that turns them by 5e-4 rad."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = np.asarray(request.param) / np.linalg.norm(request.param)
    e1 = np.cross(d, [0.3, 0.5, -0.7])
    e1 /= np.linalg.norm(e1)
    e2 = np.cross(d, e1)
    rng = np.random.default_rng(3)
    n = 400_000
    th = np.exp(rng.uniform(math.log(1e-5), math.log(3e-3), n))
    ph = rng.uniform(0.0, 2.0 * math.pi, n)
    u = 1e5 * (np.cos(th)[:, None] * d + np.sin(th)[:, None] *
               (np.cos(ph)[:, None] * e1 + np.sin(ph)[:, None] * e2))
    dtn = 2.0 * math.pi / 200.0
    b = (50.0 / dtn) * M_E * W_REF / Q_E  # Omega dt = 50
    zero = np.zeros(n)
    state = dict(x=zero, y=zero, z=zero, ux=u[:, 0].copy(), uy=u[:, 1].copy(), uz=u[:, 2].copy(),
                 w=np.ones(n))
    ctx = prad.Context(dict(omega_ref=W_REF, dt=dtn / W_REF, seed=5, rr_mode=prad.PRAD_RR_LEDGER,
                            field_kind=prad.PRAD_FIELD_CONST, B=tuple(b * e1)),
                       photon_capacity=n, max_particles=n)
    ctx.push_emit(ctx.to_device(state), 1)
    ph = {k: v.numpy() for k, v in ctx.photons(on_device=False).items() if k != "dropped"}
    assert ph["nx"].size > 20_000
    yield ctx, ph, d, e1
    ctx.close()


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("nt,nph,tmax", [(45, 72, np.pi), (45, 72, np.pi / 2), (4096, 2, np.pi),
                                         (1, 7, 3.0), (24, 5, 2e-3)])
def test_bins_at_the_poles(beam, sign, nt, nph, tmax):
    ctx, ph, d, e1 = beam
    axis, ref = tuple(sign * d), tuple(e1)
    got = ctx.angular_histogram(axis=axis, ref=ref, ntheta=nt, nphi=nph, theta_max=tmax)
    want = O.angular_histogram(ph["nx"], ph["ny"], ph["nz"], ph["eps"], ph["weight"], axis, ref,
                               nt, nph, tmax)
    np.testing.assert_array_equal(got != 0.0, want != 0.0)
    # (FP64 sums of the same terms in another order)
    np.testing.assert_allclose(got, want, rtol=ph["nx"].size * 2.0 ** -52, atol=0)
    if sign < 0 and tmax < 3.1:
        assert not want.any()  # (every record lies beyond theta_max)
