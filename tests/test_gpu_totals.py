"""The ledger totals are the exact sums of the FP64 entries, rounded once:
equal to math.fsum bit for bit, for every size, alignment, sign and exponent."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1409_5574_gb300 import prad


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    prad.load_library()


def _totals(a, b, shift=0):
    n = a.size
    pad = np.zeros(shift)
    ta, tb = (torch.as_tensor(np.concatenate([pad, v])).cuda()[shift:] for v in (a, b))
    out = torch.full((2,), 7.0, dtype=torch.float64, device="cuda")
    prad.prad_ledger_totals_noalloc(ta.data_ptr(), tb.data_ptr(), n, out.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _values(kind, n, rng):
    v = np.exp(3.0 * rng.standard_normal(n))
    if kind == "sparse":
        v *= rng.random(n) < 0.4
    elif kind == "signed":
        v *= rng.choice([-1.0, 1.0], n)
    elif kind == "wide":  # every exponent, subnormals and zeros among them
        v = rng.choice([-1.0, 1.0], n) * np.ldexp(rng.random(n), rng.integers(-1080, 1000, n))
    elif kind == "cancel":  # the large entries cancel
        h = n // 2
        v[:h] = 1e30 * rng.standard_normal(h)
        v[h:2 * h] = -v[:h][::-1]
    return v


@pytest.mark.parametrize("kind", ["plain", "sparse", "signed", "wide", "cancel"])
@pytest.mark.parametrize("n,shift", [(1, 0), (2, 1), (33, 0), (2049, 1), (300_001, 0),
                                     (2_000_000, 1), (6_000_003, 0)])
def test_totals_are_exact(kind, n, shift):
    rng = np.random.default_rng(n + shift)
    a, b = _values(kind, n, rng), _values("plain", n, rng)
    got = _totals(a, b, shift)
    assert got[0] == math.fsum(a) and got[1] == math.fsum(b)


def test_totals_of_non_finite_entries():
    a = np.ones(1000)
    for bad in (np.inf, -np.inf, np.nan):
        b = a.copy()
        b[777] = bad
        got = _totals(a, b)
        assert got[0] == 1000.0 and math.isnan(got[1])
    assert np.array_equal(_totals(-a, 0.0 * a), [-1000.0, 0.0])
    tiny = np.full(5, 5e-324)
    assert _totals(tiny, -tiny).tolist() == [25e-324, -25e-324]
