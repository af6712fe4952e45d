"""Two threads push their own electrons through one context whose Yee calls
share the binning scratch, with more electrons from call to call: the results
are those of the same calls in turn."""
import threading

import numpy as np
import pytest

from paper_1409_5574_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1409_5574_gb300 import prad

N = (524_300, 524_900, 530_001, 545_003)  # (electrons of a thread's calls)
STEPS = 8


@pytest.fixture(scope="module")
def problem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = W.yee2d(n_grid=64, slab=32, n_particles=64, seed=2, with_grid=False)
    dxn = 2 * np.pi / 32
    rng = np.random.default_rng(2)
    wl.yee = W.yee_planes(200, 130, 250.0, dxn, rng)
    states = []
    for _ in range(2):
        n = N[-1]
        u = rng.standard_normal((3, n))
        u *= np.exp(rng.uniform(np.log(10.0), np.log(2000.0), n)) / np.linalg.norm(u, axis=0)
        states.append(dict(x=rng.uniform(0, 200, n) * dxn, y=rng.uniform(0, 130, n) * dxn,
                           ux=u[0], uy=u[1], uz=u[2], w=np.ones(n)))
    return wl, states


def _run(problem, threads):
    wl, states = problem
    ctx = prad.Context(wl.problem_kwargs(), photon_capacity=1 << 23, max_particles=2 * N[-1],
                       steps_per_launch=STEPS)
    st = [ctx.to_device(s) for s in states]
    torch.cuda.synchronize()
    failed = []

    def calls(k):
        try:
            for j, n in enumerate(N):
                part = {name: v[:n] for name, v in st[k].items()}
                ctx.push_emit(part, STEPS, t0=j * STEPS, pid0=k * N[-1], ledger_offset=k * N[-1])
        except Exception as e:  # noqa: BLE001 (raised by the test)
            failed.append(e)

    if threads:
        ts = [threading.Thread(target=calls, args=(k,)) for k in range(2)]
        for t in ts:
            t.start()
        for t in ts:
            t.join(120)
    else:
        calls(0)
        calls(1)
    assert not failed, failed
    torch.cuda.synchronize()
    ph = ctx.photons(on_device=False)
    rec = np.stack([ph[k].numpy().view(np.uint32) for k in
                    ("pid", "step", "x", "y", "nx", "ny", "nz", "eps", "weight")], 1)
    le, ll = ctx.ledger()
    out = ([{k: v.cpu().numpy() for k, v in s.items()} for s in st], rec[np.lexsort(rec.T[::-1])],
           le.cpu().numpy(), ll.cpu().numpy(), ctx.energy_budget()[2])
    ctx.close()
    return out


def test_two_threads_on_one_context(problem):
    a, b = _run(problem, False), _run(problem, True)
    for k in range(2):
        for name in a[0][k]:
            np.testing.assert_array_equal(a[0][k][name], b[0][k][name], err_msg=name)
    assert 100 < len(a[1]) < 1 << 23
    np.testing.assert_array_equal(a[1], b[1])
    np.testing.assert_allclose(a[2], b[2], rtol=1e-13, atol=0)
    np.testing.assert_allclose(a[3], b[3], rtol=1e-13, atol=0)
    assert a[4] == b[4]
