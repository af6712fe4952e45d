"""The workloads the library's speed is measured on: what a program that pushes
radiating electrons with it does in one pass, through the public entry points
(``prad.Context`` and the C names behind it).

A case is a dict of plain values; ``kind`` names the workload:

``wave``    electrons against a circularly polarised plane wave: FP32, table
            or learned sampler, optionally with the angular spread of the
            emission and the Fig. 4 histogram; ``calls`` push calls a pass
``yee``     electrons on a 2D Yee grid, in the caller's own order (``sort``
            0) or reordered every ``sort`` steps
``constb``  the FP64 check in a constant magnetic field
``batch``   uneven independent ensembles in one persistent launch
``train``   training of the learned sampler's network
``totals``  totals of a caller's own FP64 ledgers

Sizes come from the library's benchmark, tests and workload generators.  A
pass of the particle workloads pushes a run's electrons, then reads the
energy budget with its counters and the per-particle ledgers; once a run's
``span`` of steps is over, the next pass starts a new run (context reset, the
initial state loaded again).
"""
import math

import numpy as np
import torch

from paper_1409_5574_gb300 import prad

C_LIGHT, Q_E, M_E = 299792458.0, 1.602176634e-19, 9.1093837015e-31
HBAR, EPS0 = 1.054571817e-34, 8.8541878128e-12
LAM = 0.8e-6
W_LASER = 2.0 * math.pi * C_LIGHT / LAM
ALPHA = Q_E * Q_E / (4.0 * math.pi * EPS0 * HBAR * C_LIGHT)
COUNTS = ("records", "dropped", "dn_gt1", "clamped", "chi_gt1", "nan_frozen", "mlp_fallback")


# ---- cases -------------------------------------------------------------------
def _wave(name=None, n=1 << 20, steps=100, per_launch=100, calls=1, span=0, a0=500.0, hand=1,
          direction=1, rr=prad.PRAD_RR_APPLY, learned=False, spread=False, specialize=False):
    c = dict(kind="wave", n=n, steps=steps, per_launch=per_launch, calls=calls,
             span=span or steps * calls, a0=a0, hand=hand, direction=direction, rr=rr,
             learned=learned, spread=spread, specialize=specialize)
    return dict(c, name=name) if name else c


def _yee(name=None, grid=2048, n=1 << 20, slab=256, steps=25, per_launch=25, sort=0, a0=300.0,
         specialize=False):
    c = dict(kind="yee", grid=grid, n=n, slab=slab, steps=steps, per_launch=per_launch, sort=sort,
             a0=a0, specialize=specialize)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest calls: a few electrons, one launch per step, as the
        # smoke check runs them (launches and latency are all there is)
        _wave("wave 1000 x 20 one-step", n=1000, steps=20, per_launch=1, a0=300.0),
        # a small set advanced in one fused launch (the parity tests' size)
        _wave("wave 4173 x 40 fused", n=4173, steps=40, per_launch=40, a0=300.0),
        # a field solver's host loop: one call of one step between two field
        # solves, state larger than L2 (the benchmark's one-step workload)
        _wave("wave 2^24 one-step calls", n=1 << 24, steps=1, per_launch=1, calls=16, span=192),
        # the benchmark's headline: strongly emitting electrons, 100 fused
        # steps, kernels specialised at run time
        _wave("wave 2^24 x 100 fused", n=1 << 24, specialize=True),
        # the same physics drawn by the learned sampler
        _wave("wave 2^22 x 100 learned", n=1 << 22, learned=True),
        # the emission's angular spread and the Fig. 4 histogram of the records
        _wave("wave 2^20 x 100 spread", n=1 << 20, spread=True),
        # a grid whose electrons stay in the caller's order (the default)
        _yee("yee 2^21 unsorted", grid=2048, n=(1 << 21) + 37, slab=512, steps=25, per_launch=25),
        # the benchmark's grid and schedule: sorted every 50 steps
        _yee("yee 2^22 sorted", grid=4096, n=(1 << 22) + 1001, slab=512, steps=100,
             per_launch=50, sort=50, specialize=True),
        # the FP64 constant-field check, full size
        dict(name="const B 10^4 FP64", kind="constb", n=10_000, steps=1000, per_launch=1000),
        # uneven ensembles under one graph, autotuned
        dict(name="64 ensembles", kind="batch", count=64, nmin=1_000, nmax=300_000, steps=100),
        # the learned sampler's network, at the batch it is trained with
        dict(name="train 65536 x 24", kind="train", batch=65536, steps=24),
        # a host code's own ledgers summed without allocation
        dict(name="totals 2^25", kind="totals", n=1 << 25),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["one-step", "one-step", "fused", "fused", "learned", "spread", "plain",
                       "sorted", "constb", "batch", "train", "totals"])
    sign = dict(hand=rng.choice([1, -1]), direction=rng.choice([1, -1]),
                a0=float(rng.randint(100, 500)))
    if kind == "one-step":  # (at most 2^24 particles, about 2.7e8 particle-steps)
        n = _log(rng, 100, 1 << 24)
        calls = max(1, min(rng.randint(4, 40), (1 << 28) // n))
        return _wave(n=n, steps=1, per_launch=1, calls=calls, span=4 * calls, **sign)
    if kind == "fused":  # (at most 1.6e9 particle-steps)
        n = _log(rng, 1000, 1 << 24)
        steps = max(5, min(_log(rng, 10, 200), 1_600_000_000 // n))
        return _wave(n=n, steps=steps, per_launch=rng.choice([steps, max(2, steps // 3)]),
                     rr=rng.choice([prad.PRAD_RR_APPLY, prad.PRAD_RR_APPLY, prad.PRAD_RR_LEDGER]),
                     specialize=rng.random() < 0.3, **sign)
    if kind == "learned":
        return _wave(n=_log(rng, 10_000, 1 << 22), steps=rng.randint(10, 100), learned=True,
                     **sign)
    if kind == "spread":
        return _wave(n=_log(rng, 10_000, 1 << 21), steps=rng.randint(10, 100), spread=True,
                     **sign)
    if kind in ("plain", "sorted"):
        grid = rng.choice([512, 1000, 2048, 3001])
        slab = rng.randint(64, min(grid - 64, 512))
        n = max(10_000, min(1 << 22, slab * slab * rng.randint(1, 16) + rng.randint(0, 99)))
        steps = rng.randint(8, 60)
        return _yee(grid=grid, n=n, slab=slab, steps=steps, per_launch=rng.choice([steps, 8, 1]),
                    sort=0 if kind == "plain" else rng.choice([16, 50]),
                    a0=float(rng.randint(100, 400)))
    if kind == "constb":
        return dict(kind="constb", n=_log(rng, 500, 30_000), steps=rng.randint(100, 500),
                    per_launch=rng.choice([100, 1000]))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(8, 96), nmin=1_000,
                    nmax=_log(rng, 10_000, 300_000), steps=rng.randint(20, 100))
    if kind == "train":
        return dict(kind="train", batch=rng.choice([4096, 10_000, 32768, 65536]),
                    steps=rng.randint(2, 24))
    return dict(kind="totals", n=_log(rng, 1000, 1 << 26))


# ---- inputs -------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _isotropic(g, n):
    v = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=0, keepdim=True)


def _state(x, y, z, u, dtype=torch.float32):
    out = dict(x=x, y=y, z=z, ux=u[0], uy=u[1], uz=u[2], w=torch.ones_like(x))
    return {k: v.to(dtype, copy=True).contiguous() for k, v in out.items()}  # (an array each)


def _wave_problem(c):
    return dict(omega_ref=W_LASER, dt=2.0 * math.pi / W_LASER / 200.0, seed=1,
                rr_mode=c.get("rr", prad.PRAD_RR_APPLY), field_kind=prad.PRAD_FIELD_PLANE_WAVE,
                a0=c["a0"], lam=LAM, direction=c.get("direction", 1), hand=c.get("hand", 1))


def _wave_state(c, g, n):
    """gamma = 1000 against the wave, 1% spread, uniform over a wavelength."""
    u0 = math.sqrt(1000.0 ** 2 - 1.0)
    u = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64) * (0.01 * u0)
    u[0] -= u0 * c.get("direction", 1)
    zero = torch.zeros(n, device="cuda", dtype=torch.float64)
    return _state(_uniform(g, n, 0.0, 2.0 * math.pi), zero, zero, u)


def _const_problem(b_tesla, omega_ref, dt, rr):
    return dict(omega_ref=omega_ref, dt=dt, seed=1, rr_mode=rr, field_kind=prad.PRAD_FIELD_CONST,
                B=(0.0, 0.0, b_tesla))


def _const_state(g, n, dtype):
    """gamma uniform in [100, 1000], isotropic, at the origin."""
    gamma = _uniform(g, n, 100.0, 1000.0)
    zero = torch.zeros(n, device="cuda", dtype=torch.float64)
    return _state(zero, zero, zero, _isotropic(g, n) * torch.sqrt(gamma * gamma - 1.0), dtype)


def _constb(c, g):
    omega = Q_E * 1.0e4 / M_E
    return (_const_problem(1.0e4, omega, 1.0e-3 * 2.0 * math.pi * 100.0 / omega,
                           prad.PRAD_RR_LEDGER), _const_state(g, c["n"], torch.float64))


def _yee_inputs(c, g):
    """Standing wave plus 1% noise on every plane, electrons uniform over the
    central slab x slab cells, gamma log-uniform in [10, 3000], isotropic."""
    grid, a0, dx = c["grid"], c["a0"], 2.0 * math.pi / 32.0
    i = torch.arange(grid, device="cuda", dtype=torch.float64)
    planes = []
    for k in range(6):
        p = torch.randn(grid, grid, generator=g, device="cuda") * (0.01 * a0)
        if k == 1:
            p += (a0 * math.cos(math.pi / 4) * torch.sin(i * dx)).float()[None, :]
        if k == 5:
            p += (a0 * math.sin(math.pi / 4) * torch.cos((i + 0.5) * dx)).float()[None, :]
        planes.append(p)
    n, lo, slab = c["n"], (grid - c["slab"]) // 2, c["slab"]
    x = (_uniform(g, n, 0.0, slab) + lo) * dx
    y = (_uniform(g, n, 0.0, slab) + lo) * dx
    gamma = torch.exp(_uniform(g, n, math.log(10.0), math.log(3000.0)))
    st = _state(x, y, torch.zeros_like(x), _isotropic(g, n) * torch.sqrt(gamma * gamma - 1.0))
    st.pop("z")
    return dict(omega_ref=W_LASER, dt=2.0 * math.pi / W_LASER / 200.0, seed=1,
                rr_mode=prad.PRAD_RR_APPLY, field_kind=prad.PRAD_FIELD_YEE2D, yee=planes, dx=dx,
                dy=dx), st


def _ensembles(c, g, seed):
    """Sizes log-uniform, a0 uniform in [50, 500], plane wave or constant B."""
    r = np.random.default_rng(seed)
    # (the sizes belong to the case: other inputs, the same work)
    sizes = np.exp(np.random.default_rng(c["count"]).uniform(
        math.log(c["nmin"]), math.log(c["nmax"]), c["count"])).astype(int)
    problems, states = [], []
    for k, n in enumerate(sizes):
        a0 = float(r.uniform(50.0, 500.0))
        if k % 2 == 0:
            problems.append(_wave_problem(dict(a0=a0)))
            states.append(_wave_state({}, g, int(n)))
        else:
            problems.append(_const_problem(a0 * M_E * W_LASER / Q_E, W_LASER,
                                           2.0 * math.pi / W_LASER / 200.0, prad.PRAD_RR_APPLY))
            states.append(_const_state(g, int(n), torch.float32))
    return problems, states


_WEIGHTS = {}


def _net_weights():
    """Weights of a usable network without training it here: random hidden
    layers, the output layer fitted by least squares to the residual
    ln G^-1(r) - prior(r) of the photon-number spectrum."""
    if "w" in _WEIGHTS:
        return _WEIGHTS["w"]
    g = torch.Generator()
    g.manual_seed(7)
    w1 = (torch.rand(64, 3, generator=g, dtype=torch.float64) * 2 - 1) * 1.5
    w1[:, 1:] *= 0.05
    b1 = (torch.rand(64, generator=g, dtype=torch.float64) * 2 - 1) * 1.5
    w2 = (torch.rand(64, 64, generator=g, dtype=torch.float64) * 2 - 1) * 0.4
    b2 = (torch.rand(64, generator=g, dtype=torch.float64) * 2 - 1) * 0.5
    w1, w2 = w1.bfloat16().double(), w2.bfloat16().double()
    # F(x) by the trapezoid rule, G(x) by the trapezoid rule in ln x
    lx = torch.linspace(math.log(1e-12), math.log(80.0), 4000, dtype=torch.float64)
    s = torch.linspace(0.0, 36.0, 1201, dtype=torch.float64)
    f = (torch.exp(-torch.exp(lx)[:, None] * torch.cosh(s)[None]) *
         (torch.cosh(5.0 * s / 3.0) / torch.cosh(s))[None])
    f = torch.exp(lx) * (f.sum(1) - 0.5 * (f[:, 0] + f[:, -1])) * (s[1] - s[0])
    cum = torch.cat([3.0 * f[:1], 3.0 * f[0] + torch.cumsum(
        0.5 * (f[1:] + f[:-1]) * (lx[1] - lx[0]), 0)])
    G = (cum / cum[-1]).numpy()
    lr = np.linspace(-13.0, 9.0, 2000)
    r = 1.0 / (1.0 + np.exp(-lr))
    target = np.interp(r, G, lx.numpy()) - (np.log(-np.log1p(-r)) + 2.0 * (1.0 - r) * np.log(r))
    feat = torch.zeros(r.size, 3, dtype=torch.float64)
    feat[:, 0] = torch.as_tensor(lr / 8.0)
    h = torch.nn.functional.silu(feat @ w1.T + b1)
    h = torch.nn.functional.silu(h @ w2.T + b2)
    a = torch.cat([h, torch.ones(r.size, 1, dtype=torch.float64)], 1)
    ridge = 1e-4 * torch.eye(65, dtype=torch.float64)
    sol = torch.linalg.solve(a.T @ a / r.size + ridge, a.T @ torch.as_tensor(target) / r.size)
    _WEIGHTS["w"] = torch.cat([w1.reshape(-1), b1, w2.reshape(-1), b2, sol[:64],
                               sol[64:]]).float().numpy()
    return _WEIGHTS["w"]


def prepare(case, seed):
    c, g = case, _gen(seed)
    kind = c["kind"]
    if kind == "totals":
        n = c["n"]
        emit = torch.exp(3.0 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
        emit *= torch.rand(n, generator=g, device="cuda") < 0.6  # (some emitted nothing)
        loss = torch.exp(torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
        return dict(kind=kind, emit=emit, loss=loss,
                    out=torch.zeros(2, dtype=torch.float64, device="cuda"), n=n)
    if kind == "train":
        ctx = prad.Context(_wave_problem(dict(a0=500.0)), photon_capacity=1024, max_particles=1024,
                           sampler=prad.PRAD_SAMPLER_MLP_FALLBACK)
        r = np.random.default_rng(seed)
        w0 = (_net_weights() * r.uniform(0.9, 1.1, 4481)).astype(np.float32)
        return dict(kind=kind, ctx=ctx, w0=w0, seed=int(seed), **{k: c[k] for k in ("batch", "steps")})
    if kind == "batch":
        problems, states = _ensembles(c, g, seed)
        total = sum(s["x"].numel() for s in states)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        ctx = prad.Context(problems[0], photon_capacity=int(0.1 * total * c["steps"]) + (1 << 20),
                           max_particles=total, steps_per_launch=c["steps"], stream=stream,
                           use_graph=True)
        ens = ctx.ensembles(states, problems)
        ctx.autotune_batch(ens, probe_steps=10, sample=4096)
        init = [{k: v.clone() for k, v in s.items()} for s in states]
        return dict(kind=kind, ctx=ctx, ens=ens, st=states, init=init, steps=c["steps"], t=0,
                    stream=stream)
    if kind == "wave":
        problem, st = _wave_problem(c), _wave_state(c, g, c["n"])
        span, calls, steps = c["span"], c["calls"], c["steps"]
    elif kind == "constb":
        problem, st = _constb(c, g)
        span, calls, steps = c["steps"], 1, c["steps"]
    else:
        problem, st = _yee_inputs(c, g)
        span, calls, steps = c["steps"], 1, c["steps"]
    n = c["n"]
    ctx = prad.Context(
        problem, precision=prad.PRAD_FP64 if kind == "constb" else prad.PRAD_FP32,
        photon_capacity=int(0.14 * n * span) + (1 << 14), max_particles=n,
        steps_per_launch=c["per_launch"], specialize=c.get("specialize", False),
        sort_interval=c.get("sort", 0),
        sampler=prad.PRAD_SAMPLER_MLP_FALLBACK if c.get("learned") else prad.PRAD_SAMPLER_TABLE,
        diagnostics=prad.PRAD_DIAG_ANGLE_SPREAD if c.get("spread") else 0)
    if c.get("learned"):
        ctx.mlp_set_weights(_net_weights())
    if c.get("sort"):
        st["pid"] = torch.arange(n, device="cuda", dtype=torch.int32)
    init = {k: v.clone() for k, v in st.items() if k != "w"}
    return dict(kind=kind, ctx=ctx, st=st, init=init, t=0, span=span, calls=calls, steps=steps,
                axis=(-float(c.get("direction", 1)), 0.0, 0.0) if c.get("spread") else None)


# ---- one pass -------------------------------------------------------------------
def _budget(ctx):
    emitted, loss, stats = ctx.energy_budget()
    return [emitted, loss, list(ctx.ledger()), [int(stats[k]) for k in COUNTS]]


def run(state):
    s = state
    kind = s["kind"]
    if kind == "totals":
        prad.prad_ledger_totals_noalloc(s["emit"].data_ptr(), s["loss"].data_ptr(), s["n"],
                                        s["out"].data_ptr(),
                                        torch.cuda.current_stream().cuda_stream)
        return [s["out"]]
    if kind == "train":
        s["ctx"].mlp_set_weights(s["w0"])
        loss = s["ctx"].mlp_train(s["steps"], batch=s["batch"], seed=s["seed"])
        return [s["ctx"].mlp_weights(), float(loss)]
    ctx = s["ctx"]
    if kind == "batch":
        with torch.cuda.stream(s["stream"]):
            if s["t"]:
                ctx.reset()
                for st, init in zip(s["st"], s["init"]):
                    for k in ("x", "y", "z", "ux", "uy", "uz"):
                        st[k].copy_(init[k])
            ctx.push_emit_batch(s["ens"], s["steps"])
            s["t"] = s["steps"]
            out = [torch.cat([st[k] for st in s["st"]]) for k in ("x", "y", "z", "ux", "uy", "uz")]
            return out + _budget(ctx)
    st = s["st"]
    if s["t"] >= s["span"]:  # the next run
        ctx.reset()
        for k, v in s["init"].items():
            st[k].copy_(v)
        s["t"] = 0
    for _ in range(s["calls"]):
        ctx.push_emit(st, s["steps"], t0=s["t"])
        s["t"] += s["steps"]
    arrays = [st[k] for k in ("x", "y", "z", "ux", "uy", "uz") if k in st]
    if "pid" in st:  # the electrons were reordered: read them by their ids
        at = st["pid"].long()
        arrays = [torch.empty_like(v).scatter_(0, at, v) for v in arrays]
    out = arrays + _budget(ctx)
    if s["axis"] is not None:
        out.append(ctx.angular_histogram(axis=s["axis"]))
    return out


# ---- what a pass cannot do without ------------------------------------------------
def work(case):
    """Bytes: each input read once, each output written once (the state, the
    ledgers read and written, 40 bytes per record).  Operations: the method's
    arithmetic per particle-step, about 250, and 150 more on the grid."""
    c = case
    if c["kind"] == "totals":
        return dict(bytes=16.0 * c["n"], flops=2.0 * c["n"])
    if c["kind"] == "train":  # forward, and twice that backward
        return dict(bytes=4.0 * 4481 * 6 * c["steps"], flops=6.0 * 4480 * c["batch"] * c["steps"])
    if c["kind"] == "batch":
        sizes = np.exp(np.random.default_rng(c["count"]).uniform(
            math.log(c["nmin"]), math.log(c["nmax"]), c["count"])).astype(int)
        n, steps, per = int(sizes.sum()), c["steps"], 250.0
    else:
        n, steps = c["n"], c["steps"] * c.get("calls", 1)
        per = 400.0 if c["kind"] == "yee" else 250.0
    elem = 8 if c["kind"] == "constb" else 4
    rate = {"wave": 0.06, "yee": 0.02, "constb": 0.005, "batch": 0.03}[c["kind"]]
    passes = c.get("calls", 1)
    bytes_ = passes * n * (13.0 * elem + 32.0) + rate * n * steps * 40.0
    if c["kind"] == "yee":  # the field values under the slab
        bytes_ += 24.0 * c["slab"] ** 2
    if c.get("spread"):
        bytes_ += rate * n * steps * 20.0
    return dict(bytes=bytes_, flops=per * n * steps)


# ---- the same in 64 bits ------------------------------------------------------------
def _gather(p, x, y, planes):
    """Fields at (x, y): quadratic splines on the six staggered planes."""
    dx, out = p["dx"], []
    stag = ((0.5, 0.0), (0.0, 0.5), (0.0, 0.0), (0.0, 0.5), (0.5, 0.0), (0.5, 0.5))
    ny, nx = planes[0].shape

    def axis(v, s, n):
        t = v / dx - s
        near = torch.floor(t + 0.5)
        d = t - near
        w = (0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2)
        return w, [torch.remainder(near + k, n).long() for k in (-1, 0, 1)]

    for plane, (sx, sy) in zip(planes, stag):
        (wx, ix), (wy, iy) = axis(x, sx, nx), axis(y, sy, ny)
        flat = plane.reshape(-1)
        out.append(sum(wy[b] * wx[a] * flat[iy[b] * nx + ix[a]].double()
                       for a in range(3) for b in range(3)))
    return out


def _trajectory(p, st, steps):
    """State and Landau-Lifshitz ledger after `steps` steps from step 0, in
    FP64 by plain tensor arithmetic (the emission does not act back)."""
    x, y, z, ux, uy, uz, w = [st[k].double() if k in st else torch.zeros_like(st["x"]).double()
                              for k in ("x", "y", "z", "ux", "uy", "uz", "w")]
    wr = p["omega_ref"]
    dt, eps_r = p["dt"] * wr, HBAR * wr / (M_E * C_LIGHT ** 2)
    ll_coef, hq = 2.0 / 3.0 * ALPHA * eps_r * dt, -0.5 * dt
    kind, rr = p["field_kind"], p["rr_mode"]
    if kind == prad.PRAD_FIELD_CONST:
        e = [0.0, 0.0, 0.0]
        b = [v * Q_E / (M_E * wr) for v in p["B"]]
    loss = torch.zeros_like(x)
    for t in range(steps):
        if kind == prad.PRAD_FIELD_PLANE_WAVE:
            phi = t * dt - p["direction"] * x
            ey, ez = p["a0"] * torch.cos(phi), p["hand"] * p["a0"] * torch.sin(phi)
            e, b = [0.0, ey, ez], [0.0, -p["direction"] * ez, p["direction"] * ey]
        elif kind == prad.PRAD_FIELD_YEE2D:
            f = _gather(p, x, y, p["yee"])
            e, b = f[:3], f[3:]
        mx, my, mz = ux + hq * e[0], uy + hq * e[1], uz + hq * e[2]
        ig = torch.rsqrt(1.0 + mx * mx + my * my + mz * mz)
        tx, ty, tz = hq * b[0] * ig, hq * b[1] * ig, hq * b[2] * ig
        sf = 2.0 / (1.0 + tx * tx + ty * ty + tz * tz)
        vx, vy, vz = (mx + (my * tz - mz * ty), my + (mz * tx - mx * tz), mz + (mx * ty - my * tx))
        nx = mx + sf * (vy * tz - vz * ty) + hq * e[0]
        ny = my + sf * (vz * tx - vx * tz) + hq * e[1]
        nz = mz + sf * (vx * ty - vy * tx) + hq * e[2]
        ax, ay, az = 0.5 * (ux + nx), 0.5 * (uy + ny), 0.5 * (uz + nz)
        ua2 = ax * ax + ay * ay + az * az
        ga = torch.sqrt(1.0 + ua2)
        bx, by, bz = ax / ga, ay / ga, az / ga
        fx, fy, fz = (e[0] + (by * b[2] - bz * b[1]), e[1] + (bz * b[0] - bx * b[2]),
                      e[2] + (bx * b[1] - by * b[0]))
        eb = e[0] * bx + e[1] * by + e[2] * bz
        om = torch.sqrt(torch.clamp(fx * fx + fy * fy + fz * fz - eb * eb, min=0.0))
        om = torch.minimum(om, ga / dt)
        loss += w * ll_coef * om * om * ua2
        if rr == prad.PRAD_RR_APPLY:
            fk = 1.0 / (1.0 + ll_coef * om * om * torch.sqrt(1.0 + nx * nx + ny * ny + nz * nz))
            nx, ny, nz = nx * fk, ny * fk, nz * fk
        ux, uy, uz = nx, ny, nz
        dtg = dt * torch.rsqrt(1.0 + ux * ux + uy * uy + uz * uz)
        x, y, z = x + dtg * ux, y + dtg * uy, z + dtg * uz
        if kind == prad.PRAD_FIELD_YEE2D:
            lx = p["dx"] * p["yee"][0].shape[1]
            ly = p["dx"] * p["yee"][0].shape[0]
            x, y = torch.remainder(x, lx), torch.remainder(y, ly)
    return [x, y, z, ux, uy, uz], loss


def exact(case, seed):
    """What follows from the inputs alone: the state and the radiation-loss
    ledger.  (The photons are random draws.)"""
    c, g = case, _gen(seed)
    kind = c["kind"]
    if kind == "train":
        return None
    if kind == "totals":
        s = prepare(c, seed)
        return [torch.tensor([math.fsum(s[k].cpu().tolist()) for k in ("emit", "loss")],
                             dtype=torch.float64)]
    if kind == "batch":
        problems, states = _ensembles(c, g, seed)
        got = [_trajectory(p, s, c["steps"]) for p, s in zip(problems, states)]
        arrays = [torch.cat([a[k] for a, _ in got]) for k in range(6)]
        loss = torch.cat([v for _, v in got])
    else:
        make = {"wave": lambda: (_wave_problem(c), _wave_state(c, g, c["n"])),
                "constb": lambda: _constb(c, g), "yee": lambda: _yee_inputs(c, g)}[kind]
        problem, st = make()
        arrays, loss = _trajectory(problem, st, c["steps"] * c.get("calls", 1))
        if kind == "yee":
            arrays = arrays[:2] + arrays[3:]
    out = arrays + [None, float(loss.sum()), [None, loss], None]
    return out + [None] if c.get("spread") else out
