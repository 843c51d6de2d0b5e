"""The workloads whose speed this framework is judged by, each through the calls a user makes.

A forecasting centre holds ONE operator (a context: block columns loaded, K
factored) for months and sends it event after event.  So `prepare` keeps the
context of a case, which depends on the case's sizes alone, and makes the
event data, windows and random draws from the seed; only the set-up case, whose
work is the loading and the factorisation, has a context and an operator of
its own for every seed.

Kinds of case:
  event    posterior mean and forecast of one event (tw_infer_forecast)
  batch    the same for several events with windows of their own (tw_infer_batch)
  samples  posterior samples with windows (tw_sample_posterior_batch)
  apply    d = F x and then F^T d, the map in both directions
  qoi      the forecast from the data alone, q = Q d, on the Phase 3 map
  setup    Phase 2: load the block column, form and factor K, and one solve

Operators follow the recipe of the repository's synthetic workloads: sensors and
forecast points uniform in the unit square, a travelling Gaussian pulse of
amplitude 1 / (1 + 10 r), a Matern prior (nu 1, length 0.1, variance 1), noise of
1% of the data's expected size.  The sizes of the large cases are the
repository's benchmark (100 sensors, 200 x 250 grid, 400 steps, 20 forecast
points; 64 events and 32 samples) and its serving workload (200 sensors,
316 x 316 grid, 50 forecast points).
"""
import math

import torch

from paper_2504_16344_gb300 import tw

PREC = {"fp64": tw.PREC_FP64, "c64": tw.PREC_C64, "bf16x2": tw.PREC_BF16X2}
KEEP = {"fp64": tw.KEEP_FP64, "c64": tw.KEEP_C64, "bf16x2": tw.KEEP_BF16X2}
NU, ELL, VAR = 1.0, 0.1, 1.0
SOURCES = 32          # grid points of an event's rupture

BENCH = dict(Nd=100, Nx=200, Ny=250, Nt=400, Nq=20)
# the benchmark's context serves FP64-class and complex64 calls, G* precomputed
BENCH_KEEP = dict(also="c64", gstar=True)


def listed():
    return [
        # the smallest call: an array of 8 sensors, where launches and latency count
        dict(name="event_tiny_fp64", kind="event", prec="fp64", Nd=8, Nx=16, Ny=16, Nt=32, Nq=4,
             window=32, also="", gstar=False),
        # early warning on a regional array: odd sizes, less than half of the window observed,
        # prior filter applied on the fly
        dict(name="event_early_fp64", kind="event", prec="fp64", Nd=26, Nx=60, Ny=75, Nt=77, Nq=3,
             window=30, also="", gstar=False),
        # the headline step: one event, the whole window, FP64-class and complex64
        dict(name="event_fp64", kind="event", prec="fp64", window=400, **BENCH, **BENCH_KEEP),
        dict(name="event_c64", kind="event", prec="c64", window=400, **BENCH, **BENCH_KEEP),
        # the Hessian's two halves, F and F^T, at the headline size
        dict(name="apply_fp64", kind="apply", prec="fp64", **BENCH, **BENCH_KEEP),
        # 64 events with windows of their own, both precisions, and 32 posterior samples
        dict(name="batch_fp64", kind="batch", prec="fp64", B=64, **BENCH, **BENCH_KEEP),
        dict(name="batch_c64", kind="batch", prec="c64", B=64, **BENCH, **BENCH_KEEP),
        dict(name="samples_fp64", kind="samples", prec="fp64", B=32, **BENCH, **BENCH_KEEP),
        # a serving batch of the 200-sensor array on its 316 x 316 grid (a radix-79 axis), the
        # first 60 steps of an event, complex64, prior on the fly
        dict(name="serve_c64", kind="batch", prec="c64", B=16, Nd=200, Nx=316, Ny=316, Nt=60, Nq=50,
             also="", gstar=False),
        # a small batch of odd size in the bf16 hi+lo storage
        dict(name="batch_bf16x2", kind="batch", prec="bf16x2", B=11, Nd=50, Nx=100, Ny=125, Nt=150, Nq=10,
             also="fp64", gstar=False),
        # the forecast straight from the data
        dict(name="qoi_fp64", kind="qoi", prec="fp64", Nd=50, Nx=60, Ny=75, Nt=120, Nq=10, also="",
             gstar=False),
        # Phase 2 for a new operator: K formed and factored
        dict(name="setup_fp64", kind="setup", prec="fp64", Nd=100, Nx=100, Ny=125, Nt=100, Nq=4, also="",
             gstar=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["event", "event", "batch", "batch", "samples", "apply", "setup"])
    prec = "fp64" if kind in ("apply", "setup") else rng.choice(["fp64", "fp64", "c64", "bf16x2"])
    while True:
        Nd, Nt, Nq = _log_int(rng, 8, 200), _log_int(rng, 32, 420), _log_int(rng, 3, 50)
        Nx, Ny = _log_int(rng, 16, 316), _log_int(rng, 16, 316)
        n, Nm = Nd * Nt, Nx * Ny
        if kind == "setup" and (n > 10_000 or n * n * Nm > 1.25e12):
            continue
        if n * Nm <= 2_000_000_000 and n <= 20_000:
            break
    c = dict(kind=kind, prec=prec, Nd=Nd, Nx=Nx, Ny=Ny, Nt=Nt, Nq=Nq, also="" if prec == "fp64" else "fp64",
             gstar=kind == "event" and prec != "bf16x2" and rng.random() < 0.5)
    if kind == "event":
        c["window"] = rng.randint(max(1, Nt // 5), Nt)
    if kind in ("batch", "samples"):
        most = 64 if kind == "batch" else 32
        c["B"] = min(_log_int(rng, 2, most), max(2, int(most * 2e7 / (Nt * Nm))))
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _points(case, salt):
    """Sensors and forecast points, uniform in the unit square."""
    g = torch.Generator().manual_seed(1000 * salt + case["Nd"] + 7 * case["Nt"] + 13 * case["Nx"])
    s = torch.rand((case["Nd"], 2), generator=g, dtype=torch.float64)
    q = torch.rand((case["Nq"], 2), generator=g, dtype=torch.float64)
    return s.cuda(), q.cuda()


def _grid(case):
    a = torch.arange(case["Nx"], dtype=torch.float64, device="cuda") / case["Nx"]
    b = torch.arange(case["Ny"], dtype=torch.float64, device="cuda") / case["Ny"]
    return torch.stack(torch.meshgrid(a, b, indexing="ij"), -1).reshape(-1, 2)


def _column(case, pts, grid):
    """The block column at these points: [Nt][points][grid]."""
    dt = 1.0 / case["Nt"]
    r = torch.sqrt(((pts[:, None, :] - grid[None, :, :]) ** 2).sum(-1))
    amp = 1.0 / (1.0 + 10.0 * r)
    r = r / 1.5
    out = torch.empty((case["Nt"],) + tuple(r.shape), dtype=torch.float64, device="cuda")
    for i in range(case["Nt"]):
        torch.mul(torch.exp(-(((i * dt - r) / (2.0 * dt)) ** 2)), amp, out=out[i])
    return out


def _spectrum(case):
    """Eigenvalues of the Matern covariance on the periodic grid."""
    kx = torch.fft.fftfreq(case["Nx"], 1.0 / case["Nx"], dtype=torch.float64, device="cuda") * 2 * math.pi
    ky = torch.fft.fftfreq(case["Ny"], 1.0 / case["Ny"], dtype=torch.float64, device="cuda") * 2 * math.pi
    s = (2.0 * NU / ELL ** 2 + kx[:, None] ** 2 + ky[None, :] ** 2) ** (-(NU + 1.0))
    return VAR * s.numel() * s / s.sum()


def _prior(case, x, power):
    """C^power x over the trailing grid axis (FP64)."""
    lam = _spectrum(case) ** power
    f = x.reshape(-1, case["Nx"], case["Ny"])
    out = torch.empty_like(f)
    for i in range(0, f.shape[0], 256):
        out[i:i + 256] = torch.fft.ifft2(torch.fft.fft2(f[i:i + 256]) * lam).real
    return out.reshape(x.shape)


def _sizes(case, sensors, grid):
    """(expected rms of F m under the prior, from a few sensors; the noise's standard deviation)."""
    few = sensors[:: max(1, case["Nd"] // 4)][:4]
    total = 0.0
    left = 1.0 - torch.arange(case["Nt"], dtype=torch.float64, device="cuda") / case["Nt"]
    for p in few:
        g = _prior(case, _column(case, p[None], grid)[:, 0], 0.5)
        total += float(((g * g).sum(1) * left).sum())
    rms = math.sqrt(total / len(few))
    return rms, 0.01 * rms


def _events(case, B, seed, sensors, grid, rms, sigma):
    """Data of B events [B][Nt][Nd]: each a rupture of some grid points with white histories, and noise."""
    Nt, g = case["Nt"], _gen(seed)
    d = torch.empty((B, Nt, case["Nd"]), dtype=torch.float64, device="cuda")
    for b in range(B):
        at = torch.randint(grid.shape[0], (SOURCES,), generator=g, device="cuda")
        z = torch.randn((Nt, SOURCES), generator=g, dtype=torch.float64, device="cuda")
        col = torch.fft.rfft(_column(case, sensors, grid[at]), n=2 * Nt, dim=0)
        x = torch.fft.irfft((col * torch.fft.rfft(z, n=2 * Nt, dim=0)[:, None, :]).sum(2), n=2 * Nt, dim=0)[:Nt]
        d[b] = x * (rms / x.square().mean().sqrt())
    return d + sigma * torch.randn(d.shape, generator=g, dtype=torch.float64, device="cuda")


# ----------------------------------------------------------------- contexts
_held = {}      # the context of the case in hand


def _load(ctx, which, case, pts, grid):
    rows = max(1, min(len(pts), int(3e8 // (case["Nt"] * len(grid)))))
    for r0 in range(0, len(pts), rows):
        ctx.set_block_column(which, r0, _column(case, pts[r0:r0 + rows], grid))


def _context(case):
    """The long-lived context of this case's sizes: operators loaded and, where the kind solves, K factored."""
    key = tuple(case[k] for k in ("Nd", "Nx", "Ny", "Nt", "Nq", "also", "gstar")) + (
        "" if case["gstar"] else case["prec"],)
    if _held.get("key") != key:
        if "ctx" in _held:
            torch.cuda.synchronize()
            _held["ctx"].close()
        _held.clear()
        torch.cuda.empty_cache()
        keep = KEEP[case["prec"]] | (KEEP[case["also"]] if case["also"] else 0) | tw.KEEP_FACTOR64
        keep |= (tw.KEEP_FP64 | tw.KEEP_G) if case["gstar"] else 0
        ctx = tw.Context(case["Nd"], case["Nq"], case["Nx"], case["Ny"], case["Nt"], keep=keep)
        ctx.set_prior(NU, ELL, VAR)
        sensors, qoi = _points(case, 1)
        grid = _grid(case)
        _load(ctx, tw.MAP_F, case, sensors, grid)
        _load(ctx, tw.MAP_FQ, case, qoi, grid)
        rms, sigma = _sizes(case, sensors, grid)
        _held.update(key=key, ctx=ctx, sensors=sensors, grid=grid, rms=rms, sigma=sigma, factored=False)
        torch.cuda.empty_cache()
    h = _held
    if case["kind"] not in ("apply", "setup") and not h["factored"]:
        h["ctx"].factor_K(h["sigma"] ** 2)
        h["factored"] = True
    if case["kind"] in ("batch", "samples", "qoi"):
        B = case.get("B", 32)
        if h["ctx"].batch_capacity() != B:
            h["ctx"].reserve_batch(B)
    if case["kind"] == "qoi" and "qoi" not in h:
        h["ctx"].qoi_build()
        h["qoi"] = True
    return h


def _windows(case, seed):
    g = torch.Generator().manual_seed(seed)
    lo = max(1, case["Nt"] // 4)
    return torch.randint(lo, case["Nt"] + 1, (case["B"],), generator=g, dtype=torch.int32).cuda()


def _data(case, seed, sensors, grid, rms, sigma):
    kind, g = case["kind"], _gen(seed + 1_000_003)
    if kind == "apply":
        return {"x": torch.randn((1, case["Nt"], case["Nx"] * case["Ny"]), generator=g, dtype=torch.float64,
                                 device="cuda")}
    s = {"d": _events(case, case.get("B", 1) if kind == "batch" else 1, seed, sensors, grid, rms, sigma)}
    if kind in ("batch", "samples"):
        s["windows"] = _windows(case, seed)
    if kind == "samples":
        B = case["B"]
        s["d"] = s["d"].expand(B, -1, -1).contiguous()       # samples of one event
        s["z_m"] = torch.randn((B, case["Nt"], case["Nx"] * case["Ny"]), generator=g, dtype=torch.float64,
                               device="cuda")
        s["z_n"] = torch.randn(s["d"].shape, generator=g, dtype=torch.float64, device="cuda")
        s["sigma"] = sigma
    return s


def _setup_operator(case, seed):
    sensors, _ = _points(case, 2 + seed % 1_000_000)
    grid = _grid(case)
    rms, sigma = _sizes(case, sensors, grid)
    return sensors, grid, rms, sigma


def prepare(case, seed):
    s = {"case": case, "prec": PREC[case["prec"]]}
    if case["kind"] == "setup":
        sensors, grid, rms, sigma = _setup_operator(case, seed)
        ctx = tw.Context(case["Nd"], case["Nq"], case["Nx"], case["Ny"], case["Nt"], keep=tw.KEEP_FP64)
        ctx.set_prior(NU, ELL, VAR)
        s.update(ctx=ctx, col=_column(case, sensors, grid), noise_var=sigma ** 2)
    else:
        h = _context(case)
        s["ctx"] = h["ctx"]
        sensors, grid, rms, sigma = h["sensors"], h["grid"], h["rms"], h["sigma"]
    s.update(_data(case, seed, sensors, grid, rms, sigma))
    return s


def run(s):
    case, ctx, prec = s["case"], s["ctx"], s["prec"]
    kind = case["kind"]
    if kind == "event":
        return ctx.infer_forecast(prec, s["d"], windows=[case["window"]])
    if kind == "batch":
        return ctx.infer_batch(prec, s["d"], s["windows"])
    if kind == "samples":
        return ctx.sample_posterior_batch(prec, s["d"], s["z_m"], s["z_n"], s["sigma"], s["windows"])
    if kind == "apply":
        d = ctx.p2o_apply(tw.MAP_F, prec, s["x"])
        return d, ctx.p2o_adjoint(tw.MAP_F, prec, d)
    if kind == "qoi":
        return ctx.qoi_apply(s["d"])
    ctx.set_block_column(tw.MAP_F, 0, s["col"])
    ctx.factor_K(s["noise_var"])
    return ctx.solve_K(prec, s["d"])


def work(case):
    """Bytes: the kept operators that the path multiplies by, the factor once a sweep, inputs and outputs.
    Flops: those of the products, solves and transforms (8 a complex multiply-add)."""
    Nd, Nq, Nt, Nm = case["Nd"], case["Nq"], case["Nt"], case["Nx"] * case["Ny"]
    Nf, n, kind = Nt + 1, Nd * Nt, case["kind"]
    el = 16 if case["prec"] == "fp64" else 8
    B = case.get("B", 1)
    fft = 5.0 * Nt * math.log2(2 * Nt) * Nm                      # a real transform of length 2 Nt a grid point
    filt = 2 * 2.5 * Nm * math.log2(Nm) * Nt                     # the prior, there and back
    if kind == "apply":
        return {"bytes": 2 * el * Nf * Nd * Nm + 8 * Nt * (2 * Nm + Nd), "flops": 16.0 * Nf * Nd * Nm + 2 * fft}
    if kind == "qoi":
        return {"bytes": 8 * Nq * Nt * n + 8 * (n + Nq * Nt), "flops": 2.0 * Nq * Nt * n}
    if kind == "setup":
        return {"bytes": 8 * n * Nm + 8 * n * (n + 1) // 2 + 16 * n, "flops": 1.0 * n * n * Nm + n ** 3 / 3 + 2.0 * n * n}
    nw = Nd * (case["window"] if kind == "event" else Nt * 5 // 8)    # rows a solve takes; batches: on average
    top = nw if kind == "event" else n                                # the factor's rows that some solve takes
    b = el * Nf * Nd * Nm + 2 * 8 * top * (top + 1) // 2 + B * 8 * (n + Nt * Nm)
    f = B * (8.0 * Nf * Nd * Nm + 2.0 * nw * nw + fft + (0 if case["gstar"] else filt))
    if kind == "samples":
        b += el * Nf * Nd * Nm * (2 if case["gstar"] else 1) + B * 8 * (Nt * Nm + n)   # F as well as G*; the draws
        f += B * (8.0 * Nf * Nd * Nm + fft + filt)
    else:
        b += el * Nf * Nq * Nm + B * 8 * Nq * Nt
        f += B * (8.0 * Nf * Nq * Nm + fft)
    return {"bytes": int(b), "flops": f}


# ------------------------------------------------------------- 64-bit values
def _toeplitz(case, pts, grid, x, adjoint):
    """F x ([B][Nt][Nm] -> [B][Nt][points]) or F^T x, some rows of F at a time."""
    Nt, B = case["Nt"], x.shape[0]
    out = torch.zeros((B, Nt, len(grid) if adjoint else len(pts)), dtype=torch.float64, device="cuda")
    rows = max(1, min(len(pts), int(1e8 // (Nt * len(grid)))))
    xh = torch.fft.rfft(x, n=2 * Nt, dim=1)
    acc = torch.zeros((B, Nt + 1, len(grid)), dtype=torch.complex128, device="cuda") if adjoint else None
    for r0 in range(0, len(pts), rows):
        Fh = torch.fft.rfft(_column(case, pts[r0:r0 + rows], grid), n=2 * Nt, dim=0)
        for b in range(B):
            if adjoint:
                for i in range(Fh.shape[1]):
                    acc[b] += Fh[:, i].conj() * xh[b, :, r0 + i, None]
            else:
                y = torch.stack([(Fh[:, i] * xh[b]).sum(1) for i in range(Fh.shape[1])], 1)
                out[b, :, r0:r0 + Fh.shape[1]] = torch.fft.irfft(y, n=2 * Nt, dim=0)[:Nt]
        del Fh
    if adjoint:
        for b in range(B):
            out[b] = torch.fft.irfft(acc[b], n=2 * Nt, dim=0)[:Nt]
    return out


def _factor(case, sensors, grid, sigma):
    """The lower Cholesky factor of K, formed from dense products."""
    Nd, Nt, n = case["Nd"], case["Nt"], case["Nd"] * case["Nt"]
    G = _prior(case, _column(case, sensors, grid), 0.5).reshape(n, -1)
    K = (G @ G.T).reshape(Nt, Nd, Nt, Nd)
    del G
    for i in range(1, Nt):
        K[i, :, 1:, :] += K[i - 1, :, :-1, :]
    K = K.reshape(n, n)
    K.diagonal().add_(sigma ** 2)
    return torch.linalg.cholesky(K)


def _solve(L, d, w, Nd):
    n = Nd * w
    y = torch.zeros_like(d)
    y.view(-1)[:n] = torch.cholesky_solve(d.reshape(-1)[:n, None], L[:n, :n])[:, 0]
    return y


def exact(case, seed):
    """`run`'s outputs in plain 64-bit torch.  The dense K bounds the sizes: None beyond some seconds' work."""
    kind, Nd, Nt, Nm = case["kind"], case["Nd"], case["Nt"], case["Nx"] * case["Ny"]
    n, B = Nd * Nt, case.get("B", 1)
    if kind == "apply":
        if Nm * n > 2.1e9:
            return None
    elif n * n * Nm > 1.3e12 or n * Nm > 4e8 or B * n * Nm > 2e9 or n > 12_000:
        return None
    if kind == "setup":
        sensors, grid, rms, sigma = _setup_operator(case, seed)
    else:
        (sensors, qoi), grid = _points(case, 1), _grid(case)
        rms, sigma = _sizes(case, sensors, grid)
    s = _data(case, seed, sensors, grid, rms, sigma)
    if kind == "apply":
        d = _toeplitz(case, sensors, grid, s["x"], False)
        return d, _toeplitz(case, sensors, grid, d, True)
    L = _factor(case, sensors, grid, sigma)
    if kind == "setup":
        return _solve(L, s["d"], Nt, Nd)
    win = [case["window"]] if kind == "event" else [Nt] if kind == "qoi" else s["windows"].tolist()
    y, prior = s["d"], None
    if kind == "samples":
        prior = _prior(case, s["z_m"], 0.5)
        y = y - _toeplitz(case, sensors, grid, prior, False) - sigma * s["z_n"]
    y = torch.cat([_solve(L, y[b:b + 1], w, Nd) for b, w in enumerate(win)])
    m = _toeplitz(case, sensors, grid, y, True)
    m = _prior(case, m, 1.0)
    for b, w in enumerate(win):
        m[b, w:] = 0.0
    if kind == "samples":
        return prior + m
    q = _toeplitz(case, qoi, grid, m, False)
    return q if kind == "qoi" else (m, q)
