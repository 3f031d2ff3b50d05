"""Timed cases of the resolvent march: what a user of the library has it do, through its Python entry points.

A case is a dict of plain values.  "system" names the operator kind and "call" the entry point:

  march      rsv_march_direct / rsv_march_adjoint of a block of Fourier coefficients (SSRM or TRM)
  rsvd       rsv_gains_modes: a whole randomized SVD (marches, per-frequency QR, gains and modes)
  refine     rsv_refine_gains: the Rayleigh-Ritz pass on a given basis
  qr         rsv_orthonormalize of a response block (out of place: the block is copied first)
  series     rsv_series_march: one run driven by a sampled series (C2 interpolation)

`exact` restates the method (frequency grid, RK4 or Crank-Nicolson step, forcing sums, rectangle-rule Fourier
sums) in plain torch FP64.
"""
import math

import numpy as np
import torch

from paper_2008_10904_gb300 import rsv

DEV = "cuda"


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _case(name, call, system, prec, **kw):
    c = dict(name=name, call=call, system=system, prec=prec, adjoint=False, variant="ssrm", trans=0, tail=0, k=1,
             n_omega=8, w0=0.0, w1=1.0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a coarse Ginzburg-Landau model being set up and tried out (one warp of points)
        _case("gl_n24_small_fp64", "march", "gl", "fp64", sizes="24", x_half=20.0, mu0=0.1, dt=0.05, k=2, n_omega=8,
              w0=-1.0, w1=1.0, trans=1),
        # the plain method on the FP64 model problem: one march of the power iteration
        _case("gl_n256_k4_w32_fp64", "march", "gl", "fp64", sizes="256", x_half=85.0, mu0=0.23, dt=0.02, k=4,
              n_omega=32, w0=-1.5, w1=1.5, trans=4),
        # gains and modes of the same model in one call
        _case("gl_n256_rsvd_fp64", "rsvd", "gl", "fp64", sizes="256", x_half=85.0, mu0=0.23, dt=0.02, k=4,
              n_omega=32, w0=-1.5, w1=1.5, trans=1, q=1, n_modes=3),
        # a parameter study: 64 models of uneven sizes in one launch
        _case("gl_batch64_k8_w32_fp32", "march", "gl", "fp32", sizes="batch64", x_half=85.0, mu0=0.2, dt=0.003, k=8,
              n_omega=32, w0=-3.0, w1=3.0),
        # the paper's validation case: Crank-Nicolson, real coefficients, mu linear in x; the adjoint run
        _case("gl_paper_n400_cn_fp64", "march", "gl", "fp64", sizes="400", paper=True, cn=True, dt=0.01, k=4,
              n_omega=61, w0=0.0, w1=15.0, adjoint=True),
        # a dense spectral operator by the transient-response method: one forced window and a decay tail
        _case("dense_n1024_k32_w32_trm_fp32", "march", "dense", "fp32", n=1024, dt=0.005, k=32, n_omega=32, w0=-2.0,
              w1=2.0, variant="trm", tail=2000),
        # a planar jet on the production grid: the march of a block of test vectors
        _case("adr2d_1024x512_k16_w32_fp32", "march", "adr2d", "fp32", nx=1024, ny=512, k=16, n_omega=32, w0=0.0,
              w1=4.0),
        # the FP64 refinement pass of a coarser, odd-sized jet
        _case("adr2d_401x203_refine_fp64", "refine", "adr2d", "fp64", nx=401, ny=203, k=6, n_omega=16, w0=0.0, w1=4.0,
              trans=1, n_modes=3),
        # one run of the time-series method: a recorded adjoint run's forcing, reversed in time
        _case("adr2d_256x128_series_fp32", "series", "adr2d", "fp32", nx=256, ny=128, k=4, n_omega=8, w0=0.0, w1=4.0,
              every=4, n_in=96, n_out=192, adjoint=True),
        # a 3-D boundary layer on the production grid: the largest call
        _case("adv3d_256x128x128_w32_fp32", "march", "adv3d", "fp32", nx=256, ny=128, nz=128, k=1, n_omega=32, w0=0.0,
              w1=2.48 * math.pi),
        # an odd-sized 3-D grid, the adjoint half of the power iteration
        _case("adv3d_97x61x43_k3_adj_fp32", "march", "adv3d", "fp32", nx=97, ny=61, nz=43, k=3, n_omega=12, w0=0.0,
              w1=1.76 * math.pi, trans=2, adjoint=True),
        # per-frequency QR of a 2-D response block between two marches
        _case("qr_adr2d_k16_w16_fp32", "qr", "adr2d", "fp32", nx=512, ny=512, k=16, n_omega=16, w0=0.0, w1=4.0),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["small", "gl64", "rsvd", "batch", "cn", "dense", "adr2d", "refine", "series", "adv3d", "adv3d", "qr"])
    adj = rng.random() < 0.5
    if kind == "small":
        n = _log_int(rng, 16, 120)
        return _unnamed("march", "gl", rng.choice(["fp64", "fp32"]), sizes=str(n), x_half=20.0, mu0=0.1,
                        dt=min(0.05, _gl_dt(n, 20.0)), k=rng.randint(1, 4), n_omega=rng.randint(4, 12), w0=-1.0, w1=1.0,
                        trans=rng.randint(0, 1), adjoint=adj)
    if kind == "gl64":
        n = _log_int(rng, 200, 512)
        return _unnamed("march", "gl", "fp64", sizes=str(n), x_half=85.0, mu0=0.15, dt=_gl_dt(n, 85.0),
                        k=rng.randint(1, 8), n_omega=rng.randint(12, 32), w0=-1.5, w1=1.5, trans=rng.randint(0, 2), adjoint=adj)
    if kind == "rsvd":
        n = _log_int(rng, 128, 320)
        return _unnamed("rsvd", "gl", "fp64", sizes=str(n), x_half=60.0, mu0=0.15, dt=min(0.02, _gl_dt(n, 60.0)),
                        k=rng.randint(4, 6), n_omega=rng.randint(8, 24), w0=-1.5, w1=1.5, trans=rng.randint(1, 2), q=1, n_modes=2)
    if kind == "batch":
        sizes = [_log_int(rng, 200, 2048) for _ in range(rng.randint(3, 40))]
        return _unnamed("march", "gl", "fp32", sizes=",".join(map(str, sizes)), x_half=85.0, mu0=0.15,
                        dt=_gl_dt(max(sizes), 85.0), k=rng.randint(1, 8), n_omega=rng.randint(8, 24), w0=-3.0, w1=3.0, adjoint=adj)
    if kind == "cn":
        return _unnamed("march", "gl", rng.choice(["fp64", "fp64", "fp32"]), sizes=str(_log_int(rng, 100, 700)), paper=True, cn=True,
                        dt=rng.choice([0.01, 0.02]), k=rng.randint(1, 4), n_omega=rng.randint(13, 61), w0=0.0, w1=15.0, adjoint=adj)
    if kind == "dense":
        return _unnamed("march", "dense", "fp32", n=rng.choice([192, 256, 384, 512, 1024]), dt=0.005, k=rng.randint(2, 32),
                        n_omega=rng.randint(12, 28), w0=-2.0, w1=2.0, variant="trm", tail=rng.randint(300, 1500), adjoint=adj)
    if kind == "adr2d":
        return _unnamed("march", "adr2d", "fp32", nx=_log_int(rng, 100, 1024), ny=_log_int(rng, 60, 512), k=rng.randint(1, 12),
                        n_omega=rng.randint(8, 32), w0=0.0, w1=4.0, trans=rng.randint(0, 1), adjoint=adj)
    if kind == "refine":
        return _unnamed("refine", "adr2d", "fp64", nx=_log_int(rng, 90, 400), ny=_log_int(rng, 60, 200), k=rng.randint(3, 6),
                        n_omega=rng.randint(8, 16), w0=0.0, w1=4.0, trans=rng.randint(0, 1), n_modes=2)
    if kind == "series":
        every = rng.randint(2, 6)
        return _unnamed("series", "adr2d", "fp32", nx=_log_int(rng, 100, 300), ny=_log_int(rng, 60, 150), k=rng.randint(1, 4),
                        n_omega=8, w0=0.0, w1=4.0, every=every, n_in=rng.randint(30, 96), n_out=rng.randint(97, 180), adjoint=adj)
    if kind == "adv3d":
        n_omega = rng.randint(8, 24)
        return _unnamed("march", "adv3d", "fp32", nx=_log_int(rng, 48, 200), ny=_log_int(rng, 32, 110), nz=_log_int(rng, 32, 110),
                        k=rng.randint(1, 2), n_omega=n_omega, w0=0.0, w1=0.08 * math.pi * (n_omega - 1), trans=rng.randint(0, 1),
                        adjoint=adj)
    return _unnamed("qr", "adr2d", rng.choice(["fp32", "fp32", "fp64"]), nx=_log_int(rng, 100, 512), ny=_log_int(rng, 60, 400),
                    k=rng.randint(2, 16), n_omega=rng.randint(2, 16), w0=0.0, w1=4.0)


def _unnamed(call, system, prec, **kw):
    c = _case("", call, system, prec, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# System parameters
# ---------------------------------------------------------------------------
def _gl_dt(n, x_half):
    """RK4 step for n points on (-x_half, x_half): h * 4 |gamma| / dx^2 = 2.4 at most."""
    dx = 2 * x_half / (n + 1)
    return min(0.02, 2.4 * dx * dx / (4 * math.sqrt(2.0)))


def _sizes(c):
    if c["sizes"] == "batch64":   # 64 instances, log-uniform in [256, 2048]
        rng = np.random.default_rng(64)
        return [int(round(v)) for v in np.exp(rng.uniform(math.log(256), math.log(2048), size=64))]
    return [int(s) for s in c["sizes"].split(",")]


def _gl_params(c):
    if c.get("paper"):
        return dict(x0=0.0, x1=40.0, nu=6.0 + 0j, gamma=1.0 + 0j, mu0=3.6, mu_shift=0.0, mu1=-0.18, mu2=0.0)
    return dict(x0=-c["x_half"], x1=c["x_half"], nu=2.0 + 0.4j, gamma=1.0 - 1.0j, mu0=c["mu0"], mu_shift=-0.04, mu1=0.0, mu2=-0.005)


def _dense_matrix(n):
    """Ginzburg-Landau operator by sinc collocation at n equispaced points on (-85, 85)."""
    x = np.linspace(-85.0, 85.0, n)
    d = x[1] - x[0]
    i = np.arange(n)
    diff = (i[:, None] - i[None, :]).astype(np.float64)
    np.fill_diagonal(diff, 1.0)
    sgn = np.where((i[:, None] - i[None, :]) % 2 == 0, 1.0, -1.0)
    d1 = sgn / diff / d
    d2 = -2.0 * sgn / diff ** 2 / d ** 2
    np.fill_diagonal(d1, 0.0)
    np.fill_diagonal(d2, -math.pi ** 2 / 3 / d ** 2)
    return -(2.0 + 0.4j) * d1 + (1.0 - 1.0j) * d2 + np.diag(0.19 - 0.005 * x ** 2)


def _dense_dt(c):
    """RK4 step inside the stability region: the largest wavenumber is pi / dx."""
    dx = 170.0 / (c["n"] - 1)
    return min(c["dt"], 2.2 / (math.sqrt(2.0) * (math.pi / dx) ** 2))


def _dims(c):
    """Points per vector and whether the state is real."""
    if c["system"] == "gl":
        return sum(_sizes(c)), False
    if c["system"] == "dense":
        return c["n"], False
    if c["system"] == "adr2d":
        return c["nx"] * c["ny"], True
    return 3 * c["nx"] * c["ny"] * c["nz"], True


def _dt(c):
    if c["system"] == "adr2d":
        return 0.5 * 40.0 / (c["nx"] + 1)
    if c["system"] == "adv3d":
        return 0.5 * 20.0 / (c["nx"] + 1)
    return _dense_dt(c) if c["system"] == "dense" else c["dt"]


def _omegas(c):
    m = c["n_omega"]
    return np.array([c["w0"] + (c["w1"] - c["w0"]) * j / (m - 1) for j in range(m)])


def _grid(c):
    """Steps per window and the step h."""
    period = 2 * math.pi * (c["n_omega"] - 1) / (c["w1"] - c["w0"])
    nt = int(math.ceil(period / _dt(c) - 1e-9))
    return nt, period / nt


def _operator(c):
    prec = rsv.RSV_PREC_FP64 if c["prec"] == "fp64" else rsv.RSV_PREC_FP32
    keep = []
    if c["system"] == "dense":
        d, keep = rsv.desc_dense(_dense_matrix(c["n"]), _dt(c), prec)
    else:
        d = rsv.rsv_operator_desc()
        d.precision, d.dt = prec, _dt(c)
        d.scheme = rsv.RSV_SCHEME_CN if c.get("cn") else rsv.RSV_SCHEME_RK4
    if c["system"] == "gl":
        p = _gl_params(c)
        n = np.array(_sizes(c), dtype=np.int32)
        mu0 = np.full(len(n), p["mu0"])
        keep = [n, mu0]
        d.kind, d.n_instances = rsv.RSV_OP_GL1D, len(n)
        d.gl_n = n.ctypes.data_as(type(d.gl_n))
        d.gl_mu0 = mu0.ctypes.data_as(type(d.gl_mu0))
        d.x0, d.x1 = p["x0"], p["x1"]
        d.nu_re, d.nu_im, d.gamma_re, d.gamma_im = p["nu"].real, p["nu"].imag, p["gamma"].real, p["gamma"].imag
        d.mu_shift, d.mu1, d.mu2 = p["mu_shift"], p["mu1"], p["mu2"]
    elif c["system"] == "adr2d":
        d.kind, d.nx, d.ny = rsv.RSV_OP_ADR2D, c["nx"], c["ny"]
        d.lx, d.ly, d.visc, d.kappa, d.jet_delta, d.sponge_amp, d.sponge_cells = 40.0, 10.0, 1e-3, 0.01, 0.05, 1.0, 32
    elif c["system"] == "adv3d":
        d.kind, d.nx, d.ny, d.nz = rsv.RSV_OP_ADV3D, c["nx"], c["ny"], c["nz"]
        d.lx, d.ly, d.lz, d.visc, d.delta0, d.delta1 = 20.0, 10.0, 10.0, 5e-4, 0.2, 1.0
    op = rsv.rsv_create_operator(d, None, keep)
    rsv.rsv_set_frequencies(op, _omegas(c))
    return op


# ---------------------------------------------------------------------------
# Inputs, one pass, work
# ---------------------------------------------------------------------------
class _State:
    """The operator (freed with the state), the input and the output buffers of one case."""

    def __init__(self, case):
        self.case = case
        self.op = _operator(case)

    def __del__(self):
        if getattr(self, "op", None) is not None:
            rsv.rsv_destroy_operator(self.op)


def _types(c):
    return (torch.float64, torch.complex128) if c["prec"] == "fp64" else (torch.float32, torch.complex64)


def _input(c, seed):
    """Gaussian test vectors [n_omega][k][n] (real in the w = 0 row of a real state), or a band-limited series."""
    rt, ct = _types(c)
    n, real = _dims(c)
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    if c["call"] == "series":
        # a few random fields in k vectors, modulated in time as a wave packet is
        t = torch.arange(c["n_in"], device=DEV, dtype=torch.float64) / c["n_in"]
        out = torch.zeros(c["n_in"], c["k"], n, device=DEV, dtype=rt)
        for m in range(4):
            field = torch.randn(c["k"], n, device=DEV, dtype=rt, generator=g)
            out += (torch.sin(math.pi * t) ** 2 * torch.cos(2 * math.pi * (m + 1) * t + m)).to(rt)[:, None, None] * field
        return out
    f = torch.randn(c["n_omega"], c["k"], n, device=DEV, dtype=ct, generator=g)
    if real:
        for j in np.nonzero(_omegas(c) == 0.0)[0]:
            f[int(j)] = torch.randn(c["k"], n, device=DEV, dtype=rt, generator=g).to(ct)
    return f


def prepare(case, seed):
    s = _State(case)
    _, ct = _types(case)
    n, real = _dims(case)
    s.f = _input(case, seed)
    if case["call"] == "series":
        s.out = torch.zeros(case["n_out"], case["k"], n, device=DEV, dtype=s.f.dtype)
    elif case["call"] in ("rsvd", "refine"):
        s.gains = np.zeros((1, case["n_omega"], case["n_modes"]))
        s.fm = torch.empty(case["n_omega"], case["n_modes"], n, device=DEV, dtype=ct)
        s.rm = torch.empty_like(s.fm)
    else:
        s.out = torch.empty_like(s.f)
    s.opts = dict(variant=case["variant"], n_transient_windows=case["trans"], tail_steps=case["tail"])
    return s


def run(s):
    c = s.case
    if c["call"] == "march":
        march = rsv.rsv_march_adjoint if c["adjoint"] else rsv.rsv_march_direct
        march(s.op, s.f, c["k"], s.out, **s.opts)
        return s.out
    if c["call"] == "rsvd":
        rsv.rsv_gains_modes(s.op, s.f, c["k"], c["q"], c["n_modes"], s.gains, s.fm, s.rm, **s.opts)
        return {"gains": s.gains, "forcing": s.fm, "response": s.rm}
    if c["call"] == "refine":
        rsv.rsv_refine_gains(s.op, s.f, c["k"], c["n_modes"], s.gains, s.fm, s.rm, **s.opts)
        return {"gains": s.gains, "forcing": s.fm, "response": s.rm}
    if c["call"] == "qr":
        s.out.copy_(s.f)
        r = np.zeros((c["n_omega"], 1, c["k"], c["k"]), dtype=np.complex128)
        rsv.rsv_orthonormalize(s.op, s.out, c["k"], r)
        return {"q": s.out, "r": r}
    n_out, _ = rsv.rsv_series_march(s.op, c["adjoint"], c["k"], s.out, c["n_out"], forcing=s.f, n_in=c["n_in"],
                                    reverse_in=True, every=c["every"], interp="c2")
    return s.out


def work(case):
    """Bytes: inputs read and outputs written once.  Flops: the operator in the four stages (two products per
    Crank-Nicolson step), one forcing sum per step, one Fourier sum per analysed step, QR and Gram products."""
    c = case
    n, real = _dims(c)
    rows = c["k"] * n
    esz = 8 if c["prec"] == "fp64" else 4
    nt, _ = _grid(c)
    block = c["n_omega"] * rows * 2 * esz
    cmul = 8 * c["n_omega"] * rows // (2 if real else 1)          # one Fourier sum over the block
    qr = 2 * 16 * c["n_omega"] * rows * c["k"]                     # two Gram and two triangular products
    if c["call"] == "qr":
        return {"bytes": 2 * block, "flops": qr}
    stage = {"gl": 24, "dense": 8 * c.get("n", 0), "adr2d": 10, "adv3d": 15}[c["system"]]
    per_step = (1 if c["system"] == "dense" else 2 if c.get("cn") else 4) * stage * rows
    if c["call"] == "series":
        return {"bytes": (c["n_in"] + c["n_out"]) * rows * esz, "flops": (c["n_out"] - 1) * c["every"] * per_step}
    total = nt + c["tail"] if c["variant"] == "trm" else (c["trans"] + 1) * nt
    forced = nt if c["variant"] == "trm" else total
    analysed = total if c["variant"] == "trm" else nt
    march = total * per_step + forced * cmul + analysed * cmul
    if c["call"] == "rsvd":
        return {"bytes": block + 2 * block * c["n_modes"] // c["k"], "flops": 2 * (c["q"] + 1) * march + (2 * c["q"] + 1) * qr}
    if c["call"] == "refine":
        return {"bytes": block + 2 * block * c["n_modes"] // c["k"], "flops": march + qr}
    return {"bytes": 2 * block, "flops": march}


# ---------------------------------------------------------------------------
# The same results in FP64
# ---------------------------------------------------------------------------
def _exact_operator(c, adjoint):
    """x -> A x (A^H x) on [..., n] FP64 tensors, in plain torch."""
    if c["system"] == "gl":
        p, lo, di, up = _gl_params(c), [], [], []
        for n in _sizes(c):
            dx = (p["x1"] - p["x0"]) / (n + 1)
            x = p["x0"] + dx * np.arange(1, n + 1)
            a = np.full(n, p["nu"] / (2 * dx) + p["gamma"] / dx ** 2)
            b = np.full(n, -p["nu"] / (2 * dx) + p["gamma"] / dx ** 2)
            a[0] = b[-1] = 0.0
            d = -2.0 * p["gamma"] / dx ** 2 + p["mu0"] + p["mu_shift"] + p["mu1"] * x + p["mu2"] * x * x
            if adjoint:
                a, b, d = np.concatenate([[0], np.conj(b[:-1])]), np.concatenate([np.conj(a[1:]), [0]]), np.conj(d)
            lo.append(a)
            up.append(b)
            di.append(d)
        lo, di, up = (torch.tensor(np.concatenate(v), device=DEV) for v in (lo, di, up))

        def apply(u):
            y = di * u
            y[..., 1:] += lo[1:] * u[..., :-1]
            y[..., :-1] += up[:-1] * u[..., 1:]
            return y
        return apply
    if c["system"] == "dense":
        a = torch.tensor(_dense_matrix(c["n"]), device=DEV)
        a = a.conj().T.contiguous() if adjoint else a
        return lambda u: u @ a.T
    if c["system"] == "adr2d":
        nx, ny = c["nx"], c["ny"]
        dx, dy, nu = 40.0 / (nx + 1), 10.0 / (ny + 1), 1e-3
        y = torch.arange(1, ny + 1, device=DEV, dtype=torch.float64) * dy - 5.0
        arg = (0.5 - y.abs()) / 0.05
        U = 0.5 * (1 + torch.tanh(arg))
        r = -0.01 * (0.5 / torch.cosh(arg) ** 2 * (-torch.sign(y) / 0.05))
        i, j = torch.arange(nx, device=DEV), torch.arange(ny, device=DEV)
        d = torch.minimum(torch.minimum(i, nx - 1 - i)[None, :], torch.minimum(j, ny - 1 - j)[:, None])
        sponge = torch.where(d < 32, ((32 - d) / 32.0) ** 2, torch.zeros((), device=DEV, dtype=torch.float64))
        ux = (-U if adjoint else U)[:, None]
        cw, ce, cc = ux / (2 * dx) + nu / dx ** 2, -ux / (2 * dx) + nu / dx ** 2, -2 * nu * (1 / dx ** 2 + 1 / dy ** 2) + r[:, None] - sponge

        def apply(u):
            v = u.reshape(*u.shape[:-1], ny, nx)
            o = cc * v
            o[..., :, 1:] += cw * v[..., :, :-1]
            o[..., :, :-1] += ce * v[..., :, 1:]
            o[..., 1:, :] += nu / dy ** 2 * v[..., :-1, :]
            o[..., :-1, :] += nu / dy ** 2 * v[..., 1:, :]
            return o.reshape(u.shape)
        return apply
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    dx, dy, dz, nu = 20.0 / (nx + 1), 10.0 / (ny + 1), 10.0 / (nz + 1), 5e-4
    ax = lambda m, d, o: torch.arange(1, m + 1, device=DEV, dtype=torch.float64) * d + o  # noqa: E731
    x, y, z = ax(nx, dx, 0.0)[None, None, :], ax(ny, dy, -5.0)[None, :, None], ax(nz, dz, -5.0)[:, None, None]
    dd = 0.8 / 20.0
    de, r = 0.2 + dd * x, torch.sqrt(y * y + z * z)
    gg = 2.0 / math.sqrt(math.pi) * torch.exp(-(r / de) ** 2)
    U = torch.erf(r / de)
    inv = torch.where(r > 0, 1.0 / torch.where(r > 0, r, 1.0), 0.0)
    grad = (gg * (-r * dd / de ** 2), gg * y * inv / de, gg * z * inv / de)

    def apply(u):
        v = u.reshape(*u.shape[:-1], 3, nz, ny, nx)
        o = -2.0 * nu * (1 / dx ** 2 + 1 / dy ** 2 + 1 / dz ** 2) * v
        w, e = v[..., :-1], v[..., 1:]
        if adjoint:   # (A^T x)_p = (U_{p+1} x_{p+1} - U_{p-1} x_{p-1}) / (2 dx)
            o[..., 1:] += (nu / dx ** 2 - U[..., :-1] / (2 * dx)) * w
            o[..., :-1] += (nu / dx ** 2 + U[..., 1:] / (2 * dx)) * e
        else:
            o[..., 1:] += (nu / dx ** 2 + U[..., 1:] / (2 * dx)) * w
            o[..., :-1] += (nu / dx ** 2 - U[..., :-1] / (2 * dx)) * e
        o[..., 1:, :] += nu / dy ** 2 * v[..., :-1, :]
        o[..., :-1, :] += nu / dy ** 2 * v[..., 1:, :]
        o[..., 1:, :, :] += nu / dz ** 2 * v[..., :-1, :, :]
        o[..., :-1, :, :] += nu / dz ** 2 * v[..., 1:, :, :]
        for a in range(3):
            if adjoint:
                o[..., a, :, :, :] -= grad[a] * v[..., 0, :, :, :]
            else:
                o[..., 0, :, :, :] -= grad[a] * v[..., a, :, :, :]
        return o.reshape(u.shape)
    return apply


def _exact_step(c, adjoint, h):
    """(u, f(t), f(t + h/2), f(t + h)) -> the state after one step."""
    A = _exact_operator(c, adjoint)
    if c["system"] == "dense" or c.get("cn"):   # the step's matrices, formed once
        n = _dims(c)[0]
        eye = torch.eye(n, device=DEV, dtype=torch.complex128)
        B = h * A(eye)                             # row i of B: h A e_i, so u -> u @ B is h A u
        if c.get("cn"):
            inv = torch.linalg.inv(eye - 0.5 * B)
            P, Q = (eye + 0.5 * B) @ inv, 0.5 * h * inv
            return lambda u, f0, fh, f1: u @ P + (f0 + f1) @ Q
        B2 = B @ B
        B3 = B2 @ B
        M = eye + B + B2 / 2 + B3 / 6 + B3 @ B / 24
        P1, P2 = h / 6 * (eye + B + B2 / 2 + B3 / 4), h / 6 * (4 * eye + 2 * B + B2 / 2)
        return lambda u, f0, fh, f1: u @ M + (f0 @ P1 + fh @ P2 + h / 6 * f1 if f0 is not None else 0)

    def step(u, f0, fh, f1):
        f0, fh, f1 = (0 if f is None else f for f in (f0, fh, f1))
        k1 = A(u) + f0
        k2 = A(u + 0.5 * h * k1) + fh
        k3 = A(u + 0.5 * h * k2) + fh
        k4 = A(u + h * k3) + f1
        return u + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
    return step


def _exact_march(c, f, adjoint):
    """Fourier coefficients of the response to f [n_omega][k][n] (complex128), by the plain march."""
    _, real = _dims(c)
    nt, h = _grid(c)
    sgn = -1.0 if adjoint else 1.0
    step = _exact_step(c, adjoint, h)
    w = torch.tensor(_omegas(c), device=DEV)
    j = torch.arange(c["n_omega"], device=DEV)
    m = w.numel()
    dw = (c["w1"] - c["w0"]) / (m - 1)
    p2 = torch.round(2 * (c["w0"] / dw + j)).to(torch.int64)       # 2 w_j / dw, an integer
    def twiddle(q):                                                # exp(i w_j q h / 2) for integer half steps q
        ph = torch.remainder(p2[None, :] * q[:, None], 4 * nt).to(torch.float64) * (math.pi / (2 * nt))
        return torch.polar(torch.ones_like(ph), sgn * ph)
    total = nt + c["tail"] if c["variant"] == "trm" else (c["trans"] + 1) * nt
    forced = nt if c["variant"] == "trm" else total
    first = 0 if c["variant"] == "trm" else total - nt
    flat = f.reshape(m, -1)
    if real:
        weight = torch.where(w == 0, 1.0, 2.0).to(torch.float64)
        flat = torch.cat([flat.real, flat.imag])
    u = torch.zeros(f.shape[1:], device=DEV, dtype=torch.float64 if real else torch.complex128)
    acc = torch.zeros(m, u.numel(), device=DEV, dtype=torch.complex128)
    S = max(4, min(64, int(2e8 // u.numel())))
    for n0 in range(0, total, S):
        ns = min(S, total - n0)
        F = None
        if n0 < forced:
            T = twiddle(torch.arange(2 * n0, 2 * (n0 + ns) + 1, device=DEV))
            T = torch.cat([weight * T.real, -weight * T.imag], 1) if real else T
            F = (T @ flat).reshape(-1, *u.shape)
        ys = []
        for s in range(ns):
            if n0 + s >= first:
                ys.append(u)
            on = F is not None and n0 + s < forced
            u = step(u, *((F[2 * s], F[2 * s + 1], F[2 * s + 2]) if on else (None,) * 3))
        if ys:
            n1 = n0 + ns
            E = twiddle(2 * torch.arange(n1 - len(ys), n1, device=DEV)).conj().T
            Y = torch.stack(ys).reshape(len(ys), -1)
            acc += torch.complex(E.real @ Y, E.imag @ Y) if real else E @ Y
    return (acc / nt).reshape(f.shape)


def _exact_series(c, g):
    """Snapshots of the run forced by the time-reversed series g, quintic Hermite interpolation (App. C)."""
    x = g.double().flip(0)
    n = x.shape[0]
    v, a = torch.zeros_like(x), torch.zeros_like(x)
    v[0], v[-1] = x[1] - x[0], x[-1] - x[-2]
    v[1:-1] = 0.5 * (x[2:] - x[:-2])
    a[1:-1] = x[2:] + x[:-2] - 2 * x[1:-1]
    v[2:-2] = (x[:-4] - 8 * x[1:-3] + 8 * x[3:-1] - x[4:]) / 12
    a[2:-2] = (-x[:-4] + 16 * x[1:-3] - 30 * x[2:-2] + 16 * x[3:-1] - x[4:]) / 12
    e = c["every"]

    def force(q):                                   # at half step q
        if q > 2 * e * (n - 1):
            return 0
        i = min(q // (2 * e), n - 2)
        s = (q - 2 * e * i) / (2 * e)
        b = [1 - 10 * s**3 + 15 * s**4 - 6 * s**5, s - 6 * s**3 + 8 * s**4 - 3 * s**5, 0.5 * s**2 - 1.5 * s**3 + 1.5 * s**4 - 0.5 * s**5,
             10 * s**3 - 15 * s**4 + 6 * s**5, -4 * s**3 + 7 * s**4 - 3 * s**5, 0.5 * s**3 - s**4 + 0.5 * s**5]
        return b[0] * x[i] + b[1] * v[i] + b[2] * a[i] + b[3] * x[i + 1] + b[4] * v[i + 1] + b[5] * a[i + 1]
    step = _exact_step(c, c["adjoint"], _grid(c)[1])
    u = torch.zeros_like(x[0])
    out = torch.zeros(c["n_out"], *u.shape, device=DEV, dtype=torch.float64)
    for s in range((c["n_out"] - 1) * e):
        u = step(u, force(2 * s), force(2 * s + 1), force(2 * s + 2))
        if (s + 1) % e == 0:
            out[(s + 1) // e] = u
    return out


def _exact_qr(x):
    """Q and R (positive real diagonal) of the k vectors of every frequency, by Cholesky of the Gram matrix."""
    g = torch.einsum("jan,jbn->jab", x.conj(), x)
    r = torch.linalg.cholesky(g).mH
    q = torch.linalg.solve_triangular(r.mT, x, upper=False)
    return q, r


def exact(case, seed):
    c = case
    f = _input(c, seed)
    if c["call"] == "series":
        return _exact_series(c, f)
    f = f.to(torch.complex128)
    if c["call"] == "qr":
        q1, r1 = _exact_qr(f)
        q, r2 = _exact_qr(q1)
        return {"q": q, "r": (r2 @ r1)[:, None].cpu().numpy()}
    nt, _ = _grid(c)
    rows = c["k"] * _dims(c)[0]
    total = nt + c["tail"] if c["variant"] == "trm" else (c["trans"] + 1) * nt
    seconds = 8e-12 * total * rows * (c["n_omega"] + (c.get("n", 0) if c["system"] == "dense" else 40)) + total * 3e-4
    if c["call"] == "march":
        return _exact_march(c, f, c["adjoint"]) if seconds < 20 else None
    if seconds * (2 * c.get("q", -0.5) + 2) > 20:
        return None
    if c["call"] == "refine":   # modes are defined up to a phase: no value for them
        y = _exact_march(c, _exact_qr(_exact_qr(f)[0])[0], False)
    else:
        y = _exact_march(c, f, False)
        for _ in range(c["q"]):
            y = _exact_march(c, _exact_qr(_exact_march(c, _exact_qr(y)[0], True))[0], False)
        y = _exact_march(c, _exact_qr(y)[0], True)
    lam = torch.linalg.eigvalsh(torch.einsum("jan,jbn->jab", y.conj(), y)).flip(-1)[:, : c["n_modes"]]
    return {"gains": lam.clamp(min=0).sqrt()[None].cpu().numpy(), "forcing": None, "response": None}
