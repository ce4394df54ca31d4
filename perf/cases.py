"""Performance cases of the library: what its users run, through paper_1201_4060_gb300.bspline and .autograd.

A case is a dict of plain values:
  kind     "eval"    Plan.eval: coefficients, u and grad u from a spectrum (a solver's step)
           "interp"  Plan.interp: u (and grad u) on coefficients that are there (particle sub-steps)
           "adjoint" Plan.spread_adjoint: gradients of spectrum, coefficients and positions
           "train"   autograd.interpolate, forward and backward (a differentiable program's step)
           "batch"   Batch.launch: many small fields of uneven size in one graph
  N, order, dtype, P and how the positions are distributed; options by kind.
The fields are dealiased Kolmogorov spectra (modes 1 <= |k| <= N/3, E(k) ~ k^(-5/3), solenoidal, Hermitian,
u_rms = 1), the positions uniform, clustered (60 % uniform, 40 % Gaussian clumps of sigma 0.1 around 64
centres) or uniform in raster order of their grid cells, the cotangents N(0, 1): the recipes of
paper_1201_4060_gb300/synth.py, drawn on the GPU.
"""
import math
import random

import torch

from paper_1201_4060_gb300 import autograd, bspline

L = 2.0 * math.pi
GRIDS = (32, 48, 64, 96, 128, 192, 256, 384, 512)
BATCH_GRIDS = (32, 48, 64, 96, 128, 192)


def listed():
    return [
        # FP64 reference run of a small solver: 10^4 tracers on 32^3, spectrum to u and grad u each step
        dict(name="solver32_f64", kind="eval", N=32, order=4, dtype="f64", P=10_000, dist="uniform", band=0),
        # a thousand probes sampled on a 64^3 field: the smallest call, all latency
        dict(name="probes64", kind="interp", N=64, order=4, dtype="f32", P=1_000, dist="uniform", grad=True),
        # passive tracers: their advection takes u alone; an odd count, an odd order
        dict(name="tracers128_u_only", kind="interp", N=128, order=5, dtype="f32", P=100_003, dist="uniform",
             grad=False),
        # a million particles kept in raster order of their cells, u and grad u of a cubic interpolant
        dict(name="particles256_cubic", kind="interp", N=256, order=4, dtype="f32", P=1_000_000, dist="cells",
             grad=True),
        # few particles in a large field: most bricks hold a handful
        dict(name="sparse512", kind="interp", N=512, order=6, dtype="f32", P=1 << 18, dist="uniform", grad=True),
        # dealiased 384^3 solver with its band declared, highest order, an odd particle count
        dict(name="band384_o8", kind="eval", N=384, order=8, dtype="f32", P=2_000_003, dist="uniform", band=128),
        # the large production step: 512^3, quintic, 16 Mi clustered particles, in both storage types
        dict(name="field512_f32", kind="eval", N=512, order=6, dtype="f32", P=1 << 24, dist="clustered", band=0),
        dict(name="field512_bf16", kind="eval", N=512, order=6, dtype="bf16", P=1 << 24, dist="clustered", band=0),
        # FP64 form of the quintic interpolant on a mid-sized field
        dict(name="field256_f64", kind="eval", N=256, order=6, dtype="f64", P=1_000_000, dist="uniform", band=0),
        # gradients of spectrum, coefficients and positions for 4 Mi particles
        dict(name="adjoint256", kind="adjoint", N=256, order=4, dtype="f32", P=1 << 22, dist="uniform",
             positions=True, deterministic=False),
        # a small differentiable program: forward and backward through torch.autograd
        dict(name="train96", kind="train", N=96, order=6, dtype="f32", P=50_001, dist="uniform"),
        # 64 independent fields of 32^3 to 192^3 with 10^3 to 10^6 particles each, one graph launch
        dict(name="batch64", kind="batch", fields=64, order=4, dtype="f32", counts=4064, lo=1_000, hi=1_000_000),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "interp", "interp", "interp", "adjoint", "adjoint", "train", "batch"])
    if kind == "batch":
        return dict(kind=kind, fields=rng.randint(8, 64), order=rng.randint(2, 6), dtype="f32",
                    counts=rng.randrange(1 << 20), lo=1_000, hi=_log_int(rng, 20_000, 1_000_000))
    dtype = rng.choice(["f32", "f32", "f32", "bf16", "f64"])
    order = rng.randint(2, 8)
    if kind == "train":
        return dict(kind=kind, N=rng.choice(GRIDS[:6]), order=order, dtype=rng.choice(["f32", "f32", "f64"]),
                    P=_log_int(rng, 1_000, 200_000), dist=rng.choice(["uniform", "clustered"]))
    if dtype == "f64":
        N, most = rng.choice(GRIDS[:7]), min(1_000_000, 216_000_000 // order ** 3)
    else:
        N, most = rng.choice(GRIDS), min(1 << 24, (1 << 24) * 216 // order ** 3)
    if kind == "adjoint":
        N, most = min(N, 256), min(most, 1 << 22, (1 << 22) * 64 // order ** 3)
        if dtype == "f64":
            N, most = min(N, 128), min(most, 100_000)
        return dict(kind=kind, N=N, order=order, dtype=dtype, P=_log_int(rng, 1_000, most),
                    dist=rng.choice(["uniform", "clustered"]), positions=rng.random() < 0.7,
                    deterministic=dtype != "f64" and rng.random() < 0.3)
    c = dict(kind=kind, N=N, order=order, dtype=dtype, P=_log_int(rng, 1_000, most),
             dist=rng.choice(["uniform", "clustered", "cells"]))
    if kind == "eval":
        c["band"] = N // 3 if rng.random() < 0.4 else 0
    else:
        c["grad"] = rng.random() < 0.75
    return c


# ---- inputs ------------------------------------------------------------------------

def _real(dtype):
    return torch.float64 if dtype == "f64" else torch.float32


def _field(N, dtype, g):
    """Dealiased Kolmogorov spectrum [3, N, N, N/2 + 1] on the GPU."""
    real = _real(dtype)
    H, kmax = N // 2 + 1, N // 3
    k = torch.arange(N, device="cuda")
    k = torch.where(k < N // 2, k, k - N).to(real)
    kx, ky, kz = k[:, None, None], k[None, :, None], torch.arange(H, device="cuda").to(real)[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    amp = torch.where((k2 >= 1) & (k2 <= kmax * kmax), k2.clamp(min=1.0) ** (-11.0 / 12.0), torch.zeros_like(k2))
    v = torch.empty((3, N, N, H, 2), dtype=real, device="cuda")
    for c in range(3):
        v[c] = torch.randn((N, N, H, 2), generator=g, dtype=real, device="cuda") * amp[..., None]
    dot = (v[0] * kx[..., None] + v[1] * ky[..., None] + v[2] * kz[..., None]) / k2.clamp(min=1.0)[..., None]
    for c, kc in enumerate((kx, ky, kz)):
        v[c] -= dot * kc[..., None]
    u = torch.view_as_complex(v)
    p = u[..., 0]                                        # the plane that holds both k and -k
    u[..., 0] = 0.5 * (p + torch.roll(p.flip(1, 2), (1, 1), (1, 2)).conj())
    e = v.square().sum(dim=(0, 1, 2, 4), dtype=torch.float64)
    energy = (2.0 * e.sum() - e[0]) / 3.0
    v *= (1.0 / energy.sqrt()).to(real)
    return u.contiguous()


def _positions(N, P, dist, g):
    x = torch.rand((P, 3), generator=g, dtype=torch.float64, device="cuda") * L
    if dist == "clustered":
        n = int(round(0.4 * P))
        centres = torch.rand((64, 3), generator=g, dtype=torch.float64, device="cuda") * L
        at = torch.randint(0, 64, (n,), generator=g, device="cuda")
        x[:n] = torch.remainder(centres[at] + 0.1 * torch.randn((n, 3), generator=g, dtype=torch.float64,
                                                                 device="cuda"), L)
        x = x[torch.randperm(P, generator=g, device="cuda")]
    elif dist == "cells":
        c = (x * (N / L)).floor().long().clamp(0, N - 1)
        x = x[((c[:, 0] * N + c[:, 1]) * N + c[:, 2]).argsort()]
    return x.contiguous()


def _cotangents(P, dtype, g):
    real = _real(dtype)
    return (torch.randn((P, 3), generator=g, dtype=real, device="cuda"),
            torch.randn((P, 3, 3), generator=g, dtype=real, device="cuda"))


def _batch_fields(case):
    """(N, P) of each field: grids in turn, counts log-uniform."""
    r = random.Random(case["counts"])
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    return [(BATCH_GRIDS[i % len(BATCH_GRIDS)], int(math.exp(r.uniform(lo, hi)))) for i in range(case["fields"])]


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["kind"] == "batch":
        return [(_field(N, "f32", g), _positions(N, P, "uniform", g)) for N, P in _batch_fields(case)]
    s = dict(u_hat=_field(case["N"], case["dtype"], g), x=_positions(case["N"], case["P"], case["dist"], g))
    if case["kind"] in ("adjoint", "train"):
        s["g_u"], s["g_grad"] = _cotangents(case["P"], case["dtype"], g)
    return s


def _even(P):
    return (P + 1) // 2 * 2


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    N, P = case["N"], case["P"]
    plan = bspline.Plan(N, case["order"], case["dtype"])
    s = dict(_inputs(case, seed), case=case, plan=plan)
    if kind == "eval":
        if case["band"]:
            plan.set_band(case["band"])
        s["coef"] = plan.empty_coeffs()
    elif kind in ("interp", "adjoint"):
        s["coef"] = plan.coeffs(s.pop("u_hat"))
    if kind in ("eval", "interp"):
        s["u"] = torch.empty((P, 3), dtype=plan.out_dtype, device="cuda")
        s["grad"] = torch.empty((P, 3, 3), dtype=plan.out_dtype, device="cuda") if case.get("grad", True) else None
    if kind == "adjoint":
        plan.set_deterministic(case["deterministic"])
    if kind == "train":
        s["u_hat"].requires_grad_()
        s["x"].requires_grad_()
    return s


def _prepare_batch(case, seed):
    """All fields' coefficients in one buffer, and their outputs (each field's from an even particle on)."""
    fields, inputs = _batch_fields(case), _inputs(case, seed)
    coef = torch.empty(sum(3 * N ** 3 for N, _ in fields), dtype=torch.float32, device="cuda")
    rows = sum(_even(P) for _, P in fields)
    u = torch.zeros((rows, 3), dtype=torch.float32, device="cuda")
    grad = torch.zeros((rows, 3, 3), dtype=torch.float32, device="cuda")
    coefs, us, grads, c, r = [], [], [], 0, 0
    for N, P in fields:
        coefs.append(coef[c:c + 3 * N ** 3].view(3, N, N, N))
        us.append(u[r:r + P])
        grads.append(grad[r:r + P])
        c, r = c + 3 * N ** 3, r + _even(P)
    batch = bspline.Batch([bspline.Plan(N, case["order"], "f32") for N, _ in fields])
    batch.capture([a for a, _ in inputs], coefs, [x for _, x in inputs], us, grads)
    return dict(case=case, batch=batch, coef=coef, u=u, grad=grad)


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        state["batch"].launch()
        return state["coef"], state["u"], state["grad"]
    plan = state["plan"]
    if kind == "eval":
        return plan.eval(state["u_hat"], state["x"], state["coef"], state["u"], state["grad"])
    if kind == "interp":
        return plan.interp(state["coef"], state["x"], state["u"], state["grad"], grad=case["grad"])
    if kind == "adjoint":
        if case["positions"]:
            return plan.spread_adjoint(state["x"], state["g_u"], state["g_grad"], coef=state["coef"])
        g_u_hat, _, g_coef = plan.spread_adjoint(state["x"], state["g_u"], state["g_grad"])
        return g_u_hat, g_coef
    u, grad = autograd.interpolate(state["u_hat"], state["x"], plan)
    g_u_hat, g_x = torch.autograd.grad((u, grad), (state["u_hat"], state["x"]), (state["g_u"], state["g_grad"]))
    return u.detach(), grad.detach(), g_u_hat, g_x


# ---- what a pass cannot do without ---------------------------------------------------

def _transform_work(N, dtype, band=0):
    cplx, coef = (16, 8) if dtype == "f64" else (8, 2 if dtype == "bf16" else 4)
    modes = (2 * band + 1) ** 2 * (band + 1) if band else N * N * (N // 2 + 1)
    return 3 * modes * cplx + 3 * N ** 3 * coef, 3 * 2.5 * N ** 3 * 3 * math.log2(N)


def _interp_work(P, n, dtype, grad=True):
    out = 8 if dtype == "f64" else 4
    fma = 3 * (2 * n ** 3 + 3 * n * n + 4 * n) + 15 * n * n if grad else 3 * (n ** 3 + n * n + n) + 8 * n * n
    return P * (24 + out * (12 if grad else 3)), 2.0 * P * fma


def work(case):
    kind, n, dtype = case["kind"], case["order"], case["dtype"]
    if kind == "batch":
        parts = [f for N, P in _batch_fields(case) for f in (_transform_work(N, dtype), _interp_work(P, n, dtype))]
    else:
        N, P = case["N"], case["P"]
        coef = 3 * N ** 3 * (8 if dtype == "f64" else 2 if dtype == "bf16" else 4)
        out = 8 if dtype == "f64" else 4
        # a stencil of n^3 nodes a particle: few particles touch a part of the coefficients only
        touched = min(coef, coef // N ** 3 * P * n ** 3)
        g_coef = 3 * N ** 3 * out
        spread = (P * (24 + 12 * out) + g_coef, 2.0 * P * (3 * 2 * n ** 3 + 15 * n * n))
        g_x = (touched + P * 24, 2.0 * P * 3 * (3 * n ** 3 + 6 * n * n + 9 * n))
        back = (3 * N * N * (N // 2 + 1) * 2 * out, 3 * 2.5 * N ** 3 * 3 * math.log2(N))
        if kind == "eval":
            parts = [_transform_work(N, dtype, case["band"]), _interp_work(P, n, dtype)]
        elif kind == "interp":
            parts = [(touched, 0.0), _interp_work(P, n, dtype, case["grad"])]
        elif kind == "adjoint":
            parts = [spread, back] + ([g_x] if case["positions"] else [])
        else:
            parts = [_transform_work(N, dtype), _interp_work(P, n, dtype), spread, back, (P * 24, g_x[1])]
    return {"bytes": float(sum(p[0] for p in parts)), "flops": float(sum(p[1] for p in parts))}


# ---- the same in 64 bits, in plain torch ----------------------------------------------

def _bsplines(t, n):
    """Node weights of the order-n B-spline and their first two derivatives, [P, n] each, node 0 leftmost."""
    def cardinal(k):                                     # M_k(t + m), m = 0..n-1 (0 outside the support)
        v = torch.zeros((t.shape[0], n + 1), dtype=t.dtype, device=t.device)
        v[:, 0] = 1.0
        m = torch.arange(n + 1, device=t.device, dtype=t.dtype)
        for q in range(2, k + 1):
            left = torch.cat([torch.zeros_like(v[:, :1]), v[:, :-1]], 1)
            v = ((t[:, None] + m) * v + (q - m - t[:, None]) * left) / (q - 1)
            v[:, q:] = 0.0
        return v[:, :n]

    def diff(v):
        return v - torch.cat([torch.zeros_like(v[:, :1]), v[:, :-1]], 1)

    d2 = diff(diff(cardinal(n - 2))) if n > 2 else torch.zeros((t.shape[0], n), dtype=t.dtype, device=t.device)
    return [w.flip(1) for w in (cardinal(n), diff(cardinal(n - 1)), d2)]


def _prefilter(N, n):
    d = torch.arange(n + 1, dtype=torch.float64, device="cuda")
    values = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    w = _bsplines(torch.full((1,), 0.5 if n % 2 else 0.0, dtype=torch.float64, device="cuda"), n)[0][0].flip(0)
    values[:n] = w                                       # M_n(t + m): the node values, m - (n/2 - t) from the centre
    off = d - (n / 2 - (0.5 if n % 2 else 0.0))
    k = torch.arange(N, dtype=torch.float64, device="cuda")
    return 1.0 / (values * torch.cos(2 * math.pi * k[:, None] * off / N)).sum(1)


def _exact_coef(u_hat, N, n):
    c = _prefilter(N, n)
    out = torch.empty((3, N, N, N), dtype=torch.float64, device="cuda")
    for i in range(3):
        a = u_hat[i].to(torch.complex128) * (c[:, None, None] * c[None, :, None] * c[None, None, :N // 2 + 1])
        out[i] = torch.fft.irfft(torch.fft.ifft2(a, dim=(0, 1), norm="forward"), n=N, dim=2, norm="forward")
        del a
    return out


def _stencil(x, N, n):
    """Flat node indices [P, n, n, n] and the weights per axis."""
    s = x * (N / L) - 0.5 * n
    base = s.floor()
    t = s - base
    j = torch.arange(1, n + 1, device=x.device)
    i = [(base[:, a].long()[:, None] + j).remainder(N) for a in range(3)]
    at = (i[0][:, :, None, None] * N + i[1][:, None, :, None]) * N + i[2][:, None, None, :]
    return at, [_bsplines(t[:, a].contiguous(), n) for a in range(3)]


def _chunks(P, n):
    step = max(1, (1 << 25) // n ** 3)
    return [slice(a, min(P, a + step)) for a in range(0, P, step)]


def _contract(a, wx, wy, wz):
    z = (a * wz[:, None, None, :]).sum(3)
    return ((z * wy[:, None, :]).sum(2) * wx).sum(1)


def _exact_interp(coef, x, N, n, grad=True):
    P, scale = x.shape[0], N / L
    u = torch.empty((P, 3), dtype=torch.float64, device="cuda")
    g = torch.empty((P, 3, 3), dtype=torch.float64, device="cuda") if grad else None
    for sl in _chunks(P, n):
        at, (wx, wy, wz) = _stencil(x[sl], N, n)
        for c in range(3):
            a = coef[c].reshape(-1)[at]
            u[sl, c] = _contract(a, wx[0], wy[0], wz[0])
            if grad:
                g[sl, c, 0] = scale * _contract(a, wx[1], wy[0], wz[0])
                g[sl, c, 1] = scale * _contract(a, wx[0], wy[1], wz[0])
                g[sl, c, 2] = scale * _contract(a, wx[0], wy[0], wz[1])
    return u, g


def _exact_spread(x, g_u, g_grad, N, n):
    scale = N / L
    out = torch.zeros((3, N ** 3), dtype=torch.float64, device="cuda")
    for sl in _chunks(x.shape[0], n):
        at, (wx, wy, wz) = _stencil(x[sl], N, n)
        for c in range(3):
            gu, gg = g_u[sl, c].double()[:, None], g_grad[sl, c].double() * scale
            p = gu * wx[0] + gg[:, :1] * wx[1]
            yz = p[:, :, None] * wy[0][:, None, :] + (gg[:, 1:2] * wx[0])[:, :, None] * wy[1][:, None, :]
            v = yz[..., None] * wz[0][:, None, None, :]
            v += ((gg[:, 2:] * wx[0])[:, :, None] * wy[0][:, None, :])[..., None] * wz[1][:, None, None, :]
            out[c].index_add_(0, at.reshape(-1), v.reshape(-1))
    return out.view(3, N, N, N)


def _exact_spectrum(g_coef, N, n):
    c = _prefilter(N, n)
    m = torch.full((N // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    m[0] = m[-1] = 1.0
    return torch.stack([torch.fft.rfftn(g_coef[i]) * (c[:, None, None] * c[None, :, None] * (c[:N // 2 + 1] * m))
                        for i in range(3)])


def _exact_positions(coef, x, g_u, g_grad, N, n):
    scale = N / L
    out = torch.zeros((x.shape[0], 3), dtype=torch.float64, device="cuda")
    for sl in _chunks(x.shape[0], n):
        at, w = _stencil(x[sl], N, n)
        for c in range(3):
            a = coef[c].reshape(-1)[at]
            for e in range(3):
                d = [int(e == 0), int(e == 1), int(e == 2)]
                out[sl, e] += g_u[sl, c].double() * scale * _contract(a, *[w[i][d[i]] for i in range(3)])
                for f in range(3):
                    dd = list(d)
                    dd[f] += 1
                    out[sl, e] += g_grad[sl, c, f].double() * scale ** 2 * _contract(a, *[w[i][dd[i]] for i in range(3)])
    return out


def exact(case, seed):
    kind, n = case["kind"], case["order"]
    if kind == "batch":
        fields = _batch_fields(case)
        rows = sum(_even(P) for _, P in fields)
        coefs = []
        u = torch.zeros((rows, 3), dtype=torch.float64, device="cuda")
        grad = torch.zeros((rows, 3, 3), dtype=torch.float64, device="cuda")
        r = 0
        for (N, P), (u_hat, x) in zip(fields, _inputs(case, seed)):
            coef = _exact_coef(u_hat, N, n)
            u[r:r + P], grad[r:r + P] = _exact_interp(coef, x, N, n)
            coefs.append(coef.reshape(-1))
            r += _even(P)
        return torch.cat(coefs), u, grad
    N, s = case["N"], _inputs(case, seed)
    x = s["x"]
    if kind == "eval":
        coef = _exact_coef(s["u_hat"], N, n)
        return (coef,) + _exact_interp(coef, x, N, n)
    if kind == "interp":
        # on the coefficients as they are stored
        plan_dtype = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[case["dtype"]]
        coef = _exact_coef(s["u_hat"], N, n).to(plan_dtype).double()
        u, g = _exact_interp(coef, x, N, n, case["grad"])
        return (u, g) if case["grad"] else u
    g_coef = _exact_spread(x, s["g_u"], s["g_grad"], N, n)
    g_u_hat = _exact_spectrum(g_coef, N, n)
    coef = _exact_coef(s["u_hat"], N, n)
    if kind == "adjoint":
        if not case["positions"]:
            return g_u_hat, g_coef
        return g_u_hat, _exact_positions(coef, x, s["g_u"], s["g_grad"], N, n), g_coef
    u, grad = _exact_interp(coef, x, N, n)
    return u, grad, g_u_hat, _exact_positions(coef, x, s["g_u"], s["g_grad"], N, n)
