"""Error of the FP64 plans' fixed-point arithmetic beside that of FP64 arithmetic on the same inputs, both against
an extended-precision evaluation (numpy's longdouble), for inputs that stress a common scale: coefficients that
decay steeply or lie in a small part of the grid, and one far larger than its neighbours."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
N = 16


@pytest.fixture(scope="module")
def B():
    from paper_1201_4060_gb300 import _build
    _build.build()
    from paper_1201_4060_gb300 import bspline
    return bspline


def weights(t, n, dtype):
    """Node weights, derivative weights and the sums of the two values that each derivative weight is the difference
    of, [P, n] of one axis, node 0 leftmost, in the arithmetic of dtype: the library's FP64 recurrence, with its
    products by 1 / (k - 1)."""
    t = t.astype(dtype)
    v = np.zeros((t.shape[0], n + 1), dtype)
    v[:, 1] = 1                                          # v[:, m + 1] = M_k(t + m)
    for k in range(2, n + 1):
        if k == n:
            dw, size = v[:, 1:] - v[:, :-1], v[:, 1:] + v[:, :-1]
        m = np.arange(k).astype(dtype)
        nv = ((t[:, None] + m) * v[:, 1:k + 1] + (dtype(k) - m - t[:, None]) * v[:, :k]) * (dtype(1) / dtype(k - 1))
        v[:, 1:k + 1] = nv
    return v[:, :0:-1], dw[:, ::-1], size[:, ::-1]


def evaluate(coef, x, n, dtype, magnitudes=False):
    """u and grad u (grid units), [P, 3] and [P, 3, 3]; with magnitudes, the sums of the magnitudes of their terms, a
    derivative weight counting as its two values.  The positions are in cells (a domain of length N), so that cell
    and offset are exact."""
    s = x - 0.5 * n
    base = np.floor(s)
    w, d, size = zip(*[weights((s - base)[:, a], n, dtype) for a in range(3)])
    i = (base.astype(np.int64)[:, :, None] + 1 + np.arange(n)) % N
    v = coef[:, i[:, 0, :, None, None], i[:, 1, None, :, None], i[:, 2, None, None, :]].astype(dtype)
    if magnitudes:
        v, d = np.abs(v), size

    def one_by_one(terms):                               # not numpy's pairwise sum
        out = terms[..., 0]
        for j in range(1, n):
            out = out + terms[..., j]
        return out

    def sums(wx, wy, wz):
        z = one_by_one(v * wz[:, None, None, :])
        return one_by_one(one_by_one(z * wy[:, None, :]) * wx).T

    u = sums(w[0], w[1], w[2])
    g = np.stack([sums(d[0], w[1], w[2]), sums(w[0], d[1], w[2]), sums(w[0], w[1], d[2])], -1)
    return u, g


def coefficients(kind, seed):
    rng = np.random.default_rng(seed)
    noise = rng.standard_normal((3, N, N, N))
    at = np.add.outer(np.add.outer(np.arange(N), np.arange(N)), np.arange(N))
    if kind == "white":
        return noise
    if kind == "outlier":                                # one value 40 times its tile's others
        noise[:, 2::8, 3::8, 1::8] = 40.0 * np.abs(noise).max()
        return noise
    if kind == "spike":
        c = 1e-6 * np.abs(noise)
        c[:, 5::8, 6::8, 4::8] = 1.0
        return c
    if kind == "gaussian":
        r2 = (np.arange(N) - 7.3) ** 2 / (2 * 1.5 ** 2)
        return np.exp(-np.add.outer(np.add.outer(r2, r2), r2)) * (1 + 0.1 * noise)
    return np.exp(-float(kind) * at) * (1 + 0.1 * noise)                         # steep


def errors(B, coef, order, P, seed):
    """Errors over the sum of magnitudes that each result is summed from: of the library and of FP64 arithmetic,
    for u and grad u."""
    x = np.random.default_rng(seed).uniform(0, N, (P, 3))
    plan = B.Plan(N, order, "f64", L=float(N))
    u, g = plan.interp(torch.from_numpy(coef).cuda(), torch.from_numpy(x).cuda())
    assert plan.status() == 0
    plan.close()
    exact, f64 = evaluate(coef, x, order, np.longdouble), evaluate(coef, x, order, np.float64)
    size = evaluate(coef, x, order, np.float64, magnitudes=True)
    out = []
    for lib, e, d, s in zip((u.cpu().numpy(), g.cpu().numpy()), exact, f64, size):
        out.append((((lib - e) / s).astype(np.float64), ((d - e) / s).astype(np.float64)))
    return out


def rms(v):
    return float(np.sqrt(np.mean(np.square(v))))


@pytest.mark.parametrize("kind", ["white", "outlier", "spike", "gaussian", "0.3", "1", "2"])
@pytest.mark.parametrize("order", [3, 4, 6, 8])
@pytest.mark.parametrize("P", [301, 2100])                # 8 bricks
def test_evaluation_error_is_no_larger_than_fp64(B, kind, order, P):
    """Where the fixed form is taken its error is below FP64 arithmetic's, elsewhere it is FP64 arithmetic in
    another order of operations, which is what the factor 1.25 allows for."""
    for lib, f64 in errors(B, coefficients(kind, order), order, P, 100 + order):
        assert rms(f64) > 0.2 * EPS                       # the comparison means something
        assert rms(lib) <= 1.25 * rms(f64), (rms(lib) / EPS, rms(f64) / EPS)


def dft(line):
    """sum_k line[k] exp(2 pi i k n / N) in extended precision."""
    n = line.shape[0]
    angle = np.arctan2(np.longdouble(0), np.longdouble(-1)) * 2 * np.arange(n) / n
    c, s = np.cos(angle), np.sin(angle)
    at = np.outer(np.arange(n), np.arange(n)) % n
    re, im = line.real.astype(np.longdouble), line.imag.astype(np.longdouble)
    return (c[at] * re - s[at] * im).sum(-1)             # the real part


@pytest.mark.parametrize("decay", [0.0, 11.0 / 6.0])
@pytest.mark.parametrize("n", [32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024])
def test_transform_error_is_below_fp64(B, n, decay):
    """One line of modes along each axis, in a component of its own: flat, and falling like a turbulent field's.
    rms error over rms result at most 1.5 units of 2^-53, less than FP64 stages of these lengths have (1.4 to 2.1).
    Order 2, whose prefilter is one."""
    g = torch.Generator(device="cuda").manual_seed(n)
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    amp = (1 + torch.minimum(k, n - k)) ** -decay
    line = torch.view_as_complex(torch.randn((3, n, 2), generator=g, dtype=torch.float64, device="cuda")) * amp
    half = torch.zeros((3, n, n, n // 2 + 1), dtype=torch.complex128, device="cuda")
    half[0, 0, 0, :] = line[0, :n // 2 + 1]
    half[1, 0, :, 0] = line[1]
    half[2, :, 0, 0] = line[2]
    plan = B.Plan(n, 2, "f64")
    coef = plan.coeffs(half)
    assert plan.status() == 0
    plan.close()
    out = [coef[0, 1, 2, :].cpu().numpy(), coef[1, 1, :, 2].cpu().numpy(), coef[2, :, 1, 2].cpu().numpy()]
    del half, coef
    torch.cuda.empty_cache()
    line = line.cpu().numpy()
    full = line[0].copy()                                # the real line whose first half these modes are
    full[n // 2 + 1:] = line[0, 1:n // 2][::-1].conj()
    full[0], full[n // 2] = full[0].real, full[n // 2].real
    for axis, (got, modes) in enumerate(zip(out, (full, line[1], line[2]))):
        ref = dft(modes)
        err = rms((got - ref).astype(np.float64)) / rms(ref.astype(np.float64))
        assert err <= 1.5 * EPS, (axis, err / EPS)
