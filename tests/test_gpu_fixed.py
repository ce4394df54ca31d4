"""The fixed-point evaluation of FP64 plans where it could go wrong: every order in both item forms (a few
and many particles per brick), coefficients over 60 decades, subnormal, zero, infinite and NaN ones.

Held to the oracle's evaluation of the same coefficients particle by particle: the error of u relative to
the largest coefficient in the particle's own stencil, that of grad u to 2 N / L times it (the derivative
weights of an axis sum to at most 2 in magnitude), at most 1e-12, the FP64 bar of the parity tests."""
import math

import numpy as np
import pytest

from oracle import bspline_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = 2.0 * math.pi
TOL = 1e-12


@pytest.fixture(scope="module")
def B():
    from paper_1201_4060_gb300 import _build
    _build.build()
    from paper_1201_4060_gb300 import bspline
    return bspline


def stencil_max(coef, x, N, order):
    """Largest |coefficient| of each particle's stencil, [P, 3]."""
    nodes, _ = O.locate(x, N, order)
    i = nodes % N
    v = np.abs(coef)[:, i[:, 0, :, None, None], i[:, 1, None, :, None], i[:, 2, None, None, :]]
    return v.max(axis=(2, 3, 4)).T


def check(B, coef, x, N, order):
    plan = B.Plan(N, order, "f64")
    c = torch.from_numpy(coef).cuda()
    u, g = plan.interp(c, torch.from_numpy(x).cuda())
    u1 = plan.interp(c, torch.from_numpy(x).cuda(), grad=False)
    assert plan.status() == 0
    assert torch.equal(torch.nan_to_num(u), torch.nan_to_num(u1))
    u, g = u.cpu().numpy(), g.cpu().numpy()
    with np.errstate(all="ignore"):
        ru, rg = O.evaluate(coef, x, order)
    plan.close()
    ok = np.isfinite(ru)
    assert np.array_equal(np.isfinite(u), ok)
    m = np.where(ok, stencil_max(np.nan_to_num(coef, posinf=0.0, neginf=0.0), x, N, order), 1.0)
    tiny = 5e-324
    assert (np.abs(u[ok] - ru[ok]) <= TOL * m[ok] + tiny).all()
    gok = np.isfinite(rg)
    assert np.array_equal(np.isfinite(g), gok)
    bound = (TOL * 2 * N / L * m + tiny)[:, :, None] * np.ones(3)
    assert (np.abs(g[gok] - rg[gok]) <= bound[gok]).all()
    return u, g


def positions(P, seed):
    x = np.random.default_rng(seed).uniform(0, L, (P, 3))
    x[0] = 0.0
    x[1] = [math.nextafter(L, 0.0), 1e-20, L / 2]
    return x


@pytest.mark.parametrize("order", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("P", [43, 2049])                # 16^3: 8 bricks, 256 particles each take the long items
def test_orders_in_both_item_forms(B, order, P):
    N = 16
    coef = np.random.default_rng(order).standard_normal((3, N, N, N))
    check(B, coef, positions(P, order), N, order)


@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("P", [300, 3000])
def test_coefficients_over_many_decades(B, order, P):
    """Neighbouring coefficients 60 decades apart: the particles away from a tile's largest ones take the
    FP64 evaluation, lane by lane beside others that do not."""
    N = 16
    rng = np.random.default_rng(10 + order)
    coef = rng.standard_normal((3, N, N, N)) * 10.0 ** rng.uniform(-30, 30, (3, N, N, N))
    check(B, coef, positions(P, 20 + order), N, order)
    smooth = np.exp(-np.add.outer(np.add.outer(np.arange(N), np.arange(N)), np.arange(N)) * 1.5)
    check(B, np.stack([smooth, -smooth, smooth[::-1]]).copy(), positions(P, 30 + order), N, order)


@pytest.mark.parametrize("scale", [1e-310, 1e-280, 1e300])
def test_extreme_scales_and_a_zero_component(B, scale):
    N, order = 16, 4
    coef = np.random.default_rng(3).standard_normal((3, N, N, N)) * scale
    coef[1] = 0.0
    u, g = check(B, coef, positions(2500, 4), N, order)
    assert (u[:, 1] == 0).all() and (g[:, 1] == 0).all()


@pytest.mark.parametrize("P", [400, 4000])
def test_non_finite_coefficients_reach_only_their_stencils(B, P):
    N, order = 16, 5
    coef = np.random.default_rng(5).standard_normal((3, N, N, N))
    coef[0, 3, 4, 5] = np.nan
    coef[2, 10, 11, 12] = np.inf
    x = np.random.default_rng(6).uniform(0, L, (P, 3))
    u, _ = check(B, coef, x, N, order)
    assert 0 < np.isnan(u[:, 0]).sum() < P / 4 and np.isfinite(u[:, 1]).all()


@pytest.mark.parametrize("N", [32, 48, 64])
@pytest.mark.parametrize("scale", [1.0, 1e-250, 1e-300, 1e300])
def test_transform_scales(B, N, scale):
    """Spectra inside and outside the fixed-point range (2^-895 to 2^977), and tiles that mix both: one column
    of modes 10^300 below its neighbours takes the FP64 stages with the rest of its tile."""
    rng = np.random.default_rng(N)
    half = rng.standard_normal((3, N, N, N // 2 + 1)) + 1j * rng.standard_normal((3, N, N, N // 2 + 1))
    half[2] = 0.0
    half *= scale
    half[1, :, 1, 1] *= 1e-300
    plan = B.Plan(N, 4, "f64")
    c = plan.coeffs(torch.from_numpy(half).cuda()).cpu().numpy()
    assert plan.status() == 0
    ref = O.coefficients(half / scale, 4) * scale
    assert (c[2] == 0).all()
    for k in range(2):
        assert np.abs(c[k] - ref[k]).max() <= 1e-12 * np.abs(ref[k]).max()
    plan.close()


def test_transform_non_finite_modes_reach_their_component(B):
    N = 32
    half = np.random.default_rng(1).standard_normal((3, N, N, N // 2 + 1)).astype(np.complex128)
    ref = O.coefficients(half, 6)
    half[0, 3, 4, 5] = np.nan
    half[2, 0, 0, 0] = np.inf
    plan = B.Plan(N, 6, "f64")
    c = plan.coeffs(torch.from_numpy(half).cuda()).cpu().numpy()
    assert np.isnan(c[0]).all() and not np.isfinite(c[2]).any()
    assert np.abs(c[1] - ref[1]).max() <= 1e-12 * np.abs(ref[1]).max()
    plan.close()
