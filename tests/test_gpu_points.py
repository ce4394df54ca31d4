"""Calls too small to be sorted: the direct gather in the caller's order gives the staged gather's bits, for
every order, at counts around its particles per CTA, with non-finite positions in between."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = 2.0 * math.pi


@pytest.fixture(scope="module")
def B():
    from paper_1201_4060_gb300 import _build
    _build.build()
    from paper_1201_4060_gb300 import bspline
    return bspline


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("order", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("N", [8, 48])
def test_unsorted_calls_give_the_staged_bits(B, dtype, order, N):
    g = torch.Generator(device="cuda").manual_seed(order)
    plan = B.Plan(N, order, dtype)
    coef = torch.randn((3, N, N, N), generator=g, device="cuda").to(plan.coef_dtype)
    per_cta = 4 if order == 8 else 128 // (3 * order)
    for P in (1, per_cta, per_cta + 1, 1501):
        x = (torch.rand((P, 3), generator=g, dtype=torch.float64, device="cuda") * 3 - 1) * L
        x[P // 2, order % 3] = math.nan
        x[P - 1] = torch.tensor([L, 0.0, math.nextafter(L, 0.0)])
        bad = int((~torch.isfinite(x)).any(dim=1).sum())
        outs = []
        for split in (0, B.GATHER_SPLIT_AUTO, 2 ** 32 - 1):
            plan.set_gather_split(split)
            u, grad = plan.interp(coef, x)
            assert plan.status() == bad
            u1 = plan.interp(coef, x, grad=False)
            assert torch.equal(torch.nan_to_num(u, 7.0), torch.nan_to_num(u1, 7.0))
            outs.append((u, grad))
        for u, grad in outs[1:]:
            assert torch.equal(torch.nan_to_num(u, 7.0), torch.nan_to_num(outs[0][0], 7.0))
            assert torch.equal(torch.nan_to_num(grad, 7.0), torch.nan_to_num(outs[0][1], 7.0))
        assert int(torch.isnan(outs[1][0]).any(dim=1).sum()) == bad
    plan.close()


@pytest.mark.parametrize("NB_target", [(64, 3000), (128, 40000)])
def test_split_scan_over_several_runs(B, NB_target):
    """Bricks on both sides of the split, more bricks than one run of the scan: every split the same bits."""
    N, P = NB_target
    order = 4
    rng = np.random.default_rng(N)
    x = rng.uniform(0, L, (P, 3))
    x[: P // 2] = rng.normal(L / 3, 0.05 * L, (P // 2, 3)) % L
    xt = torch.from_numpy(x).cuda()
    plan = B.Plan(N, order, "f32")
    coef = torch.randn((3, N, N, N), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    plan.set_gather_split(0)
    u0, g0 = plan.interp(coef, xt)
    for split in (3, 20, 64, 1 << 30):
        plan.set_gather_split(split)
        u, g = plan.interp(coef, xt)
        assert plan.status() == 0 and torch.equal(u, u0) and torch.equal(g, g0), split
    plan.close()
