"""Rules that pick a route by a call's size, from outside: workspaces that smaller calls never outgrow, the autotuner's
choice and its cache for calls with and without a sort, and the sorted route at sizes whose calls AUTO does not sort."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = 2.0 * math.pi
ALL_DIRECT = 2 ** 32 - 1


@pytest.fixture(scope="module")
def B():
    from paper_1201_4060_gb300 import _build
    _build.build()
    from paper_1201_4060_gb300 import bspline
    return bspline


def positions(P, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand((P, 3), generator=g, dtype=torch.float64, device="cuda") * L


def field(plan, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    N = plan.N
    return torch.randn((3, N, N, N // 2 + 1), generator=g, dtype=plan.uhat_dtype, device="cuda")


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("N", [32, 64])
def test_workspace_never_shrinks_with_more_particles(B, dtype, N):
    """A call of fewer particles after a larger one allocates nothing (it may be captured): across every rule
    that depends on the count, such as the work items' length of FP64 plans."""
    plan = B.Plan(N, 4, dtype)
    bricks = (N // 8) ** 3
    counts = sorted({p + d for p in (1, 42, 512, 2048, 8192, 16 * bricks, 48 * bricks, 64 * bricks, 96 * bricks,
                                     256 * bricks, 196608, 300000) for d in (-1, 0, 1) if p + d > 0})
    sizes = [plan.workspace_bytes(p) for p in counts]
    assert sizes == sorted(sizes)
    plan.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_workspace_holds_ranks_only_where_the_count_draws_them(B, dtype):
    """4 bytes a particle, beside the record's 32 and an FP64 item's 4 for 42, only from 64 particles a brick on."""
    plan = B.Plan(64, 4, dtype)
    bricks = 512 if dtype == "f64" else 96
    edge = max(8192, 64 * bricks)
    per_particle = 32 + (4 / 42 if dtype == "f64" else 4 / 2048)
    fixed = plan.workspace_bytes(1)
    assert plan.workspace_bytes(edge - 1) <= fixed + per_particle * edge + 4096
    assert plan.workspace_bytes(edge) >= fixed + (per_particle + 4) * edge - 4096
    plan.close()


def key(N, order, P, route):
    return (f"{torch.cuda.get_device_properties(0).name}|N{N}|o{order}|f32|p2^{max(P - 1, 1).bit_length()}"
            + (f"|{route}" if route else ""))


@pytest.mark.parametrize("route", ["", "unsorted"])
def test_all_direct_timed_without_a_sort_is_not_taken_for_a_sorted_call(B, route, tmp_path, monkeypatch):
    """Order 6 sorts from 58255 particles on: a choice of "every brick direct" that was timed for fewer of the same
    power of two, without a sort, says nothing about 60000."""
    N, order, P = 32, 6, 60000
    cache = tmp_path / "autotune.jsonl"
    cache.write_text('{"key": "%s", "direct_below": %d, "ms": 0.0100}\n' % (key(N, order, P, route), ALL_DIRECT))
    monkeypatch.setenv("BSPLINE_AUTOTUNE_CACHE", str(cache))
    plan = B.Plan(N, order, "f32")
    coef = plan.coeffs(field(plan, 1))
    _, ms = plan.autotune(coef, positions(P, 2))
    assert ms > 0                                        # timed, not taken from the file
    plan.close()


def test_all_direct_chosen_without_a_sort_leaves_larger_calls_to_the_rule(B, tmp_path, monkeypatch):
    """A plan tuned on few particles: more of them, or a call beside a transform, are not sorted into the direct
    gather (whose stage is then timed), which was not what was timed."""
    N, order, P = 32, 6, 40000                           # beside a transform 14563 particles are sorted already
    cache = tmp_path / "autotune.jsonl"
    cache.write_text('{"key": "%s", "direct_below": %d, "ms": 0.0100}\n' % (key(N, order, P, "unsorted"), ALL_DIRECT))
    monkeypatch.setenv("BSPLINE_AUTOTUNE_CACHE", str(cache))
    plan = B.Plan(N, order, "f32")
    u_hat = field(plan, 1)
    coef = plan.coeffs(u_hat)
    x = positions(P, 2)
    split, ms = plan.autotune(coef, x)
    assert (split, ms) == (ALL_DIRECT, 0.0)
    plan.set_timing(True)
    for calls, direct in ((lambda: plan.interp(coef, x), 1), (lambda: plan.interp(coef, positions(100000, 3)), 0),
                          (lambda: plan.eval(u_hat, x), 0)):
        plan.stage_times()
        calls()
        assert plan.stage_times()["gather_direct"][1] == direct
    plan.close()


@pytest.mark.parametrize("N", [768, 1024])
def test_largest_grids_sorted_and_unsorted_agree(B, N):
    """The sort, the scan of the most bricks and the staged gather, against the call that AUTO does not sort."""
    order, P = 6, 4096
    plan = B.Plan(N, order, "f32")
    g = torch.Generator(device="cuda").manual_seed(N)
    coef = torch.randn((3, N, N, N), generator=g, device="cuda")
    x = positions(P, N)
    x[:2000] = x[:2000] * 0.01 + 1.0                     # some bricks hold many
    outs = []
    for split in (B.GATHER_SPLIT_AUTO, 0, 16, ALL_DIRECT - 2):
        plan.set_gather_split(split)
        u, grad = plan.interp(coef, x)
        assert plan.status() == 0
        outs.append((u, grad))
    for u, grad in outs[1:]:
        assert torch.equal(u, outs[0][0]) and torch.equal(grad, outs[0][1])
    plan.close()
    del coef, outs
    torch.cuda.empty_cache()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("split", [0, 32])
def test_sort_beside_the_transform_agrees_with_the_unsorted_call(B, dtype, split):
    """bspline_eval and bspline_run_host with the sort on the second stream, at sizes that AUTO does not sort."""
    N, order, P = 32, 6, 5000
    plan = B.Plan(N, order, dtype)
    u_hat, x = field(plan, 3), positions(P, 4)
    x[17, 1] = math.nan
    coef, u, grad = plan.eval(u_hat, x)
    assert plan.status() == 1
    plan.set_gather_split(split)
    coef2, u2, grad2 = plan.eval(u_hat, x)
    assert plan.status() == 1
    uh, xh = u_hat.cpu().pin_memory(), x.cpu().pin_memory()
    uo, go = torch.empty((P, 3)).pin_memory(), torch.empty((P, 3, 3)).pin_memory()
    plan.run_host(uh, xh, uo, go)
    assert plan.status() == 1 and torch.equal(coef, coef2)
    for a, b in ((u, u2), (grad, grad2), (u, uo.cuda()), (grad, go.cuda())):
        assert torch.equal(torch.nan_to_num(a, 7.0), torch.nan_to_num(b, 7.0))
    plan.close()


@pytest.mark.parametrize("dtype,N", [("f64", 32), ("f64", 64), ("f64", 128), ("f32", 64), ("bf16", 128)])
def test_counting_by_runs_and_by_particles_agree(B, dtype, N):
    """Both sides of the rule that counts particles by runs in shared memory (8192 of them, 64 a brick): every
    particle is placed once, and its results are the same bits."""
    order = 3
    plan = B.Plan(N, order, dtype)
    plan.set_gather_split(0)
    bricks = (N // 8) ** 3 if dtype == "f64" else (N // 16) ** 2 * -(-N // 12)
    edge = max(8192, 64 * bricks)
    g = torch.Generator(device="cuda").manual_seed(N)
    real = torch.float64 if dtype == "f64" else torch.float32
    coef = torch.randn((3, N, N, N), generator=g, dtype=real, device="cuda").to(plan.coef_dtype)
    x = positions(edge + 1, N)
    x[5, 2] = math.nan
    x[edge // 2] = 1.0
    outs = []
    for P in (edge + 1, edge, edge - 1):
        u, grad = plan.interp(coef, x[:P].contiguous())
        assert plan.status() == 1
        perm = plan.sort_order(x[:P].contiguous())
        assert torch.equal(perm.sort().values.long(), torch.arange(P, device="cuda")) and int(perm[-1]) == 5
        outs.append((u[:edge - 1], grad[:edge - 1]))
    for u, grad in outs[1:]:
        assert torch.equal(torch.nan_to_num(u, 7.0), torch.nan_to_num(outs[0][0], 7.0))
        assert torch.equal(torch.nan_to_num(grad, 7.0), torch.nan_to_num(outs[0][1], 7.0))
    plan.close()


@pytest.mark.parametrize("N", [96, 192, 256])             # 288, 2304 and 5632 bricks: one to a thread, four, two tiles
def test_scan_places_every_split(B, N):
    """Bricks on both sides of the split and empty ones, some of them staged: every split gives the same bits."""
    order, P = 4, 60000
    plan = B.Plan(N, order, "f32")
    g = torch.Generator(device="cuda").manual_seed(N)
    coef = torch.randn((3, N, N, N), generator=g, device="cuda")
    x = positions(P, N)
    x[: P // 2] = torch.remainder(2.0 + 0.05 * L * torch.randn((P // 2, 3), generator=g, dtype=torch.float64, device="cuda"), L)
    x[7, 0] = math.nan
    plan.set_gather_split(0)
    u0, g0 = plan.interp(coef, x)
    assert plan.status() == 1
    for split in (2, 16, 64, 1 << 30):
        plan.set_gather_split(split)
        u, grad = plan.interp(coef, x)
        assert plan.status() == 1
        for a, b in ((u, u0), (grad, g0)):
            assert torch.equal(torch.nan_to_num(a, 7.0), torch.nan_to_num(b, 7.0)), split
    plan.close()


@pytest.mark.parametrize("order", [2, 3, 4, 5, 6, 7, 8])
def test_long_and_short_items_of_fp64_plans_agree(B, order):
    """200000 particles, 390 a brick, take items of 512, a tenth of them items of 42: the same bits, in a field some of
    whose particles are left to FP64."""
    N, P = 64, 200000
    plan = B.Plan(N, order, "f64")
    g = torch.Generator(device="cuda").manual_seed(order)
    coef = torch.randn((3, N, N, N), generator=g, dtype=torch.float64, device="cuda")
    coef[:, ::8, ::8, ::8] *= 100.0
    x = positions(P, order)
    x[1] = torch.tensor([0.0, L / 2, math.nextafter(L, 0.0)])
    x[2, 0] = math.inf
    u, grad = plan.interp(coef, x)
    assert plan.status() == 1
    u_few, grad_few = plan.interp(coef, x[: P // 10].contiguous())
    for a, b in ((u, u_few), (grad, grad_few)):
        assert torch.equal(torch.nan_to_num(a[: P // 10], 7.0), torch.nan_to_num(b, 7.0))
    plan.close()
