"""Rules that pick a route by a call's size, from outside: workspaces that smaller calls never outgrow."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_1201_4060_gb300 import _build
    _build.build()
    from paper_1201_4060_gb300 import bspline
    return bspline


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("N", [32, 64])
def test_workspace_never_shrinks_with_more_particles(B, dtype, N):
    """A call of fewer particles after a larger one allocates nothing (it may be captured): across every rule
    that depends on the count, such as the work items' length of FP64 plans (256 particles a brick)."""
    plan = B.Plan(N, 4, dtype)
    bricks = (N // 8) ** 3
    counts = sorted({p + d for p in (1, 42, 512, 2048, 16 * bricks, 64 * bricks, 96 * bricks, 128 * bricks, 256 * bricks,
                                     300000) for d in (-1, 0, 1) if p + d > 0})
    sizes = [plan.workspace_bytes(p) for p in counts]
    assert sizes == sorted(sizes)
    plan.close()
