"""The FP32 runs inside a mixed solve go to inner_rtol or inner_max
iterations, however slowly they converge and in whatever replays."""
import pytest

from cases import cyl_thin

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_06893_gb300 import build
    build.build()


@pytest.mark.parametrize("inner_max", [40, 41, 2000])
def test_inner_run_reaches_its_limit(inner_max):
    """diag(A) on layers of 4e-4: thousands of iterations to inner_rtol, the
    residual norm not halved for many hundreds at a time."""
    from paper_2111_06893_gb300 import thermonoise
    ctx = thermonoise.setup(cyl_thin(4))
    _, rep = ctx.solve(mode="mixed", precond="jacobi", rtol=1e-12, inner_rtol=1e-9, inner_max=inner_max, max_outer=1,
                       raise_on_error=False)
    assert rep["inner_iters"] == inner_max and rep["applies_f32"] == inner_max
