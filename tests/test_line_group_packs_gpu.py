"""The FP32 grouped-line solve over several rounds of its work queue, in each of
its builds: four CTAs per SM (packs of groups for more than one round and at
most two), and seven (six at p = 6) where four would need three rounds; p = 7
has the first build only.

Against the FP64 solve within 2e-5, as elsewhere; repeated, the queue starts
empty again."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_06893_gb300 import build
    build.build()


def packs(nx, ny, N):
    """Packs of a box's groups: 4 lines, 2 + 2, singles by four."""
    g4 = (nx - 1) * (ny - 1)
    g2 = ((nx - 1) * ny + (ny - 1) * nx) * (N - 2) + 2 * (nx - 1) + 2 * (ny - 1)
    g1 = nx * ny * (N - 2) ** 2 + 2 * (nx + ny) * (N - 2) + 4
    assert 4 * g4 + 2 * g2 + g1 == nx * ny * N * N
    return g4 + g2 // 2 + g2 % 2 + -(-(g1 - (2 if g2 % 2 else 0)) // 4)


@pytest.mark.parametrize("p", [2, 3, 5, 6, 7])
@pytest.mark.parametrize("rounds", [2, 3])
def test_rounds_of_packs(p, rounds):
    from paper_2111_06893_gb300 import thermonoise
    once = 4 * torch.cuda.get_device_properties(0).multi_processor_count  # packs four CTAs per SM take at once
    ny = 5
    nx = next(n for n in range(2, 10000) if packs(n, ny, p + 1) > (rounds - 1) * once)
    assert (rounds - 1) * once < packs(nx, ny, p + 1) <= rounds * once
    desc = W.box([0.25 * i for i in range(nx + 1)], [0.3 * i for i in range(ny + 1)], [0.0, -0.3, -0.7, -1.5], p,
                 W.FUSED_SILICA)
    ctx = thermonoise.setup(desc)
    r = torch.tensor(np.random.default_rng(p).uniform(-1, 1, ctx.ndof), dtype=torch.float64, device="cuda")
    z = ctx.precond_apply(r, precond="zgroup")
    first = ctx.precond_apply(r.float(), precond="zgroup")
    assert float((first.double() - z).norm() / z.norm()) < 2e-5
    assert torch.equal(first, ctx.precond_apply(r.float(), precond="zgroup"))
