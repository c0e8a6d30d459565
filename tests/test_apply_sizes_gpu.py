"""The operator at the sizes where its launches change: elements spread over
the CTAs of the second launch (whole CTAs, remainders, the largest few-element
mesh and the smallest of many).  Results do not depend on the form, so they are
compared bit by bit."""
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


def field(n, dtype, seed=0):
    return torch.tensor(np.random.default_rng(seed).uniform(-1, 1, size=n), dtype=dtype, device="cuda")


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def few_limit():
    return 8 * sms()


def block(nx, ny, slabs, p):
    return W.box([0.5 * i for i in range(nx + 1)], [0.4 * i for i in range(ny + 1)], [-0.3 * i for i in range(slabs + 1)],
                 p, W.FUSED_SILICA)


def elements(d):
    return (len(d["x_breaks"]) - 1) * (len(d["y_breaks"]) - 1) * (len(d["slab_z"]) - 1)


# columns along x in SMs and ones, columns along y, slabs
SIZES = [((1, -1), 2, 1), ((1, 0), 2, 1), ((2, 1), 2, 1), ((1, 5), 3, 2), ((4, -1), 1, 2), ((4, 0), 1, 2),
         ((4, 1), 1, 2)]


@pytest.mark.parametrize("p", [2, 5])
@pytest.mark.parametrize("cols,ny,slabs", SIZES)
def test_elements_spread_over_ctas(cols, ny, slabs, p):
    """Alone, and in a batch whose launches are split otherwise."""
    from paper_2111_06893_gb300 import thermonoise
    desc = block(cols[0] * sms() + cols[1], ny, slabs, p)
    assert (elements(desc) > few_limit()) == (cols == (4, 1))
    alone = thermonoise.setup(desc)
    batch = thermonoise.Context().build_batch([desc, block(60, 60, 1, 2)])
    for dtype in (torch.float64, torch.float32):
        u = field(batch.ndof, dtype, seed=p)
        y = batch.apply_operator(u)[:alone.ndof]
        assert torch.equal(y, alone.apply_operator(u[:alone.ndof].clone())), dtype


@pytest.mark.parametrize("cols,ny,slabs", [((1, 5), 3, 2), ((4, 1), 1, 2)])
def test_residual_update_over_split_elements(cols, ny, slabs):
    """The same launch inside a PCG iteration: the solve's recursive residual
    has to agree with the true one it returns."""
    from paper_2111_06893_gb300 import thermonoise
    ctx = thermonoise.setup(block(cols[0] * sms() + cols[1], ny, slabs, 2))
    ctx.set_beam(1.0, 1.0)
    for mode in ("f64", "mixed"):
        _, rep = ctx.solve(mode=mode, rtol=1e-9)
        assert rep["rel_residual"] <= 1e-9
