"""The operator's kernel forms agree bit for bit: few elements (three threads
per pencil, one element per CTA; several in a batch) and many (one thread per
pencil), for every degree, boundary condition and face orientation; the
oracle parity of the few-element form then carries over.  A captured apply
owns its scratch: replays may overlap."""
import numpy as np
import pytest

import workloads as W
from cases import box_layers, box_tiny, cyl_small

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


@pytest.mark.parametrize("p", range(2, 9))
def test_few_and_many_element_forms_bit_identical(p):
    """Each mirror alone and in a batch of few elements (three threads per
    pencil) against the same mirrors in a batch filled up with a mesh of 2304
    elements (one thread per pencil)."""
    from paper_2111_06893_gb300 import thermonoise
    mirrors = [cyl_small(p, 1), cyl_small(p, 2, bc_side="fixed", bc_bottom="free"), box_layers(p), box_tiny(p)]
    br = [float(i) for i in range(17)]
    filler = W.box(br, br, [-0.5 * i for i in range(10)], 2, W.FUSED_SILICA)
    few = thermonoise.Context().build_batch(mirrors)
    many = thermonoise.Context().build_batch(mirrors + [filler])
    n = few.ndof
    for dtype in (torch.float64, torch.float32):
        u = field(many.ndof, dtype, seed=p)
        y = many.apply_operator(u)[:n]
        assert torch.equal(y, few.apply_operator(u[:n].clone())), dtype
        for i, d in enumerate(mirrors):
            lo, hi = few.dof_off[i], few.dof_off[i + 1]
            yi = thermonoise.setup(d).apply_operator(u[lo:hi].clone())
            assert torch.equal(y[lo:hi], yi), (dtype, i)


def test_captured_applies_overlap():
    from paper_2111_06893_gb300 import thermonoise
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        ctx = thermonoise.setup(cyl_small(5, 2), stream=st)
        u = [field(ctx.ndof, torch.float64, s) for s in (1, 2)]
        ref = [ctx.apply_operator(v) for v in u]
        y = [torch.zeros_like(v) for v in u]
    graphs = []
    for v, w in zip(u, y):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            ctx.apply_operator(v, w)
        graphs.append(g)
    torch.cuda.synchronize()
    side = [torch.cuda.Stream() for _ in graphs]
    for _ in range(20):
        for g, s in zip(graphs, side):
            with torch.cuda.stream(s):
                g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(y, ref))
