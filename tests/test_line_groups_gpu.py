"""The FP64 grouped-line solve (chains of interface numbers) at its edges:
one slab, two, the block of slabs the chain kernel holds (32) less one, full,
plus one and several, every degree, groups of 1 to 4 lines; and a batch of
mirrors with different degrees and slab counts.

The blocks are applied with the operator itself (a vector that lives on one
group, restricted to the group), so no matrix is assembled.  Tolerances: the
residual of a group's solve relative to max|A| max|z| (A is positive definite:
its largest entry is on the diagonal) is held to 1e-13 on meshes of up to ten
slabs elsewhere; rounding errors add up at most linearly along the chain, so
1e-13 max(1, S / 10).  FP32 and FP64 solves agree within 2e-5."""
import numpy as np
import pytest

import workloads as W
from cases import cyl_small
from oracle import Mesh
from test_parity_gpu import group_index_sets

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_06893_gb300 import build
    build.build()


def columns(p, nslab):
    br = [-1.0, 0.2, 1.0]
    return W.box(br, br, [-0.3 * s for s in range(nslab + 1)], p, W.FUSED_SILICA)


CASES = [(2, 1), (3, 2), (4, 31), (5, 32), (6, 33), (7, 3), (8, 2), (2, 65), (3, 130)]


@pytest.mark.parametrize("p,nslab", CASES + [("cyl", 8), ("cyl", 5)])
def test_chain_solve_inverts_the_group_blocks(p, nslab):
    from paper_2111_06893_gb300 import thermonoise
    desc = cyl_small(nslab, 2) if p == "cyl" else columns(p, nslab)
    mesh = Mesh(desc)
    ctx = thermonoise.setup(desc)
    assert ctx.ndof == mesh.ndof
    S = mesh.nslab
    r = torch.tensor(W.random_field(desc, 7), dtype=torch.float64, device="cuda")
    z = ctx.precond_apply(r, precond="zgroup")
    z32 = ctx.precond_apply(r.float(), precond="zgroup").double()
    assert float((z32 - z).norm() / z.norm()) < 2e-5
    scale = float(ctx.diagonal().abs().max())
    sets, sizes = group_index_sets(mesh)
    assert set(sizes) >= ({1, 2, 3} if p == "cyl" else {1, 2, 4})
    rng = np.random.default_rng(3)
    pick = rng.permutation(len(sets))[:40].tolist() + [int(np.argmax(sizes)), int(np.argmin(sizes))]
    for g in pick:
        at = torch.tensor(sets[g], device="cuda")
        x = torch.zeros_like(z)
        x[at] = z[at]
        res = (ctx.apply_operator(x)[at] - r[at]).abs().max() / (scale * z[at].abs().max())
        assert float(res) < 1e-13 * max(1.0, S / 10), (g, sizes[g], float(res))


def test_chain_solve_of_a_batch_is_the_single_solves():
    from paper_2111_06893_gb300 import thermonoise
    mirrors = [columns(2, 33), columns(4, 1), cyl_small(4, 2), columns(2, 5), columns(4, 40)]
    batch = thermonoise.Context().build_batch(mirrors)
    r = torch.tensor(np.random.default_rng(5).uniform(-1, 1, batch.ndof), dtype=torch.float64, device="cuda")
    z = batch.precond_apply(r, precond="zgroup")
    for i, d in enumerate(mirrors):
        lo, hi = batch.dof_off[i], batch.dof_off[i + 1]
        zi = thermonoise.setup(d).precond_apply(r[lo:hi].clone(), precond="zgroup")
        assert torch.equal(z[lo:hi], zi), i


@pytest.mark.parametrize("nx", [30, 40])
def test_fp32_solve_of_many_packs(nx):
    """More packs of line groups than the GPU holds at once, several times over
    (nx = 40: the build with seven CTAs per SM; 30: four), against the FP64
    solve; 2e-5 as above.  Repeated, the work queue starts empty again."""
    from paper_2111_06893_gb300 import thermonoise
    br = [0.25 * i for i in range(nx + 1)]
    desc = W.box(br, br, [0.0, -0.3, -0.7], 2, W.FUSED_SILICA)
    ctx = thermonoise.setup(desc)
    r = torch.tensor(np.random.default_rng(nx).uniform(-1, 1, ctx.ndof), dtype=torch.float64, device="cuda")
    z = ctx.precond_apply(r, precond="zgroup")
    first = ctx.precond_apply(r.float(), precond="zgroup")
    assert float((first.double() - z).norm() / z.norm()) < 2e-5
    assert torch.equal(first, ctx.precond_apply(r.float(), precond="zgroup"))
