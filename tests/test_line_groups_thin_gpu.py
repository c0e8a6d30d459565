"""The FP64 grouped-line solve (independent slab products, chains of interface
numbers) on long thin stacks: its error against that of the serial block
elimination, slab after slab, with the same explicit inverses.

The error is the residual of a group's solve scaled by the block's diagonal,
max_i |r - B z|_i / (d_i sum_j d_j |z_j|), d = sqrt(diag B): thin and thick
slabs count alike, unlike in max|B| max|z|, which the stiffest dominate.
Residuals are formed in extended precision.  Both forms round the same
products in different orders, so the bound is eight times the serial form's
error."""
import numpy as np
import pytest

import workloads as W
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


def stack(thick, p):
    mats = [W.CRYSTAL_A if i % 2 == 0 else W.CRYSTAL_B for i in range(len(thick))]
    return W.cylinder(10.0, 10.0, thick, mats, W.FUSED_SILICA, 1, p, 4)


def serial_solve(B, r, slab):
    """Block elimination from the top slab down and back up."""
    n = slab.max() + 1
    at = [np.flatnonzero(slab == s) for s in range(n)]
    inv, w = [], []
    S, b = B[np.ix_(at[0], at[0])], r[at[0]]
    for s in range(n):
        inv.append(np.linalg.inv(S))
        w.append(inv[s] @ b)
        if s + 1 < n:
            O = B[np.ix_(at[s], at[s + 1])]
            S = B[np.ix_(at[s + 1], at[s + 1])] - O.T @ inv[s] @ O
            b = r[at[s + 1]] - O.T @ w[s]
    z = np.zeros_like(r)
    z[at[-1]] = w[-1]
    for s in range(n - 2, -1, -1):
        z[at[s]] = w[s] - inv[s] @ (B[np.ix_(at[s], at[s + 1])] @ z[at[s + 1]])
    return z


def scaled_residual(B, r, z):
    L = np.longdouble
    d = np.sqrt(np.diag(B))
    res = np.abs(r.astype(L) - B.astype(L) @ z.astype(L)).astype(np.float64)
    return float((res / d).max() / (d @ np.abs(z)))


@pytest.mark.parametrize("name", ["40 of 4e-4", "20 of 1e-4 to 5e-2"])
def test_chain_solve_on_thin_stacks(name):
    from paper_2111_06893_gb300 import thermonoise
    rng = np.random.default_rng(11)
    thick = np.exp(rng.uniform(np.log(1e-4), np.log(5e-2), 20)).tolist()
    desc = stack([4e-4] * 40, 3) if name.startswith("40") else stack(thick, 4)
    mesh = Mesh(desc)
    ctx = thermonoise.setup(desc)
    r = torch.tensor(W.random_field(desc, 31), dtype=torch.float64, device="cuda")
    z = ctx.precond_apply(r, precond="zgroup")
    sets, sizes = group_index_sets(mesh)
    per_slab = mesh.ncol * 3 * mesh.N ** 3
    x, y = torch.zeros_like(z), torch.empty_like(z)
    for size in sorted(set(sizes)):
        g = sets[int(rng.choice([i for i, s in enumerate(sizes) if s == size]))]
        at = torch.tensor(g, device="cuda")
        B = np.empty((len(g), len(g)))
        for j in range(len(g)):
            x[at[j]] = 1.0
            B[:, j] = ctx.apply_operator(x, y)[at].cpu().numpy()
            x[at[j]] = 0.0
        B = 0.5 * (B + B.T)
        rg, slab = r[at].cpu().numpy(), np.asarray(g) // per_slab
        ours = scaled_residual(B, rg, z[at].cpu().numpy())
        serial = scaled_residual(B, rg, serial_solve(B, rg, slab))
        assert ours <= 8.0 * serial, (size, ours, serial)
