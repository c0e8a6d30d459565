"""Layer energies and their parts for every degree, one element per CTA (small
meshes) and full CTAs with a last one partly filled (a batch of many
elements), against the oracle.  Tolerances: 1e-12 relative, as for the other
energy tests (sums of ~10^4 terms of one sign per layer); parts agree with
the energies to the same; a batch sums an element's energies in another order
than a mirror alone, 1e-13."""
import numpy as np
import pytest

import workloads as W
from cases import box_layers, box_tiny, cyl_small
from oracle import Mesh, Operator, observables as ob

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_06893_gb300 import build
    build.build()


@pytest.mark.parametrize("p", range(2, 9))
def test_energies_of_every_degree(p):
    from paper_2111_06893_gb300 import thermonoise
    br = [0.1 * i for i in range(14)]
    filler = W.box(br, br, [-0.5 * i for i in range(12)], p, W.FUSED_SILICA)  # 1859 elements
    mirrors = [cyl_small(p, 1), box_layers(p), box_tiny(p), filler]
    batch = thermonoise.Context().build_batch(mirrors)
    u = torch.tensor(np.random.default_rng(p).uniform(-1, 1, batch.ndof), dtype=torch.float64, device="cuda")
    Ub = np.asarray(batch.layer_energies(u))
    Pb = np.asarray(batch.layer_energy_parts(u)).reshape(-1, 3)
    at = 0
    for i, d in enumerate(mirrors):
        ui = u[batch.dof_off[i]:batch.dof_off[i + 1]].clone()
        U = np.asarray(thermonoise.setup(d).layer_energies(ui))
        if i < 3:
            Uo = ob.layer_energies(Operator(Mesh(d)), ui.cpu().numpy())
            assert np.max(np.abs(U - Uo) / np.abs(Uo)) < 1e-12
        sl = slice(at, at + len(U))
        at += len(U)
        assert np.max(np.abs(Ub[sl] - U) / U) < 1e-13
        assert np.max(np.abs(Pb[sl].sum(axis=1) - U) / U) < 1e-12
