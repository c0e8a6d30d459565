"""Both occupancy variants of the FP32 operator kernel where they are used:
meshes and batches above the few-element limit (8 per SM), every degree.

Results do not depend on the variant, so they are compared bit by bit; FP32
against FP64 within 2e-5, as elsewhere."""
import numpy as np
import pytest

import workloads as W
from cases import box_layers, cyl_small

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


@pytest.mark.parametrize("p", range(2, 9))
def test_variants_of_many_elements_bit_identical(p):
    from paper_2111_06893_gb300 import thermonoise
    desc = block(-(-(few_limit() + 1) // 6), 3, 2, p)
    assert elements(desc) > few_limit()
    ctx = thermonoise.setup(desc)
    u = field(ctx.ndof, torch.float32, seed=p)
    ys = []
    for v in (0, 1):
        ctx.set_apply_variant(p, v)
        assert ctx.apply_tuning()[p]["variant"] == v
        ys.append(ctx.apply_operator(u))
    assert torch.equal(ys[0], ys[1])
    y64 = ctx.apply_operator(u.double())
    assert float((ys[0].double() - y64).abs().max() / y64.abs().max()) < 2e-5


def test_variants_of_a_large_batch_bit_identical():
    """Every degree, one variant throughout and both mixed over the degrees."""
    from paper_2111_06893_gb300 import thermonoise
    descs = [cyl_small(p, 1 + p % 2) for p in range(2, 9)] + [box_layers(4), block(-(-few_limit() // 4), 2, 2, 2)]
    bc = thermonoise.Context().build_batch(descs)
    u = field(bc.ndof, torch.float32, seed=1)
    ys = []
    for pick in (lambda p: 0, lambda p: 1, lambda p: p % 2):
        for p in range(2, 9):
            bc.set_apply_variant(p, pick(p))
        ys.append(bc.apply_operator(u))
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])
    y64 = bc.apply_operator(u.double())
    for i in range(len(descs)):
        a, b = (v[bc.dof_off[i]:bc.dof_off[i + 1]].double() for v in (ys[0], y64))
        assert float((a - b).abs().max() / b.abs().max()) < 2e-5, i


def test_tuner_settles_a_batch_on_one_variant():
    """By the sums over the degrees it times; a degree the caller has fixed
    keeps its variant and is not timed."""
    from paper_2111_06893_gb300 import thermonoise
    descs = [W.sweep_instance(i) for i in range(40)]
    for fixed in (None, 6):
        bc = thermonoise.Context().build_batch(descs)
        if fixed:
            bc.set_apply_variant(fixed, 1)
        bc.apply_operator(field(bc.ndof, torch.float32, seed=2))
        t = bc.apply_tuning()
        assert set(t) == {d["degree"] for d in descs} and len(t) == 5
        timed = [v for p, v in t.items() if p != fixed]
        us0, us1 = (sum(v["us"][i] for v in timed) for i in (0, 1))
        assert us0 > 0 and us1 > 0
        assert {v["variant"] for v in timed} == {1 if us1 < 0.98 * us0 else 0}
        if fixed:
            assert t[fixed] == {"variant": 1, "us": [0.0, 0.0]}
