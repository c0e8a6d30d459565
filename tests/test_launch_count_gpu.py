"""The launches a solve reports are the kernels it runs (FP64 and mixed,
every preconditioner, one mesh and a batch), as the profiler counts them."""
import pytest

from cases import box_layers, cyl_small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2111_06893_gb300 import build
    build.build()
    kernels_of(lambda: torch.zeros(1, device="cuda"))  # the first profile of a process may stay empty


def kernels_of(call):
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA]
    return [n for n in names if not n.startswith(("Memcpy", "Memset"))]


@pytest.mark.parametrize("kind", ["mesh", "batch"])
@pytest.mark.parametrize("precond", ["jacobi", "zline", "zgroup"])
@pytest.mark.parametrize("mode", ["f64", "mixed"])
def test_reported_launches(kind, precond, mode):
    from paper_2111_06893_gb300 import thermonoise
    if kind == "mesh":
        ctx = thermonoise.setup(box_layers(3))
    elif precond == "jacobi":
        pytest.skip("a batch is solved with line blocks")
    else:
        ctx = thermonoise.Context().build_batch([cyl_small(3, 1), box_layers(3), box_layers(4), box_layers(3)])
    kw = dict(mode=mode, precond=precond, rtol=1e-8, raise_on_error=False, max_iter=300, max_outer=3)
    ctx.solve(**kw)  # factors, tuning
    rep = {}
    names = kernels_of(lambda: rep.update(ctx.solve(**kw)[1]))
    if not names:
        pytest.skip("no kernel records")
    assert rep["launches"] == len(names)
