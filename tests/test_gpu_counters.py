"""The launch counters: kernel_launches against the profiler's count of kernels,
list_launches where one of a call's two lists is missing."""
import numpy as np
import pytest

from paper_1807_10459_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("dims,listed", [((1, 1, 2), 1), ((2, 1, 1), 1), ((1, 1, 0), 0),
                                         ((1, 2, 0), 1)])
def test_launches_are_counted(dims, listed):
    """At most 4096 samples, where a sort of CUB's is one kernel."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    from paper_1807_10459_gb300 import build
    build.build()
    from torch.profiler import ProfilerActivity, profile
    g = synth.gaussian_problem(1500, *dims, seed=3)
    dev = [_dev(g.x), _dev(g.y), _dev(g.z if dims[2] else None)]
    for kernel in (idtx.KERNEL_LIST, idtx.KERNEL_TILE):
        ctx = idtx.Context(0)
        ctx.set_kernel(kernel)

        def call():
            idtx.cmi_ksg(*dev, k=4, n_surr=40, seed=2, ctx=ctx)
            torch.cuda.synchronize()

        call()
        with profile(activities=[ProfilerActivity.CUDA]):
            call()  # the profiler's own start-up
        ctx.reset_stats()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
        st = ctx.stats()
        names = [e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA]
        kernels = [n for n in names if not n.startswith("Mem")]
        if not kernels:
            pytest.skip("the profiler sees no kernels here")
        assert st["kernel_launches"] == len(kernels), kernels
        assert st["fused_launches"] == 1
        assert st["list_launches"] == (listed if kernel == idtx.KERNEL_LIST else 0)
