"""The bits of an estimate: the sum over the samples is exact and rounded once,
so they depend neither on the kernel nor on the call that computes it (the
specialisation, its query tiles, the order of the samples)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1807_10459_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("k", [3, 4, 7])
def test_batch_kernel_and_schedule_do_not_change_the_bits(k):
    """One problem of three x columns takes the others of a batch of another k
    to a wider specialisation; one or no z column changes the samples' order."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    from paper_1807_10459_gb300 import build
    build.build()
    shapes = [(700, 1, 1, 2), (1030, 1, 1, 2), (385, 2, 1, 3), (260, 1, 2, 1), (129, 1, 1, 2),
              (300, 3, 1, 1), (1100, 1, 1, 0), (257, 2, 2, 0)]
    probs = []
    for i, (n, dx, dy, dz) in enumerate(shapes):
        g = synth.gaussian_problem(n, dx, dy, dz, seed=60 + i)
        probs.append((g.x, g.y, g.z if dz else None))
    dev = [dict(x=_dev(x), y=_dev(y), z=_dev(z), n_surr=9, seed=5 + i)
           for i, (x, y, z) in enumerate(probs)]
    got = {}
    for kernel in (idtx.KERNEL_TILE, idtx.KERNEL_LIST, idtx.KERNEL_AUTO):
        ctx = idtx.Context(0)
        ctx.set_kernel(kernel)
        got["batch", kernel] = idtx.cmi_batch(dev, k=k, ctx=ctx)
        for mode in (idtx.MODE_BATCHED, idtx.MODE_PLAIN):
            got[mode, kernel] = [
                idtx.cmi_ksg(p["x"], p["y"], p["z"], k=k, n_surr=9, seed=p["seed"], mode=mode,
                             ctx=ctx) for p in dev]
    want = [o.cpu().numpy() for o in got["batch", idtx.KERNEL_TILE]]
    for key, out in got.items():
        for i, (a, b) in enumerate(zip(want, out)):
            assert np.array_equal(a, b.cpu().numpy()), (key, shapes[i])
    for (x, y, z), p, a in zip(probs, dev, want):
        ref = oracle.cmi_surrogates(x, y, z, k, 2, p["seed"])
        assert np.max(np.abs(a[:3] - ref)) < 1e-10


def test_the_allocation_free_entry_point_gives_the_same_bits():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    lib = idtx.load()
    vp, ci, cl = ctypes.c_void_p, ctypes.c_int, ctypes.c_int64
    lib.idtx_cmi_ksg_noalloc.argtypes = [vp, ci, vp, ci, vp, ci, cl, cl,
                                         ctypes.POINTER(idtx.Settings), vp, vp]
    for n, dx, dy, dz, k in [(1000, 1, 1, 2, 4), (601, 2, 1, 1, 3)]:
        g = synth.gaussian_problem(n, dx, dy, dz, seed=n)
        x, y, z = _dev(g.x), _dev(g.y), _dev(g.z)
        out = torch.empty(8, dtype=torch.float64, device="cuda")
        s = idtx.Settings(k, 7, 3, 0.05, 0, 0)
        assert lib.idtx_cmi_ksg_noalloc(x.data_ptr(), dx, y.data_ptr(), dy, z.data_ptr(), dz, n, n,
                                        ctypes.byref(s), out.data_ptr(),
                                        torch.cuda.current_stream().cuda_stream) == 0
        assert torch.equal(out, idtx.cmi_ksg(x, y, z, k=k, n_surr=7, seed=3))
