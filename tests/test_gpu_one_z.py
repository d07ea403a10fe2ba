"""One z column: n_z by bisection of what the count walk reached, over list B
(calls without the order by z: up to 256 samples, above 65536) and over the
order's two sides, with equal values and samples at either end of the order."""
import numpy as np
import pytest

import oracle
from paper_1807_10459_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dims,caps", [(40, (1, 1, 1), (32, 32)), (256, (2, 1, 1), (0, 0)),
                                         (257, (1, 2, 1), (32, 0)), (1500, (1, 1, 1), (0, 0)),
                                         (65700, (1, 1, 1), (256, 512))])
def test_one_z_column(n, dims, caps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    from paper_1807_10459_gb300 import build
    build.build()
    g = synth.gaussian_problem(n, *dims, seed=n)
    for grid in (False, True):
        x, y, z = g.x, g.y, (np.round(g.z) if grid else g.z).astype(np.float32)
        dev = [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in (x, y, z)]
        out = []
        for kernel in (idtx.KERNEL_LIST, idtx.KERNEL_TILE):
            ctx = idtx.Context(0)
            ctx.set_kernel(kernel)
            ctx.set_list_caps(*caps)
            out.append([t.cpu().numpy() for t in idtx.cmi_ksg(
                *dev, k=4, n_surr=3, seed=11, want_eps=True, want_counts=True, ctx=ctx)])
        for a, b in zip(*out):
            assert np.array_equal(a, b)
        if n < 2000:
            e, a, b, c = oracle.ksg_counts(x, y, z, 4)
            assert np.array_equal(out[0][1][0], e)
            assert np.array_equal(out[0][2][0], np.stack([a, b, c]))
