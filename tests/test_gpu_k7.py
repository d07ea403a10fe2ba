"""The runtime-k specialisations for k <= 7 against the oracle: every k, their
dimensions with and without zero padding, and one dimension or k more, which
goes to the generic one."""
import numpy as np
import pytest

import oracle
from paper_1807_10459_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 0), (1, 1, 1), (2, 1, 1), (1, 2, 2), (2, 2, 3), (1, 1, 4),
                                  (2, 1, 7), (1, 2, 11), (2, 3, 2), (3, 1, 1)])
@pytest.mark.parametrize("n,k", [(9, 7), (300, 1), (300, 2), (700, 3), (700, 5), (1030, 6),
                                 (1030, 7), (1030, 8)])
def test_both_kernels_match_the_oracle(dims, n, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    from paper_1807_10459_gb300 import build
    build.build()
    g = synth.gaussian_problem(n, *dims, seed=n + k)
    z = g.z if dims[2] else None
    e, a, b, c = oracle.ksg_counts(g.x, g.y, z, k)
    ref = oracle.cmi_surrogates(g.x, g.y, z, k, 2, 11)
    dev = [None if v is None else torch.from_numpy(np.ascontiguousarray(v)).cuda()
           for v in (g.x, g.y, z)]
    for kernel in (idtx.KERNEL_TILE, idtx.KERNEL_LIST):
        ctx = idtx.Context(0)
        ctx.set_kernel(kernel)
        ctx.set_list_caps(64, 96)
        cmi, eps, cnt = (t.cpu().numpy() for t in idtx.cmi_ksg(
            *dev, k=k, n_surr=2, seed=11, want_eps=True, want_counts=True, ctx=ctx))
        assert np.array_equal(eps[0], e)
        assert np.array_equal(cnt[0], np.stack([a, b, c]))
        assert np.max(np.abs(cmi - ref)) < 1e-10
