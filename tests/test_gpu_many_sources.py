"""Calls without z: the source columns sorted together, at the edges of the
tiles (1024) and of one column's other sort (4096), on continuous data and on
data full of equal values, against the tile kernel; and no more launches for
more sources."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def idtx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as m
    from paper_1807_10459_gb300 import build
    build.build()
    return m


def _ctx(idtx, kernel):
    ctx = idtx.Context(0)
    ctx.set_kernel(kernel)
    return ctx


@pytest.mark.parametrize("n", [257, 1024, 1025, 2049, 4097, 9000])
@pytest.mark.parametrize("grid", [False, True])
def test_step_without_target_past(idtx, n, grid):
    rng = np.random.default_rng(n)
    s = rng.standard_normal((3, n + 2)).astype(np.float32)
    s = torch.from_numpy(np.round(s * 4) if grid else s).cuda()
    out = [idtx.mte_step(s, 0, 0, 1, 2, (), 0, k=4, n_surr=3, seed=9, want_estimates=True,
                         ctx=_ctx(idtx, kern)) for kern in (idtx.KERNEL_LIST, idtx.KERNEL_TILE)]
    assert np.array_equal(out[0][1], out[1][1], equal_nan=True)
    assert tuple(out[0][0]) == tuple(out[1][0])


@pytest.mark.parametrize("n", [4096, 4097, 65536])
def test_one_source(idtx, n):
    rng = np.random.default_rng(n)
    x, y = (torch.from_numpy(rng.standard_normal((1, n)).astype(np.float32)).cuda() for _ in range(2))
    a, b = (idtx.cmi_ksg(x, y, None, k=4, n_surr=1, seed=9, ctx=_ctx(idtx, kern))
            for kern in (idtx.KERNEL_LIST, idtx.KERNEL_TILE))
    assert torch.equal(a, b)


def test_launches_do_not_grow_with_the_sources(idtx):
    rng = np.random.default_rng(1)
    launches = []
    for nodes in (3, 30):
        s = torch.from_numpy(rng.standard_normal((nodes, 902)).astype(np.float32)).cuda()
        ctx = _ctx(idtx, idtx.KERNEL_LIST)
        for _ in range(2):
            ctx.reset_stats()
            idtx.mte_step(s, 0, 0, 1, 2, (), 0, k=4, n_surr=3, seed=9, ctx=ctx)
        launches.append(ctx.stats()["kernel_launches"])
    assert launches[0] == launches[1]
