"""List building where it can go wrong: more queries than one chunk of scratch,
an odd query count, scratch buffers that overflow (a radius sampled too wide)
and runs of equal distances longer than a sorting bin.  The estimates, eps and
counts over the lists are compared with the tile kernel's, which uses no lists
(bit for bit, as both sum in the same order), or with the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1807_10459_gb300 import synth

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


def _both(idtx, x, y, z, caps, S=2, k=4, full=True):
    out = []
    for kernel in (idtx.KERNEL_LIST, idtx.KERNEL_TILE):
        ctx = idtx.Context(0)
        ctx.set_kernel(kernel)
        ctx.set_list_caps(*caps)
        dev = [None if c is None else torch.from_numpy(np.ascontiguousarray(c)).cuda()
               for c in (x, y, z)]
        r = idtx.cmi_ksg(*dev, k=k, n_surr=S, seed=11, want_eps=full, want_counts=full, ctx=ctx)
        out.append([t.cpu().numpy() for t in (r if full else (r,))])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    return out[0]


@pytest.mark.parametrize("n,dims,caps", [
    (18501, (1, 1, 2), (0, 0)),      # two chunks of scratch, the second one short
    (4097, (1, 1, 7), (96, 160)),    # a tile of one sample; first dimensions tested first
    (2047, (2, 2, 3), (512, 1024)),
    (700, (1, 1, 1), (32, 64)),
])
def test_lists_give_the_tile_kernels_results(idtx, n, dims, caps):
    g = synth.gaussian_problem(n, *dims, seed=n)
    _both(idtx, g.x, g.y, g.z, caps)


def test_lists_of_uneven_density_and_equal_distances(idtx):
    """Half of the samples in tight clusters the sampled rows hardly meet, a
    fifth on a coarse grid (equal distances by the hundred), the rest wide."""
    rng = np.random.default_rng(8)
    n = 1500
    s = rng.standard_normal((4, n)) * 5
    c = rng.random(n) < 0.5
    s[:, c] = rng.integers(0, 3, (4, c.sum())) + 1e-4 * rng.standard_normal((4, c.sum()))
    g = rng.random(n) < 0.2
    s[:, g] = rng.integers(-2, 3, (4, g.sum()))
    s = s.astype(np.float32)
    x, y, z = s[:1], s[1:2], s[2:]
    for caps in ((32, 32), (96, 160), (512, 1024)):
        _, eps, cnt = _both(idtx, x, y, z, caps)
        e, a, b, d = oracle.ksg_counts(x, y, z, 4)
        assert np.array_equal(eps[0], e)
        assert np.array_equal(cnt[0], np.stack([a, b, d]))


@pytest.mark.parametrize("n", [65536, 65537])
def test_both_forms_of_the_list_kernel_at_their_boundary(idtx, n):
    """Up to 65536 samples the counts leave the list kernel as 16-bit numbers,
    above as 32-bit ones."""
    g = synth.gaussian_problem(n, 1, 1, 2, seed=9)
    _both(idtx, g.x, g.y, g.z, (256, 512), S=1)


def test_more_groups_than_the_count_buffers_hold(idtx):
    """1301 estimates of 65537 samples: the counts of 40 groups fit, so 41 take
    two turns, the second one with 21 jobs."""
    g = synth.gaussian_problem(65537, 1, 1, 3, seed=4)
    _both(idtx, g.x, g.y, g.z, (64, 128), S=1300, full=False)


@pytest.mark.parametrize("n,S,caps", [(129, 0, (32, 32)), (1000, 33, (32, 64)), (3000, 95, (96, 96))])
def test_queued_full_scans(idtx, n, S, caps):
    """Lists so short that most (query, group)s, some, or the far ones only go
    to the scan kernel, with one job in the last group and with full groups."""
    g = synth.gaussian_problem(n, 1, 1, 3, seed=n)
    _both(idtx, g.x, g.y, g.z, caps, S=S)


@pytest.mark.parametrize("dims", [(1, 1, 0), (1, 2, 0), (2, 1, 0), (1, 1, 1), (2, 2, 1), (3, 1, 1)])
@pytest.mark.parametrize("n,k", [(257, 4), (1100, 4), (3001, 4), (700, 7)])
def test_at_most_one_z_column(idtx, dims, n, k):
    """Walks over the order by the z or y column and counts in sorted columns
    instead of lists: against the tile kernel and the oracle, on continuous
    data and on data full of equal values."""
    g = synth.gaussian_problem(n, *dims, seed=n + k)
    rng = np.random.default_rng(n)
    for grid in (False, True):
        x, y, z = (rng.integers(-3, 4, c.shape).astype(np.float32) if grid else c
                   for c in (g.x, g.y, g.z))
        cmi, eps, cnt = _both(idtx, x, y, z if dims[2] else None, (0, 0), S=34, k=k)
        e, a, b, c = oracle.ksg_counts(x, y, z if dims[2] else None, k)
        assert np.array_equal(eps[0], e)
        assert np.array_equal(cnt[0], np.stack([a, b, c]))
        ref = oracle.cmi_surrogates(x, y, z if dims[2] else None, k, 1, 11)
        assert np.max(np.abs(cmi[:2] - ref)) < 1e-10


def test_long_runs_of_equal_distances(idtx):
    """Distances in a few far-apart values, each many hundred times: bins that
    the second binning cannot split, cut lists that end inside one."""
    rng = np.random.default_rng(2)
    n = 2600
    z = rng.choice(np.array([0.0, 1.0, 1.0 + 1e-6, 1000.0], np.float32), (2, n))
    x, y = (rng.standard_normal((1, n)).astype(np.float32) * 1e-3 for _ in range(2))
    for caps in ((64, 96), (0, 0)):
        _, eps, cnt = _both(idtx, x, y, z, caps)
        e, a, b, c = oracle.ksg_counts(x, y, z, 4)
        assert np.array_equal(eps[0], e)
        assert np.array_equal(cnt[0], np.stack([a, b, c]))
