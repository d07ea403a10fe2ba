"""The gather of many job groups with their source columns in shared memory:
one source over partial tiles and chunks, and groups that two candidates of a
greedy step share, against the oracle."""
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


@pytest.mark.parametrize("n,S", [(257, 2015), (320, 2048), (2305, 2079)])
def test_one_source(idtx, n, S):
    """64 groups, full; 65, the last of one job; 65, 2305 rows in two chunks."""
    g = synth.gaussian_problem(n, 1, 1, 2, seed=n)
    dev = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (g.x, g.y, g.z)]
    got = idtx.cmi_ksg(*dev, k=4, n_surr=S, seed=11, ctx=idtx.Context(0)).cpu().numpy()
    m = S if n < 1000 else 40
    ref = oracle.cmi_surrogates(g.x, g.y, g.z, 4, m, 11)
    assert np.max(np.abs(got[: m + 1] - ref)) < 1e-10
    if m < S:  # the others against a call of few groups, by the other gather
        few = idtx.cmi_ksg(*dev, k=4, n_surr=1500, seed=11, ctx=idtx.Context(0)).cpu().numpy()
        assert np.array_equal(got[:1501], few)


def test_two_sources_in_a_group(idtx):
    net = synth.var_network(n_nodes=5, order=3, T=420, density=0.4, weight=0.6, seed=21)
    S = 200   # 201 estimates a candidate: groups of 32 straddle two of them
    ref = oracle.select_target(net.series, 0, n_past=2, min_lag=1, max_lag=3, k=4, n_surr=S,
                               alpha=0.05, seed=17, max_parents=1, want_first_step=True)
    _, est = idtx.mte_step(torch.from_numpy(net.series).cuda(), 0, 2, 1, 3, (), 0, k=4, n_surr=S,
                           alpha=0.05, seed=17, want_estimates=True, ctx=idtx.Context(0))
    alive = ~np.isnan(ref["first_step"][:, 0])
    assert alive.sum() * (S + 1) > 64 * 32
    assert np.max(np.abs(est[alive] - ref["first_step"][alive])) < 1e-10
    bad = net.series.copy()
    bad[3, 100] = np.nan
    with pytest.raises(Exception):
        idtx.mte_step(torch.from_numpy(bad).cuda(), 0, 2, 1, 3, (), 0, k=4, n_surr=S, seed=17,
                      ctx=idtx.Context(0))
