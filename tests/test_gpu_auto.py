"""The kernel choice without a trial, where one kernel is always the faster."""
import numpy as np
import pytest

import oracle
from paper_1807_10459_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n,dims,k,trials", [(64, (1, 1, 2), 4, 1), (65, (1, 1, 2), 4, 0),
                                             (511, (2, 1, 1), 3, 0), (512, (1, 1, 2), 4, 1),
                                             (2000, (1, 1, 0), 4, 0), (2000, (1, 2, 0), 4, 1),
                                             (2000, (2, 1, 0), 4, 0), (385, (2, 1, 0), 3, 0),
                                             (2430, (2, 2, 0), 7, 0), (2433, (2, 2, 0), 7, 0)])
def test_trials(n, dims, k, trials):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    from paper_1807_10459_gb300 import build
    build.build()
    g = synth.gaussian_problem(n, *dims, seed=n)
    z = g.z if dims[2] else None
    ctx = idtx.Context(0)
    for _ in range(2):
        got = idtx.cmi_ksg(_dev(g.x), _dev(g.y), _dev(z), k=k, n_surr=5, seed=2, ctx=ctx)
    assert ctx.stats()["tune_trials"] == trials
    ref = oracle.cmi_surrogates(g.x, g.y, z, k, 5, 2)
    assert np.max(np.abs(got.cpu().numpy() - ref)) < 1e-10


def test_a_call_of_one_estimate_after_a_trial_of_many():
    """A trial's times of 32 job groups do not fall to a 32nd for one group, which
    leaves most SMs idle: the lists, half as long as the tile kernel there, are
    still taken."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    g = synth.gaussian_problem(2000, 1, 1, 2, seed=3)
    dev = [_dev(v) for v in (g.x, g.y, g.z)]
    ctx = idtx.Context(0)
    idtx.cmi_ksg(*dev, k=4, n_surr=1000, seed=2, ctx=ctx)
    ctx.reset_stats()
    idtx.cmi_ksg(*dev, k=4, n_surr=0, seed=2, ctx=ctx)
    st = ctx.stats()
    assert st["tune_trials"] == 0 and st["list_launches"] == 1
