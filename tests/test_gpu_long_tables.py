"""Substep tables around the lengths at which they leave shared memory (276 substeps
with the increment form's table, 531 without), each family, filters alone and in a batch
with shorter ones: one epoch against the oracle within the repository's bounds."""
import numpy as np
import pytest

import oracle
from paper_1411_1702_gb300 import build as B
from paper_1411_1702_gb300 import workloads as W
from parity_util import begin_epoch, check_epoch, finish_epoch

pytestmark = pytest.mark.gpu


def _workload(problem, lmm, S, N=37):
    if problem == "linear2":
        w = W.linear2(N=N, T=2)
        hi = [10.0, 400.0] if lmm > 20 else w.prior_hi
        return w.with_(lmm=lmm, dt=0.1 / S, prior_hi=hi)
    w = W.robertson(N=N, T=2)
    return w.with_(lmm=lmm, spacing=W.SPACING_UNIFORM, dt=1e-4 / S, t_obs=np.array([1e-4, 2e-4]), noise=W.NOISE_ADDITIVE,
                   sigma=[0.01, 0.01])


@pytest.fixture(scope="module")
def pf():
    B.build()
    oracle.build()
    from paper_1411_1702_gb300 import pf as _pf
    return _pf


@pytest.mark.parametrize("problem,lmm,S", [("robertson", W.LMM_BDF2, 276), ("robertson", W.LMM_BDF2, 277), ("robertson", W.LMM_BDF2, 640),
                                           ("robertson", W.LMM_BDF3, 277), ("robertson", W.LMM_AM2, 640), ("robertson", W.LMM_BDF1, 531),
                                           ("robertson", W.LMM_BDF1, 532), ("linear2", W.LMM_BDF2, 531), ("linear2", W.LMM_BDF2, 532),
                                           ("linear2", W.LMM_BDF2, 640), ("linear2", W.LMM_AM3, 640), ("linear2", W.LMM_AB2, 640)])
def test_epochs(pf, problem, lmm, S):
    w = _workload(problem, lmm, S)
    g, o = pf.Filter.from_workload(w), oracle.Filter(w)
    o.init()
    for k in range(2):
        assert o.substeps(w.t_obs[k])[1] == S
        check_epoch(g, o, w.t_obs[k], w.y_obs[k], exempt_dead=True)
    g.close()


def test_batch_of_long_and_short(pf):
    """A batch reserves what its longest member takes and what its shorter ones do."""
    ws = [_workload("linear2", W.LMM_BDF2, S, N=129) for S in (640, 531, 40)]
    ws += [_workload("robertson", W.LMM_BDF2, S, N=129) for S in (640, 276, 30)]
    fs, os_ = [pf.Filter.from_workload(w) for w in ws], [oracle.Filter(w) for w in ws]
    for o in os_:
        o.init()
    batch = pf.Batch(fs)
    pre = [begin_epoch(f, o) for f, o in zip(fs, os_)]
    st = batch.pf_batch_assimilate([w.t_obs[0] for w in ws], [w.y_obs[0] for w in ws])
    assert st == [pf.PF_OK] * len(ws)
    for f, o, w, p in zip(fs, os_, ws, pre):
        finish_epoch(f, o, w.t_obs[0], w.y_obs[0], p, exempt_dead=True)
