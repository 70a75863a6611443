"""One and two Newton iterations a substep, where the Brusselator's substeps in increments
and in FP64 take turns: the K-th iterate from the predictor, to FP64's rounding, against the
oracle's."""
import numpy as np
import pytest

import oracle
from paper_1411_1702_gb300 import build as B
from paper_1411_1702_gb300 import workloads as W
from parity_util import begin_epoch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,S", [(2, 5), (2, 20), (1, 5), (1, 20)])
def test_kth_iterate(K, S):
    B.build()
    oracle.build()
    from paper_1411_1702_gb300 import pf
    w = W.brusselator(N=64, T=4)
    w = w.with_(newton_iters=K, substeps=S, dt=1 / (3.0 * S), kappa=1e-60, sigma=[1.0] * 8)
    g, o = pf.Filter.from_workload(w), oracle.Filter(w)
    o.init()
    for k in range(4):
        begin_epoch(g, o)
        g.pf_assimilate(w.t_obs[k], w.y_obs[k])
        tab, n = o.substeps(w.t_obs[k])
        assert n == S and o.stage1(tab, n, w.y_obs[k]) == oracle.OK and o.cumulative() == oracle.OK
        assert o.stage2(tab, n, w.y_obs[k], g.pf_get_work()["idx"]) == oracle.OK and o.commit(w.t_obs[k]) == oracle.OK
        a, b = g.pf_get_ensemble(), o.state()
        for key in ("x", "h1", "h2"):
            # a few roundings a substep on both sides, and their growth over an interval
            assert np.max(np.abs(a[key] - b[key]) / np.abs(b[key])) <= 16 * S * 2.0 ** -53, (k, key)
    g.close()
