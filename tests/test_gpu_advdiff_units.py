"""The 2D system in other units.  It is linear, so the states, the observations and
their noise times a power of two give the same weights and the same states times it,
whatever the kernels sum their squared error estimates in: two epochs against
the CPU oracle within the repository's bounds, and against the unscaled epochs."""
import numpy as np
import pytest

import oracle
from paper_1411_1702_gb300 import build as B
from paper_1411_1702_gb300 import workloads as W
from parity_util import check_epoch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    B.build()
    oracle.build()
    from paper_1411_1702_gb300 import pf as _pf
    return _pf


def _scaled(n, N, T, k):
    w = W.advdiff(n, N, T)
    s = 2.0 ** k
    return w.with_(x0=w.x0 * s, y_obs=w.y_obs * s, x_true=w.x_true * s, sigma=[30.0 * v * s for v in w.sigma])


@pytest.mark.parametrize("n,N,T", [(20, 9, 2), (40, 3, 1)])
@pytest.mark.parametrize("k", [34, 45, 70, -30, -60])
def test_scaled_epochs(pf, n, N, T, k):
    runs = []
    for w in (_scaled(n, N, T, 0), _scaled(n, N, T, k)):
        g, o = pf.Filter.from_workload(w), oracle.Filter(w)
        o.init()
        for j in range(T):
            check_epoch(g, o, w.t_obs[j], w.y_obs[j])
        runs.append(g.pf_get_ensemble())
        g.close()
    a, b = runs
    # both sides carry the oracle's state bound (1e-10)
    for key in ("x", "h1", "h2"):
        top = np.max(np.abs(a[key]), axis=1, keepdims=True)
        assert np.all(np.abs(b[key] * 2.0 ** -k - a[key]) <= 2e-10 * top)
    assert np.all(np.isfinite(b["lw"]))
