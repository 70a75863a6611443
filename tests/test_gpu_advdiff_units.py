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
@pytest.mark.parametrize("k", [34, 45, 70, 300, -30, -60, -300])
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


@pytest.mark.parametrize("n,N,full", [(20, 3, 4), (8, 5, 8), (8, 7, 8)])
def test_ragged_last_block(pf, n, N, full):
    """The particles of a ragged last block have the states, to the last bit, that they have
    in a full one (equal ensembles and moments, resampling by equal weights)."""
    out = []
    for size in (N, full):
        w = _scaled(n, size, 1, 0)
        f = pf.Filter.from_workload(w)
        f.pf_set_ensemble(phi=np.tile(w.theta_true, (size, 1)), x=np.tile(w.x0, (size, 1)))
        f.pf_set_moments(w.theta_true, 0.01 * np.eye(5))
        f.pf_assimilate(w.t_obs[0], w.y_obs[0])
        assert np.array_equal(f.pf_get_work()["idx"], np.arange(size))
        out.append(f.pf_get_ensemble())
        f.close()
    for key in ("x", "h1", "h2", "phi"):
        assert np.array_equal(out[0][key], out[1][key][:N]), key


@pytest.mark.parametrize("n,N", [(8, 7), (20, 9)])
def test_dead_neighbours(pf, n, N):
    """Particles that share a block with ones that are not finite, and the ragged last
    block, have the states they have without them (to the state bound)."""
    w = _scaled(n, N, 1, 0)
    out = []
    for bad in (False, True):
        f = pf.Filter.from_workload(w, N=N)
        if bad:
            x = f.pf_get_ensemble()["x"]
            x[[1, 4], 3] = np.nan, -np.inf
            f.pf_set_ensemble(x=x)
        f.pf_assimilate(w.t_obs[0], w.y_obs[0])
        out.append((f.pf_get_work()["lg"], f.pf_get_ensemble()["x"]))
        f.close()
    (lg0, x0), (lg1, x1) = out
    live = np.setdiff1d(np.arange(N), [1, 4])
    assert np.isneginf(lg1[[1, 4]]).all()
    # (log weights: the repository's log-likelihood bound; every resampled state is one of the live ones')
    assert np.all(np.abs(lg1[live] - lg0[live]) <= 1e-9 * (1 + np.abs(lg0[live])))
    assert np.isfinite(x1).all()
