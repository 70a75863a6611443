"""Error sums of the substeps (Step 4b) where the squared estimates leave the range of
floats: the Brusselator with a source that makes its states large, on the FP64 path
(parameters above 2^40) and before it, beyond the floats' own range, and tiny; and
Robertson with a history far from its state.  Against the CPU oracle within the
repository's bounds."""
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


@pytest.mark.parametrize("A,u0", [(2.0 ** 38, 2.0 ** 18), (2.0 ** 45, 2.0 ** 44), (2.0 ** 200, 2.0 ** 199),
                                  (2.0 ** -60, 2.0 ** -61), (2.0 ** -115, 2.0 ** -116)])
def test_brusselator_sources(pf, A, u0):
    """u' = A - u + ...: with v = 0, next to no B and no diffusion the rest vanishes beside A."""
    w = W.brusselator(N=11, T=3)
    eps = 2.0 ** -700
    x0 = np.zeros(64)
    x0[0::2] = u0 * (1 + np.arange(32) / 64)
    t = w.t_obs
    x_true = np.zeros((3, 64))
    for k in range(3):
        x_true[k, 0::2] = A + (x0[0::2] - A) * np.exp(-t[k])
    y = x_true[:, w.obs_idx] * 1.01
    w = w.with_(x0=x0, x_true=x_true, y_obs=y, sigma=[0.3 * A] * len(w.obs_idx), prior_lo=[0.5 * A, eps, eps],
                prior_hi=[1.5 * A, 2 * eps, 2 * eps])
    g, o = pf.Filter.from_workload(w), oracle.Filter(w)
    o.init()
    for k in range(3):
        check_epoch(g, o, w.t_obs[k], w.y_obs[k])
    assert np.isfinite(g.pf_get_ensemble()["lw"]).all()
    g.close()


@pytest.mark.parametrize("jump", [2.0 ** 10, 2.0 ** 29])
@pytest.mark.parametrize("lmm", [W.LMM_BDF2, W.LMM_BDF3])
def test_robertson_far_history(pf, lmm, jump):
    """A past `jump` away from the state, in a regime where the reactions are slow."""
    w = W.robertson(N=33, T=3)
    w = w.with_(lmm=lmm, spacing=W.SPACING_UNIFORM, dt=0.1, t_obs=np.array([1.0, 2.0, 3.0]), noise=W.NOISE_ADDITIVE,
                sigma=[jump, jump], prior_lo=[0.02, 2.0 ** -39, 2.0 ** -39], prior_hi=[0.08, 2.0 ** -38, 2.0 ** -38],
                x0=np.array([2.0 ** 9, 1.0, 1.0]))
    y = np.array([[2.0 ** 9, 1.0]] * 3)
    g, o = pf.Filter.from_workload(w), oracle.Filter(w)
    o.init()
    check_epoch(g, o, w.t_obs[0], y[0])
    e = g.pf_get_ensemble()
    h1 = e["h1"].copy()
    h1[:, 0] += jump
    g.pf_set_ensemble(h1=h1)
    check_epoch(g, o, w.t_obs[1], y[1])
    assert np.isfinite(g.pf_get_ensemble()["lw"]).all()
    g.close()
