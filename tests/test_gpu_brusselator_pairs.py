"""Two Brusselator particles share a warp: what one of them is does not change the
other's states by a bit."""
import numpy as np
import pytest

from paper_1411_1702_gb300 import build as B
from paper_1411_1702_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,S", [(1, 20), (2, 20), (3, 5), (3, 20)])
def test_states_do_not_depend_on_the_partner(K, S):
    B.build()
    from paper_1411_1702_gb300 import pf
    # noise so large that every weight is the same and every particle its own parent
    w = W.brusselator(N=8, T=2)
    w = w.with_(newton_iters=K, substeps=S, dt=1.0 / (3.0 * S), sigma=[1e9] * 8)
    x = np.tile(w.x0, (8, 1)) * (1 + 0.01 * np.arange(8))[:, None]
    out = []
    for other in (1.0, 2.5, 40.0, 1e8):
        y = x.copy()
        y[1::2] *= other
        f = pf.Filter.from_workload(w)
        f.pf_set_ensemble(x=y, h1=y, h2=y, phi=np.tile(np.log(w.theta_true), (8, 1)))
        f.pf_set_moments(np.log(w.theta_true), 1e-4 * np.eye(3))
        for k in range(2):
            f.pf_assimilate(w.t_obs[k], w.y_obs[k])
            assert np.array_equal(f.pf_get_work()["idx"][::2], np.arange(8)[::2])
            # (the moments follow all particles: back to the same ones)
            f.pf_set_moments(np.log(w.theta_true), 1e-4 * np.eye(3))
        out.append((f.pf_get_work()["ll1"][::2], *(f.pf_get_ensemble()[key][::2] for key in ("x", "h1", "h2"))))
        f.close()
    assert np.isfinite(out[0][1]).all()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.array_equal(a, b)
