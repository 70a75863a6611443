"""The 2D system's kernels over their launch shapes (grid sides from the smallest
to the largest, ragged blocks) and over intervals on which the error estimate
stays in FP64 (two substeps, cold starts) or leaves it: one or two epochs
against the oracle, every stage output."""
import numpy as np
import pytest

import oracle
from paper_1411_1702_gb300 import build as B
from paper_1411_1702_gb300 import workloads as W
from parity_util import check_epoch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N,dt,T", [(4, 7, 0.1, 2), (10, 5, 0.5, 2), (16, 6, 0.05, 2), (22, 3, 0.1, 2), (26, 3, 0.25, 1),
                                      (42, 2, 0.5, 1), (44, 2, 0.5, 1), (46, 2, 0.5, 1)])
def test_epochs_by_grid_side(n, N, dt, T):
    B.build()
    oracle.build()
    from paper_1411_1702_gb300 import pf
    w = W.advdiff(n, N, T)
    w = w.with_(dt=dt, sigma=[30.0 * s for s in w.sigma])
    g, o = pf.Filter.from_workload(w, N=N), oracle.Filter(w, N=N)
    o.init()
    for k in range(T):
        check_epoch(g, o, w.t_obs[k], w.y_obs[k])


@pytest.mark.parametrize("history", [W.HIST_CARRY, W.HIST_RESTART])
def test_geometric_grid(history):
    """Substeps whose gammas all differ (each its own reference), carried and cold."""
    B.build()
    oracle.build()
    from paper_1411_1702_gb300 import pf
    w = W.advdiff(12, 9, 3)
    w = w.with_(spacing=W.SPACING_GEOMETRIC, substeps=12, q0=1.2, history=history, sigma=[30.0 * s for s in w.sigma])
    g, o = pf.Filter.from_workload(w, N=9), oracle.Filter(w, N=9)
    o.init()
    for k in range(3):
        check_epoch(g, o, w.t_obs[k], w.y_obs[k])


def test_dead_particles_stay_dead():
    """States that are not finite give zero weight, as before the integer transforms."""
    B.build()
    from paper_1411_1702_gb300 import pf
    w = W.advdiff(8, 6, 1)
    w = w.with_(sigma=[30.0 * s for s in w.sigma])
    f = pf.Filter.from_workload(w, N=6)
    e = f.pf_get_ensemble()
    e["x"][2, 5] = np.nan
    e["x"][3, 0] = np.inf
    f.pf_set_ensemble(x=e["x"])
    f.pf_assimilate(w.t_obs[0], w.y_obs[0])
    lg = f.pf_get_work()["lg"]
    assert np.isneginf(lg[[2, 3]]).all() and np.isfinite(lg[[0, 1, 4, 5]]).all()
    assert np.isfinite(f.pf_get_ensemble()["x"]).all()
