"""The Brusselator's substeps (csrc/pf_bruss.cu) where their form changes: blocks
of eight particles and their remainders, each number of Newton iterations, steps
so long that the last correction is solved for twice or a substep falls back to
FP64, and a problem whose constants take the FP64 path throughout; against the
CPU oracle within the repository's bounds."""
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
    _pf.load()
    return _pf


@pytest.mark.parametrize("N,K,S,scale", [(1, 3, 20, 1.0), (7, 1, 20, 1.0), (8, 2, 20, 1.0), (9, 3, 3, 1.0),
                                         (17, 2, 1, 1.0), (33, 4, 2, 1.0), (23, 2, 5, 2.0 ** 62)])
def test_epochs(pf, N, K, S, scale):
    """scale: the diffusion in time units of 1/scale, where the reaction vanishes."""
    w = W.brusselator(N=N, T=3)
    hi, lo = list(w.prior_hi), list(w.prior_lo)
    hi[2], lo[2] = hi[2] * scale, lo[2] * scale
    t = w.t_obs / scale
    w = w.with_(newton_iters=K, substeps=S, dt=1.0 / (3.0 * S * scale), prior_lo=lo, prior_hi=hi, t_obs=t)
    g, o = pf.Filter.from_workload(w), oracle.Filter(w)
    o.init()
    for k in range(3):
        check_epoch(g, o, w.t_obs[k], w.y_obs[k], exempt_dead=True)
    g.close()
