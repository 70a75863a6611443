"""pf_get_ensemble's reordering on the device: what pf_set_ensemble put in comes
back bit for bit, at the edges of the kernel's tiles and row lengths."""
import numpy as np
import pytest

from paper_1411_1702_gb300 import build as B
from paper_1411_1702_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,kw,N", [("linear2", {}, 1), ("robertson", {}, 33), ("michaelis", {}, 1025),
                                       ("brusselator", {}, 65), ("advdiff", {"n": 4}, 31), ("advdiff", {"n": 20}, 257)])
def test_set_then_get(name, kw, N):
    B.build()
    from paper_1411_1702_gb300 import pf
    w = (W.advdiff(N=N, T=2, **kw) if name == "advdiff" else W.get(name, N=N, T=2))
    f = pf.Filter.from_workload(w, N=N)
    rng = np.random.default_rng(N)
    want = {k: rng.standard_normal((N, w.d)) for k in ("x", "h1", "h2")}
    want["phi"], want["lw"] = rng.standard_normal((N, w.p)), rng.standard_normal(N)
    f.pf_set_ensemble(**want)
    got = f.pf_get_ensemble()
    for k in want:
        assert np.array_equal(got[k], want[k]), k
    again = f.pf_get_ensemble()
    assert all(np.array_equal(again[k], want[k]) for k in want)
