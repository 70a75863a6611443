"""The increment form (csrc/pf_fast.cuh) component by component: Robertson's y2 and y3 are
1e-5 to 1e-9 of y1, so a bound on the norm says nothing of them.  Particles of the whole
prior, from t = 0 on, few and many substeps an interval, stage 1's form and stage 2's,
against Newton's iterates in extended precision (CPU); and one iteration a substep on
the device against the oracle (GPU)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1411_1702_gb300 import workloads as W
from test_increment_form import _extended

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1411_1702_gb300", "csrc")


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    oracle.build()
    out = str(tmp_path_factory.mktemp("intervalshim") / "libinterval_shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-fPIC",
                    "-shared", "-I", CSRC, os.path.join(ROOT, "tests", "interval_shim.cpp"), "-o", out], check=True)
    L = C.CDLL(out)
    L.shim_run.argtypes = [C.c_int] * 3 + [C.c_void_p] * 2 + [C.c_int] * 2 + [C.c_void_p] * 2
    return L


def _rows(rows, w):
    adams = rows[0]["kind"] > 10
    return np.array([[r["kind"], r["gamma"], *((r["beta"][1], r["beta"][2], 0.0, *r["bab"][:3], 0.0) if adams
                     else (r["rho1"], r["rho2"], r["rho3"], r["pi0"], r["pi1"], r["pi2"], r["pi3"])),
                     r["mu"], oracle.mm_input(r["t"]) if w.ode == W.MICHAELIS else 0.0] for r in rows])


@pytest.mark.parametrize("S,K,intervals", [(50, 2, 3), (10, 2, 5), (5, 2, 8), (2, 2, 8), (5, 3, 5), (2, 4, 5)])
@pytest.mark.parametrize("err", [0, 1])
def test_robertson_components(shim, S, K, intervals, err):
    """A component is off by at most, a substep, its own rounding and 2^-46 (the pairs of
    floats) of an increment no larger than itself.  (The cold start's FP64 steps are the
    oracle's on both sides.)"""
    if np.finfo(np.longdouble).eps > 2.0 ** -62:
        pytest.skip("no extended precision on this machine")
    w = W.robertson(T=40)
    w = w.with_(substeps=S, q0=10.0 ** (8.0 / (39.0 * S)))
    cfg, rng = oracle.make_config(w), np.random.default_rng(77)
    taken = total = 0
    for _ in range(12):
        th = np.exp(rng.uniform(np.log(w.prior_lo), np.log(w.prior_hi)))
        x = h1 = h2 = np.array(w.x0)
        t, depth, hp1, hp2 = 0.0, 0, 0.0, 0.0
        for k in range(intervals):
            tab, _, dout = oracle.build_substeps(cfg, t, w.t_obs[k], depth, hp1, hp2)
            rows = oracle.substep_dicts(tab, S)
            cold = sum(r["kind"] == 1 for r in rows)
            head = oracle.propagate(w.ode, K, th, tab, cold, x, h1, h2) if cold else (x, h1, h2)
            ref = _extended("robertson", th, rows, K, x, h1, h2)
            if cold < S:
                mid = _extended("robertson", th, rows[cold:], K, *head[:3])
                s, E = np.concatenate([*head[:3], np.zeros(9)]), np.zeros(3)
                tht, tbl = np.ascontiguousarray(th), _rows(rows[cold:], w)
                n = shim.shim_run(0, 0, err, tht.ctypes.data, tbl.ctypes.data, S - cold, K, s.ctypes.data, E.ctypes.data)
                total, taken = total + 1, taken + (n == S - cold)
                if n == S - cold:
                    tol = S * (2.0 ** -53 + 2.0 ** -46)
                    for i in range(3):
                        assert np.all(np.abs(s[3 * i:3 * i + 3] - mid[i]) <= tol * np.abs(mid[i]))
            x, h1, h2 = (np.asarray(v, dtype=np.float64) for v in ref[:3])
            t, depth, hp2, hp1 = w.t_obs[k], dout, (rows[-2]["h"] if S > 1 else hp1), rows[-1]["h"]
    # most intervals are the increment form's, none is left out for being stiff
    assert taken >= 0.9 * total


@pytest.mark.parametrize("lmm", [W.LMM_BDF2, W.LMM_AM1, W.LMM_AM3])
def test_michaelis_components(shim, lmm):
    """Intervals after the first over the prior: a component is rounded once a substep (half
    an ulp, 2^-53 of it at most), at random, so over the particles its error's root mean
    square is at most sqrt(S) 2^-53, twice that allowed for the values converted on the way."""
    if np.finfo(np.longdouble).eps > 2.0 ** -62:
        pytest.skip("no extended precision on this machine")
    w = W.michaelis(T=6, lmm=lmm)
    cfg, rng = oracle.make_config(w), np.random.default_rng(78)
    errs = []
    for _ in range(40):
        th = np.ascontiguousarray(np.exp(rng.uniform(np.log(w.prior_lo), np.log(w.prior_hi))))
        x = h1 = h2 = np.array(w.x0)
        t, depth, hp1, hp2 = 0.0, 0, 0.0, 0.0
        for k in range(4):
            tab, S, dout = oracle.build_substeps(cfg, t, w.t_obs[k], depth, hp1, hp2)
            rows = oracle.substep_dicts(tab, S)
            ref = _extended("michaelis", th, rows, 4, x, h1, h2)
            if k > 0:
                h = rows[0]["h"]
                f = [oracle.ode_f(w.ode, th, v, rows[0]["tn"] - j * h) for j, v in enumerate((x, h1, h2))]
                s, E, tbl = np.concatenate([x, h1, h2, *f]), np.zeros(3), _rows(rows, w)
                n = shim.shim_run(1, 2 if lmm > 10 else 0, 1, th.ctypes.data, tbl.ctypes.data, S, 4, s.ctypes.data, E.ctypes.data)
                if n == S:
                    errs.append(np.asarray((s[:3] - ref[0]) / np.abs(ref[0]), dtype=float))
            x, h1, h2 = (np.asarray(v, dtype=np.float64) for v in ref[:3])
            t, depth, hp2, hp1 = w.t_obs[k], dout, rows[-2]["h"], rows[-1]["h"]
    assert len(errs) >= 100
    assert np.all(np.sqrt(np.mean(np.square(errs), axis=0)) <= 2 * np.sqrt(S) * 2.0 ** -53)


@pytest.mark.gpu
@pytest.mark.parametrize("problem,lmm", [("robertson", W.LMM_BDF2), ("michaelis", W.LMM_BDF2), ("michaelis", W.LMM_AM3)])
def test_single_iteration_on_the_device(problem, lmm):
    """K = 1: the first Newton iterate from the predictor, component by component: the device's
    pivots are reciprocals to 2^-40, a substep, of a correction no larger than the component."""
    from paper_1411_1702_gb300 import build as B
    B.build()
    oracle.build()
    from paper_1411_1702_gb300 import pf
    if problem == "robertson":
        w = W.robertson(N=200, T=4)
        w = w.with_(substeps=10, q0=10.0 ** (8.0 / 390.0), noise=W.NOISE_ADDITIVE, sigma=[0.3, 0.3])
    else:
        w = W.michaelis(N=200, T=4, lmm=lmm)
        w = w.with_(noise=W.NOISE_ADDITIVE, sigma=[3.0] * 3, prior_lo=list(0.6 * w.theta_true), prior_hi=list(1.6 * w.theta_true))
    w = w.with_(newton_iters=1, kappa=1e-60)
    g, o = pf.Filter.from_workload(w), oracle.Filter(w)
    o.init()
    from parity_util import begin_epoch
    for k in range(4):
        begin_epoch(g, o)
        g.pf_assimilate(w.t_obs[k], w.y_obs[k])
        tab, S = o.substeps(w.t_obs[k])
        assert o.stage1(tab, S, w.y_obs[k]) == oracle.OK
        ll = o.work()["ll1"]
        assert np.all(np.abs(g.pf_get_work()["ll1"] - ll) <= 1e-9 * (1 + np.abs(ll)))
        assert o.cumulative() == oracle.OK
        assert o.stage2(tab, S, w.y_obs[k], g.pf_get_work()["idx"]) == oracle.OK
        assert o.commit(w.t_obs[k]) == oracle.OK
        a, b = g.pf_get_ensemble(), o.state()
        for key in ("x", "h1"):
            assert np.all(np.abs(a[key] - b[key]) <= S * 2.0 ** -40 * np.abs(b[key])), (k, key)
    g.close()
