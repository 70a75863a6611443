"""The increment form of the implicit substeps (csrc/pf_fast.cuh): a host build
against Newton solves in extended precision over whole intervals (CPU), and the
filters on the device where the form hands substeps back to FP64 (GPU)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1411_1702_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1411_1702_gb300", "csrc")


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    oracle.build()
    out = str(tmp_path_factory.mktemp("fastshim") / "libfast_shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-fPIC",
                    "-shared", "-I", CSRC, os.path.join(ROOT, "tests", "fast_shim.cpp"), "-o", out], check=True)
    L = C.CDLL(out)
    L.shim_interval.argtypes = [C.c_int] * 2 + [C.c_void_p] * 2 + [C.c_int] * 2 + [C.c_void_p] * 2
    L.shim_pairs.argtypes = [C.c_void_p] * 3 + [C.c_long]
    return L


def test_double_to_pair_and_back(shim):
    """A double's pair holds it to 2^-47, the leading float goes back exactly,
    zeros and signs included; values under the floats' range give 0."""
    rng = np.random.default_rng(1)
    a = rng.standard_normal(4000) * 2.0 ** rng.uniform(-70, 90, 4000)
    a = np.concatenate([a, [0.0, 1.0, -1.0, 2.0, 1 - 2 ** -53, -(2 - 2 ** -52), 2.0 ** -126, 2.0 ** 100]])
    hl, back = np.empty((len(a), 2)), np.empty(len(a))
    shim.shim_pairs(a.ctypes.data, hl.ctypes.data, back.ctypes.data, len(a))
    assert np.all(np.abs(hl.sum(1) - a) <= 2.0 ** -47 * np.abs(a))
    assert np.array_equal(back, hl[:, 0]) and np.array_equal(hl[:, 0], hl[:, 0].astype(np.float32))
    tiny = np.array([2.0 ** -127, -2.0 ** -300, 5e-324])
    hl, back = np.empty((3, 2)), np.empty(3)
    shim.shim_pairs(tiny.ctypes.data, hl.ctypes.data, back.ctypes.data, 3)
    assert np.all(hl == 0.0) and np.all(back == 0.0)


LD = np.longdouble


def _rhs(problem, th, u, x):
    if problem == "robertson":
        a, b, c = th[0] * x[0], th[2] * x[1] * x[2], th[1] * x[1] * x[1]
        q, p, s = th[2] * x[1], th[2] * x[2], 2 * th[1] * x[1]
        return np.array([b - a, a - b - c, c]), np.array([[-th[0], p, q], [th[0], -p - s, -q], [0, s, 0]], dtype=LD)
    s1, s2 = x[0] + th[2], x[1] + th[3]
    j1, j2, a, b = th[0] * x[0] / s1, th[1] * x[1] / s2, th[0] * th[2] / s1 ** 2, th[1] * th[3] / s2 ** 2
    half = LD(0.5)
    return (np.array([u - j1, j1 - j2, j2 - half * (x[2] - 2)]), np.array([[-a, 0, 0], [a, -b, 0], [0, b, -half]], dtype=LD))


def _extended(problem, th, rows, K, x, h1, h2):
    """The interval in extended precision: the FP64 table's weights, K full Newton steps."""
    th = [LD(v) for v in th]
    x, h1, h2, E = (np.array(v, dtype=LD) for v in (x, h1, h2, np.zeros(3)))
    u = (lambda t: oracle.mm_input(t)) if problem == "michaelis" else (lambda t: 0.0)
    f = lambda t, v: _rhs(problem, th, LD(u(t)), v)[0]  # noqa: E731
    F = []
    if rows[0]["kind"] > 10:
        h = rows[0]["h"]
        F = [f(rows[0]["tn"] - j * h, (x, h1, h2)[j]) for j in range(rows[0]["kind"] % 10)]
    for r in rows:
        if r["kind"] > 10:
            xp = x + sum(LD(r["bab"][j]) * F[j] for j in range(r["kind"] % 10))
            rr = x + sum(LD(r["beta"][j]) * F[j - 1] for j in range(1, r["kind"] % 10))
        elif r["kind"] == 1:
            xp, rr = x + LD(r["h"]) * f(r["tn"], x), x
        else:
            xp = LD(r["pi0"]) * x + LD(r["pi1"]) * h1 + LD(r["pi2"]) * h2
            rr = LD(r["rho1"]) * x + LD(r["rho2"]) * h1
            if r["kind"] == 3:
                xp, rr = xp + LD(r["pi3"]) * f(r["tn"], x), rr + LD(r["rho3"]) * h2
        y = np.array(x if r["kind"] == 1 else xp)
        for _ in range(K):
            fy, J = _rhs(problem, th, LD(u(r["t"])), y)
            A, b = np.eye(3, dtype=LD) - LD(r["gamma"]) * J, rr - y + LD(r["gamma"]) * fy
            for i in range(3):
                for k in range(i + 1, 3):
                    m = A[k, i] / A[i, i]
                    A[k], b[k] = A[k] - m * A[i], b[k] - m * b[i]
            for i in (2, 1, 0):
                b[i] = (b[i] - A[i, i + 1:] @ b[i + 1:]) / A[i, i]
            y = y + b
        E = E + (LD(r["mu"]) * (y - xp)) ** 2
        if r["kind"] > 10:
            F = [f(r["t"], y)] + F[:2]
        x, h1, h2 = y, x, h1
    return x, h1, h2, E


@pytest.mark.parametrize("problem,lmm,K", [("robertson", W.LMM_BDF2, 2), ("robertson", W.LMM_BDF2, 1),
                                           ("robertson", W.LMM_BDF3, 3), ("robertson", W.LMM_AM3, 2),
                                           ("michaelis", W.LMM_BDF2, 4), ("michaelis", W.LMM_BDF3, 4),
                                           ("michaelis", W.LMM_AM1, 4), ("michaelis", W.LMM_AM2, 3),
                                           ("michaelis", W.LMM_AM3, 4)])
def test_interval_against_extended(shim, problem, lmm, K):
    """Particles around the true parameter over eight intervals: each interval
    from the same state in extended precision and in increments.  16 roundings of
    the state's size a substep (FP64 steps of the plain form round 8 times)."""
    if np.finfo(LD).eps > 2.0 ** -62:
        pytest.skip("no extended precision on this machine")
    w = W.michaelis(T=8, lmm=lmm) if problem == "michaelis" else W.robertson(T=40)
    t_obs = w.t_obs[:8]
    if problem == "robertson":
        t_obs = w.t_obs[20:28]
        if lmm != W.LMM_BDF2:
            t_obs = t_obs[0] + 1e-2 * np.arange(8)
            w = w.with_(lmm=lmm, spacing=W.SPACING_UNIFORM, dt=1e-3)
    cfg = oracle.make_config(w)
    rng = np.random.default_rng(5)
    fam = 2 if lmm > 10 else 1 if lmm == W.LMM_BDF3 else 0
    for _ in range(12):
        th = w.theta_true * np.exp(rng.uniform(-0.3, 0.3, w.p))
        x = np.array(w.x0 if problem == "michaelis" else [0.98, 3.5e-5 * th[0] / 0.04, 0.02], dtype=float)
        h1, h2, depth, hp1, hp2, t = x.copy(), x.copy(), 0, 0.0, 0.0, 0.0 if problem == "michaelis" else t_obs[0] * 0.7
        if problem == "robertson" and lmm != W.LMM_BDF2:
            t = t_obs[0] - 1e-2
        for t1 in t_obs:
            tab, S, dout = oracle.build_substeps(cfg, t, t1, depth, hp1, hp2)
            rows = oracle.substep_dicts(tab, S)
            cold = 0 if fam == 2 else sum(r["kind"] == 1 for r in rows)
            ref = _extended(problem, th, rows, K, x, h1, h2)
            # the increment form starts after a cold start's BDF1 steps
            head = oracle.propagate(w.ode, K, th, tab, cold, x, h1, h2, with_error=True) if cold else (x, h1, h2, np.zeros(3))
            s = np.concatenate(head[:3])
            q0 = rows[0]["kind"] % 10 if fam == 2 else 0
            f = [oracle.ode_f(w.ode, th, head[0], rows[cold]["tn"] if cold < S else 0.0)]
            if fam == 2:
                h = rows[0]["h"]
                f.append(oracle.ode_f(w.ode, th, h1, rows[0]["tn"] - h) if q0 >= 2 else f[0])
                f.append(oracle.ode_f(w.ode, th, h2, rows[0]["tn"] - 2 * h) if q0 >= 3 else f[1])
            else:
                f += [f[0], f[0]]
            s = np.concatenate([s] + f)
            tbl = np.array([[r["kind"], r["gamma"], *((r["beta"][1], r["beta"][2], 0.0, *r["bab"][:3], 0.0) if fam == 2
                             else (r["rho1"], r["rho2"], r["rho3"], r["pi0"], r["pi1"], r["pi2"], r["pi3"])),
                             r["mu"], oracle.mm_input(r["t"]) if problem == "michaelis" else 0.0] for r in rows[cold:]])
            E, tht = np.zeros(3), np.ascontiguousarray(th)
            n = shim.shim_interval(0 if problem == "robertson" else 1, fam, tht.ctypes.data, tbl.ctypes.data, S - cold, K,
                                   s.ctypes.data, E.ctypes.data)
            assert n == S - cold
            tol = 16 * S * 2.0 ** -53 * np.max(np.abs(ref[0]))
            for i in range(3):
                assert np.max(np.abs(s[3 * i:3 * i + 3] - ref[i])) <= tol
            assert np.max(np.abs(np.sqrt(E + head[3]) - np.sqrt(ref[3]))) <= tol
            x, h1, h2 = (np.asarray(v, dtype=np.float64) for v in ref[:3])
            t, depth, hp2, hp1 = t1, dout, rows[-2]["h"], rows[-1]["h"]


@pytest.mark.parametrize("lmm,K", [(W.LMM_BDF2, 4), (W.LMM_BDF2, 2), (W.LMM_BDF3, 4), (W.LMM_AM3, 4)])
def test_unconverged_iterations_are_refused(shim, lmm, K):
    """M1's first interval over the whole prior, where some particles' Newton iterations
    have not settled after K: the increment form stops before a substep whose K-th
    iterate it would not give.  The tolerance is test_interval_against_extended's."""
    if np.finfo(LD).eps > 2.0 ** -62:
        pytest.skip("no extended precision on this machine")
    w = W.michaelis(T=1, lmm=lmm)
    cfg, rng = oracle.make_config(w), np.random.default_rng(9)
    fam = 2 if lmm > 10 else 1 if lmm == W.LMM_BDF3 else 0
    tab, S, _ = oracle.build_substeps(cfg, 0.0, w.t_obs[0], 0, 0.0, 0.0)
    rows = oracle.substep_dicts(tab, S)
    cold = 0 if fam == 2 else sum(r["kind"] == 1 for r in rows)
    done = 0
    for _ in range(60):
        th = np.exp(rng.uniform(np.log(w.prior_lo), np.log(w.prior_hi)))
        x = np.array(w.x0, dtype=float)
        head = oracle.propagate(w.ode, K, th, tab, cold, x, x, x, with_error=True) if cold else (x, x, x, np.zeros(3))
        f = [oracle.ode_f(w.ode, th, head[0], rows[cold]["tn"])] * 3
        s, E, tht = np.concatenate([*head[:3], *f]), np.zeros(3), np.ascontiguousarray(th)
        tbl = np.array([[r["kind"], r["gamma"], *((r["beta"][1], r["beta"][2], 0.0, *r["bab"][:3], 0.0) if fam == 2
                         else (r["rho1"], r["rho2"], r["rho3"], r["pi0"], r["pi1"], r["pi2"], r["pi3"])),
                         r["mu"], oracle.mm_input(r["t"])] for r in rows[cold:]])
        n = shim.shim_interval(1, fam, tht.ctypes.data, tbl.ctypes.data, S - cold, K, s.ctypes.data, E.ctypes.data)
        if n == 0:
            continue
        ref = _extended("michaelis", th, rows[:cold + n], K, x, x, x)
        tol = 16 * S * 2.0 ** -53 * np.max(np.abs(ref[0]))
        for i in range(3):
            assert np.max(np.abs(s[3 * i:3 * i + 3] - ref[i])) <= tol
        done += n
    # most of the substeps do settle (at K = 2 fewer)
    assert done >= (30 if K == 4 else 5) * (S - cold)


@pytest.mark.gpu
@pytest.mark.parametrize("lmm", [W.LMM_BDF2, W.LMM_BDF3, W.LMM_AM2])
@pytest.mark.parametrize("N,K,scale", [(33, 1, 1.0), (129, 3, 1.0), (65, 2, 2.0 ** 30)])
def test_device_epochs(lmm, N, K, scale):
    """Ragged ensembles, one and three Newton iterations, and the same problem with
    time in units of 2^-30, whose rate constants are beyond the floats' range and
    take the FP64 path."""
    from paper_1411_1702_gb300 import build as B
    B.build()
    from paper_1411_1702_gb300 import pf
    from parity_util import check_epoch
    w = W.robertson(N=N, T=3)
    star = np.array([0.04, 3e7, 1e4]) * scale
    w = w.with_(lmm=lmm, newton_iters=K, spacing=W.SPACING_UNIFORM, dt=2e-6 / scale, prior_lo=list(star / 2), prior_hi=list(star * 2),
                t_obs=np.array([1e-4, 2e-4, 3e-4]) / scale, y_obs=w.y_obs[:3], x_true=w.x_true[:3],
                noise=W.NOISE_ADDITIVE, sigma=[0.01, 0.01])
    g, o = pf.Filter.from_workload(w), oracle.Filter(w)
    o.init()
    for k in range(3):
        check_epoch(g, o, w.t_obs[k], w.y_obs[k], exempt_dead=True)
