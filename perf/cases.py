"""Performance cases of the LMM PF-SMC library: what its users run.

A filter's user creates it once and then, for every data set, restarts it (pf_reset), assimilates the
observations in order, reads the estimates (theta-bar, C, x-bar) after each, and takes the posterior
ensemble at the end.  That is one pass here, for the problems and integrators of this repository's
workloads, from 2000 particles (a call's latency counts) to a million.  Two cases drive many filters at
once (a batch, a server), one is the stand-alone systematic resampler.

Observations are the workload's reference trajectory with noise drawn from the seed, which is also the
filter's random seed.
"""
import functools
import math

import numpy as np
import torch

from paper_1411_1702_gb300 import pf, workloads as W

# Passes are a few epochs long rather than the whole series where a whole series would take seconds.
CASES = [
    # The smallest filter of the repository: 2000 particles, the whole 50-observation series, one
    # synchronous call per observation.  Latency and launches.
    dict(name="linear2_2000", kind="filter", problem="linear2", lmm="BDF2", N=2000, epochs=50),
    # A ragged small ensemble of the stiff three-state problem, half its series.
    dict(name="robertson_3001", kind="filter", problem="robertson", lmm="BDF2", N=3001, epochs=20),
    # The benchmark's ensemble: Robertson kinetics, 131072 particles, host observations.
    dict(name="robertson_131072", kind="filter", problem="robertson", lmm="BDF2", N=131072, epochs=10),
    # A million particles, the series loaded once and run on the device without host round trips.
    dict(name="robertson_1m_series", kind="series", problem="robertson", lmm="BDF2", N=1 << 20, epochs=3),
    # The paper's first system (three compartments, Tables 1-2) at its larger ensemble: the default
    # integrator, and a third-order Adams-Moulton method.
    dict(name="michaelis_bdf2_50000", kind="filter", problem="michaelis", lmm="BDF2", N=50000, epochs=20),
    dict(name="michaelis_am3_50000", kind="filter", problem="michaelis", lmm="AM3", N=50000, epochs=20),
    # The one-dimensional Brusselator (64 states a particle): block-tridiagonal Newton systems.
    dict(name="brusselator_16384", kind="filter", problem="brusselator", lmm="BDF2", N=16384, epochs=5),
    # The paper's second system (Sec. 4, Table 3) on both of its grids, with sensors noisy enough that
    # the ensemble keeps a posterior (NOISE below).
    dict(name="advdiff20_5000", kind="filter", problem="advdiff20", lmm="BDF2", N=5000, epochs=5),
    dict(name="advdiff40_1000", kind="filter", problem="advdiff40", lmm="BDF2", N=1000, epochs=3),
    # Many independent filters of uneven size and mixed problems advanced together, ten rounds.
    dict(name="batch_24", kind="batch", filters=24, log2_min=10.0, log2_max=14.0, epochs=10),
    # Sessions served through the continuous-batching server: opened, their observations queued,
    # drained, read and closed.
    dict(name="server_6", kind="server", sessions=6, log2_min=11, log2_max=14, epochs=6),
    # Systematic resampling of caller-owned log weights without allocation.
    dict(name="resample_1m", kind="resample", N=1000003),
]

SUBSTEPS = {"linear2": 20, "robertson": 50, "michaelis": 10, "brusselator": 20, "advdiff20": 10, "advdiff40": 10}
# FP64 operations of one particle-substep of the method as stated (full Newton, analytic Jacobian; the
# 2D system solved in its Fourier basis), for work()
FLOPS = {"linear2": 49, "robertson": 192, "michaelis": 364, "brusselator": 7247, "advdiff20": 21600, "advdiff40": 151000}
DIMS = {"linear2": (2, 2), "robertson": (3, 3), "michaelis": (3, 4), "brusselator": (64, 3),
        "advdiff20": (361, 5), "advdiff40": (1521, 5)}
SERIES = {"linear2": 50, "robertson": 40, "michaelis": 50, "brusselator": 30, "advdiff20": 30, "advdiff40": 30}
# particles of the largest ensemble each problem is run with
LARGEST = {"linear2": 1 << 20, "robertson": 1 << 20, "michaelis": 1 << 18, "brusselator": 16384,
           "advdiff20": 5000, "advdiff40": 1000}
# The 2D workload's own sensor noise leaves one particle of 5000 with all the weight after the first
# observation, a singular covariance and nothing that two computations could agree on; 30 times that noise
# leaves tens of particles.
NOISE = {"advdiff20": 30.0, "advdiff40": 30.0}
# The explicit Adams-Bashforth methods are left out: they are unstable on these stiff problems and are in
# the library for the paper's comparison only.
IMPLICIT = ["BDF1", "BDF2", "BDF3", "AM1", "AM2", "AM3"]


def listed():
    return [dict(c) for c in CASES]


def _steps(c):
    return 2 * SUBSTEPS[c["problem"]] * c["N"] * c["epochs"]


def draw(rng):
    """A case of the same ranges: a problem, an integrator it takes, any size up to the largest, odd ones included."""
    what = rng.choice(["filter"] * 7 + ["series"] * 2 + ["batch", "server", "resample"])
    if what == "batch":
        return dict(kind="batch", filters=rng.randint(2, 24), log2_min=10.0, log2_max=rng.choice([11.0, 12.0, 13.0, 14.0]), epochs=rng.randint(3, 10))
    if what == "server":
        return dict(kind="server", sessions=rng.randint(2, 6), log2_min=10, log2_max=rng.randint(11, 14), epochs=rng.randint(3, 6))
    if what == "resample":
        return dict(kind="resample", N=int(2.0 ** rng.uniform(10.0, 20.0)))
    problem = rng.choice(["linear2", "robertson", "robertson", "michaelis", "michaelis", "brusselator", "advdiff20", "advdiff40"])
    lmm = rng.choice(IMPLICIT) if problem == "michaelis" else "BDF2"
    low = 64 if problem.startswith("advdiff") else 1000
    N = int(math.exp(rng.uniform(math.log(low), math.log(LARGEST[problem]))))
    most = max(_steps(c) * FLOPS[c["problem"]] for c in CASES if c.get("problem") == problem)
    # (a small Brusselator epoch is a serial chain that costs what a large one does)
    epochs = min(SERIES[problem], rng.randint(2, 5 if problem == "brusselator" else 20), max(2, most // (2 * SUBSTEPS[problem] * N * FLOPS[problem])))
    return dict(kind=what, problem=problem, lmm=lmm, N=N, epochs=int(epochs))


# ------------------------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _base(problem, lmm):
    """The workload with its reference trajectory (solved once per process: it does not depend on the seed)."""
    if problem == "michaelis":
        return W.michaelis(lmm=W.LMM_NAMES[lmm])
    w = W.get(problem)
    return w.with_(sigma=[s * NOISE.get(problem, 1.0) for s in w.sigma])


def _workload(problem, lmm, N, epochs, seed, stream=0):
    """The problem with `epochs` observations: the reference states plus noise drawn from the seed."""
    b = _base(problem, lmm)
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 0x0B5, stream])
    xs = b.x_true[:epochs][:, b.obs_idx]
    noise = rng.standard_normal(xs.shape) * np.asarray(b.sigma)[None, :]
    y = xs * (1.0 + noise) if b.noise == W.NOISE_RELATIVE else xs + noise
    return b.with_(N=int(N), seed=int(seed) & 0x7FFFFFFF, stream=stream, t_obs=b.t_obs[:epochs], y_obs=np.ascontiguousarray(y),
                   x_true=b.x_true[:epochs])


def _members(case, seed):
    """The workloads of a batch or of a server's sessions: sizes and problems from the case, data from the seed."""
    rng = np.random.default_rng([0x5123, case["epochs"], case.get("filters", case.get("sessions", 0))])
    out = []
    count = case["filters"] if case["kind"] == "batch" else case["sessions"]
    for f in range(count):
        N = int(round(2.0 ** rng.uniform(case["log2_min"], case["log2_max"])))
        problem = ("linear2", "robertson", "michaelis")[int(rng.integers(3))]
        out.append(_workload(problem, "BDF2", N, case["epochs"], seed, stream=f))
    return out


def _log_weights(N, seed):
    """First-stage log weights: Gaussian log likelihoods of three observations, widely spread, with some particles dead."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
    z = torch.randn(3, N, generator=g, device="cuda", dtype=torch.float64) * 3.0
    lw = -0.5 * (z * z).sum(0)
    lw[torch.rand(N, generator=g, device="cuda") < 0.01] = -math.inf
    return lw


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("filter", "series"):
        w = _workload(case["problem"], case["lmm"], case["N"], case["epochs"], seed)
        f = pf.Filter.from_workload(w, filter_id=w.stream)
        if kind == "series":
            f.pf_load_observations(w.t_obs, w.y_obs)
        return dict(kind=kind, w=w, f=f)
    if kind == "batch":
        ws = _members(case, seed)
        fs = [pf.Filter.from_workload(w, filter_id=w.stream) for w in ws]
        return dict(kind=kind, ws=ws, fs=fs, batch=pf.Batch(fs))
    if kind == "server":
        return dict(kind=kind, ws=_members(case, seed), server=pf.Server(budget_bytes=1 << 28))
    lw = _log_weights(case["N"], seed)
    u = float(np.random.default_rng([int(seed) & 0x7FFFFFFF, 7]).random())
    return dict(kind=kind, lw=lw, u=u, c=torch.empty_like(lw), idx=torch.empty(case["N"], dtype=torch.int32, device="cuda"))


# --------------------------------------------------------------------------------------------- pass
def _joined(fs):
    """Estimates and ensembles of several filters, one array per quantity."""
    est = [f.pf_estimates() for f in fs]
    ens = [f.pf_get_ensemble() for f in fs]
    out = {k: np.concatenate([e[i].ravel() for e in est]) for i, k in enumerate(("theta", "C", "xbar"))}
    return out | {k: np.concatenate([e[k].ravel() for e in ens]) for k in ("x", "h1", "h2", "phi", "lw")}


def run(state):
    kind = state["kind"]
    if kind == "filter":
        w, f = state["w"], state["f"]
        f.pf_reset()
        est = []
        for t, y in zip(w.t_obs, w.y_obs):
            f.pf_assimilate(t, y)
            est.append(f.pf_estimates())
        out = {k: np.stack([e[i] for e in est]) for i, k in enumerate(("theta", "C", "xbar"))}
        return out | f.pf_get_ensemble()
    if kind == "series":
        w, f = state["w"], state["f"]
        f.pf_reset()
        f.pf_run(0, w.T)
        f.pf_synchronize()
        theta, C, xbar = f.pf_estimates()
        return dict(theta=theta, C=C, xbar=xbar) | f.pf_get_ensemble()
    if kind == "batch":
        for f in state["fs"]:
            f.pf_reset()
        for k in range(len(state["ws"][0].t_obs)):
            status = state["batch"].pf_batch_assimilate([w.t_obs[k] for w in state["ws"]], [w.y_obs[k] for w in state["ws"]])
        return _joined(state["fs"]) | dict(status=np.array(status))
    if kind == "server":
        server = state["server"]
        ids = [server.pf_server_open(w, filter_id=w.stream) for w in state["ws"]]
        for s, w in zip(ids, state["ws"]):
            for t, y in zip(w.t_obs, w.y_obs):
                server.pf_server_submit(s, t, y)
        server.pf_server_drain()
        out = _joined([server.pf_server_session(s)[0] for s in ids])
        for s in ids:
            server.pf_server_close(s)
        server.pf_server_step()
        return out
    lw, stream = state["lw"], torch.cuda.current_stream().cuda_stream
    pf.pf_resample_systematic_noalloc(lw.data_ptr(), lw.numel(), state["u"], state["c"].data_ptr(), state["idx"].data_ptr(), stream)
    return dict(c=state["c"], idx=state["idx"])


def work(case):
    """Bytes: the ensemble read and written once an epoch; operations: the method's, two propagations an epoch."""
    if case["kind"] == "resample":
        return dict(bytes=20.0 * case["N"], flops=0.0)
    if case["kind"] in ("batch", "server"):
        parts = [dict(problem={2: "linear2", 3: "robertson", 4: "michaelis"}[w.p], N=w.N, epochs=case["epochs"]) for w in _members(case, 0)]
    else:
        parts = [case]
    total = dict(bytes=0.0, flops=0.0)
    for c in parts:
        d, p = DIMS[c["problem"]]
        total["bytes"] += 16.0 * c["N"] * (3 * d + p + 1) * c["epochs"]
        total["flops"] += float(_steps(c)) * FLOPS[c["problem"]]
    return total


# -------------------------------------------------------------------- the same, in plain 64-bit torch
# Algorithm 1 restated without the library: dense Newton, cumulative sums, binary search.  Particles of
# several filters on the same problem and time grid are propagated together.
F64 = torch.float64


def _philox(c0, c1, c2, c3, seed):
    def mul(m, x):  # high and low words of a 32 x 32 bit product, in int64 without overflow
        p0, p1 = (m & 0xFFFF) * x, (m >> 16) * x
        mid = p1 + (p0 >> 16)
        return mid >> 16, ((mid & 0xFFFF) << 16) | (p0 & 0xFFFF)

    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    c = [c0, torch.full_like(c0, c1), torch.full_like(c0, c2), torch.full_like(c0, c3)]
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _bits53(n, seed, stream, purpose, epoch, count):
    """The first `count` 53-bit integers of each particle's stream."""
    out = []
    for b in range((count + 1) // 2):
        w = _philox(n, epoch, purpose | (b << 8), stream, seed)
        out += [((w[0] >> 5) << 26) | (w[1] >> 6), ((w[2] >> 5) << 26) | (w[3] >> 6)]
    return out


def _uniforms(*a):
    return [k.to(F64) * 2.0 ** -53 for k in _bits53(*a)[: a[-1]]]


def _normals(n, seed, stream, purpose, epoch, count):
    k, out = _bits53(n, seed, stream, purpose, epoch, 2 * ((count + 1) // 2)), []
    for b in range(0, len(k), 2):
        r = torch.sqrt(-2.0 * torch.log(((1 << 53) - k[b]).to(F64) * 2.0 ** -53))
        a = k[b + 1].to(F64) * (2.0 ** -52 * math.pi)
        out += [r * torch.cos(a), r * torch.sin(a)]
    return out[:count]


def _table(w, t_prev, t_next, hist):
    """Substeps of (t_prev, t_next]: (kind, h, t0, t1, h1, h2); hist = (depth, last two steps)."""
    depth, h1, h2 = hist
    if w.spacing == W.SPACING_UNIFORM:
        S = int(round((t_next - t_prev) / w.dt))
        t = [t_prev + i * ((t_next - t_prev) / S) for i in range(S)] + [t_next]
    else:
        S = w.substeps
        if t_prev > 0.0:
            q = (t_next / t_prev) ** (1.0 / S)
            t = [t_prev * q ** i for i in range(S)] + [t_next]
        else:
            t = [t_next * (w.q0 ** i - 1.0) / (w.q0 ** S - 1.0) for i in range(S)] + [t_next]
    rows, adams = [], w.lmm // 10 == 1
    if w.lmm == W.LMM_BDF1:
        depth = 0
    for i in range(S):
        h = t[i + 1] - t[i]
        if depth >= 1 and h / h1 >= 2.0:
            depth = 0
        if adams:
            kind = 10 + min(w.lmm % 10, depth + 1)
        else:
            kind = w.lmm if depth >= 2 and w.lmm in (W.LMM_BDF2, W.LMM_BDF3) else 1
        rows.append((kind, h, t[i], t[i + 1], h1, h2))
        h1, h2 = h, h1
        depth = min(2, depth + 1)
    return rows, (0 if w.lmm == W.LMM_BDF1 else depth, h1, h2)


def _rhs(ode, th, t, x):
    """f and the nonzero entries of its Jacobian, {(i, j): value}, of the small problems (x: list of components)."""
    if ode == W.LINEAR2:
        return [th[1] * x[1] - th[0] * x[0], -th[1] * x[1]], {(0, 0): -th[0], (0, 1): th[1], (1, 1): -th[1]}
    if ode == W.ROBERTSON:
        a, b, c = th[0] * x[0], th[2] * x[1] * x[2], th[1] * x[1] * x[1]
        q, p, s = th[2] * x[1], th[2] * x[2], 2.0 * th[1] * x[1]
        return [b - a, a - b - c, c], {(0, 0): -th[0], (0, 1): p, (0, 2): q, (1, 0): th[0], (1, 1): -p - s, (1, 2): -q, (2, 1): s}
    v1, v2, k1, k2 = th
    s1, s2 = x[0] + k1, x[1] + k2
    j1, j2, a, b = v1 * x[0] / s1, v2 * x[1] / s2, v1 * k1 / (s1 * s1), v2 * k2 / (s2 * s2)
    lam, c0 = W.MM_KNOWN["lam"], W.MM_KNOWN["c0"]
    return ([W.mm_input(t) - j1, j1 - j2, j2 - lam * (x[2] - c0)],
            {(0, 0): -a, (1, 0): a, (1, 1): -b, (2, 1): b, (2, 2): torch.full_like(a, -lam)})


def _newton(ode, th, t, g, r, y, K):
    """K Newton steps on y - r - g f(y) = 0 by Gaussian elimination."""
    d = len(y)
    for _ in range(K):
        f, J = _rhs(ode, th, t, y)
        A = [[(1.0 if i == j else 0.0) - g * J[i, j] if (i, j) in J else (1.0 if i == j else 0.0) for j in range(d)] for i in range(d)]
        b = [r[i] - y[i] + g * f[i] for i in range(d)]
        for i in range(d):
            for k in range(i + 1, d):
                if isinstance(A[k][i], float) and A[k][i] == 0.0:
                    continue
                m = A[k][i] / A[i][i]
                A[k] = [A[k][j] - m * A[i][j] if j > i else A[k][j] for j in range(d)]
                b[k] = b[k] - m * b[i]
        for i in reversed(range(d)):
            for j in range(i + 1, d):
                b[i] = b[i] - A[i][j] * b[j]
            b[i] = b[i] / A[i][i]
        y = [y[i] + b[i] for i in range(d)]
    return y


def _newton_brusselator(th, t, g, r, y, K):
    """The same for the Brusselator, y = (64, n): block elimination over its 2 x 2 blocks."""
    A, B, D = th[0], th[1], th[2] * 33.0 ** 2
    for _ in range(K):
        u, v = y[0::2], y[1::2]
        pad = lambda z, e: torch.cat([torch.full_like(z[:1], e), z, torch.full_like(z[:1], e)])  # noqa: E731
        up, vp = pad(u, 1.0), pad(v, 3.0)
        uuv = u * u * v
        Gu = r[0::2] - u + g * (A + uuv - (B + 1.0) * u + D * (up[:-2] - 2.0 * u + up[2:]))
        Gv = r[1::2] - v + g * (B * u - uuv + D * (vp[:-2] - 2.0 * v + vp[2:]))
        a, b = 1.0 - g * (2.0 * u * v - (B + 1.0) - 2.0 * D), -g * u * u
        c, e = -g * (B - 2.0 * u * v), 1.0 + g * (u * u + 2.0 * D)
        gD, Wi, z = g * D, [], []
        for i in range(len(u)):
            p, q, s, o, x0, x1 = a[i], b[i], c[i], e[i], Gu[i], Gv[i]
            if i:
                M = Wi[-1]
                p, q, s, o = p - gD * gD * M[0], q - gD * gD * M[1], s - gD * gD * M[2], o - gD * gD * M[3]
                x0, x1 = x0 + gD * z[-1][0], x1 + gD * z[-1][1]
            det = p * o - q * s
            Wi.append((o / det, -q / det, -s / det, p / det))
            z.append((Wi[-1][0] * x0 + Wi[-1][1] * x1, Wi[-1][2] * x0 + Wi[-1][3] * x1))
        d, du, dv = [None] * len(z), 0.0, 0.0
        for i in reversed(range(len(z))):
            M = Wi[i]
            du, dv = z[i][0] + gD * (M[0] * du + M[1] * dv), z[i][1] + gD * (M[2] * du + M[3] * dv)
            d[i] = torch.stack([du, dv])
        y = y + torch.cat(d)
    return y


def _bdf2(h, h1, h2):
    w = h / h1
    den = 1.0 + 2.0 * w
    a, b, c = h, h + h1, h + h1 + h2
    ec, ep = -a ** 3 * (1.0 + w) ** 2 / (6.0 * w * den), a * b * c / 6.0
    return (h * (1.0 + w) / den, (1.0 + w) ** 2 / den, -w * w / den, b * c / (h1 * (h1 + h2)), -a * c / (h1 * h2),
            a * b / ((h1 + h2) * h2), ec / (ep - ec))


AB = {1: (1.0,), 2: (1.5, -0.5), 3: (23 / 12, -16 / 12, 5 / 12)}
AM = {1: (1.0,), 2: (0.5, 0.5), 3: (5 / 12, 8 / 12, -1 / 12)}
AB_ERR, AM_ERR = {1: 1 / 2, 2: 5 / 12, 3: 3 / 8}, {1: -1 / 2, 2: -1 / 12, 3: -1 / 24}


def _propagate(w, th, rows, X):
    """x_n, x_{n-1}, x_{n-2} (each (d, n)) over the substeps, and the sums of squared Milne estimates."""
    if w.ode == W.ADVDIFF:
        return _propagate_spectral(w, th, rows, X)
    x, h1, h2 = X
    E = torch.zeros_like(x)
    rhs = lambda t, z: torch.stack(_rhs(w.ode, th, t, list(z))[0])  # noqa: E731
    if w.ode == W.BRUSSELATOR:
        def rhs(t, z):
            u, v, D = z[0::2], z[1::2], th[2] * 33.0 ** 2
            up = torch.cat([torch.ones_like(u[:1]), u, torch.ones_like(u[:1])])
            vp = torch.cat([torch.full_like(v[:1], 3.0), v, torch.full_like(v[:1], 3.0)])
            fu = th[0] + u * u * v - (th[1] + 1.0) * u + D * (up[:-2] - 2.0 * u + up[2:])
            return torch.stack([fu, th[1] * u - u * u * v + D * (vp[:-2] - 2.0 * v + vp[2:])], 1).reshape(z.shape)

    def solve(t, g, r, y):
        if w.ode == W.BRUSSELATOR:
            return _newton_brusselator(th, t, g, r, y, w.newton_iters)
        return torch.stack(_newton(w.ode, th, t, g, list(r), list(y), w.newton_iters))

    F = []
    if rows[0][0] > 10:
        q, h, t0 = rows[0][0] % 10, rows[0][1], rows[0][2]
        F = [rhs(t0 - j * h, (x, h1, h2)[j]) for j in range(q)]
    for kind, h, t0, t1, hp1, hp2 in rows:
        if kind > 10:
            q = kind % 10
            xp = x + sum(h * AB[q][j] * F[j] for j in range(q))
            r = x + sum(h * AM[q][j] * F[j - 1] for j in range(1, q)) if q > 1 else x
            y = solve(t1, h * AM[q][0], r, xp)
            mu = AM_ERR[q] / (AB_ERR[q] - AM_ERR[q])
            F = [rhs(t1, y)] + F[:2]
        elif kind == 1:
            y, xp, mu = solve(t1, h, x, x), x + h * rhs(t0, x), -0.5
        elif kind == 2:
            g, r1, r2, p0, p1, p2, mu = _bdf2(h, hp1, hp2)
            xp = p0 * x + p1 * h1 + p2 * h2
            y = solve(t1, g, r1 * x + r2 * h1, xp)
        else:
            xp = -1.5 * x + 3.0 * h1 - 0.5 * h2 + 3.0 * h * rhs(t0, x)
            y, mu = solve(t1, 6.0 * h / 11.0, (18.0 * x - 9.0 * h1 + 2.0 * h2) / 11.0, xp), -6.0 / 17.0
        E = E + (mu * (y - xp)) ** 2
        x, h1, h2 = y, x, h1
    return x, h1, h2, E


def _propagate_spectral(w, th, rows, X):
    """The 2D system is linear with a circulant operator: each step is a division in its Fourier basis."""
    nt = int(round(math.sqrt(w.d)))
    a = 1.0 - torch.exp(-2j * math.pi * torch.arange(nt, device=X[0].device, dtype=F64) / nt)
    ax, ay = a[None, None, :], a[None, :, None]
    k1, k2, k3, c1, c2 = (v[:, None, None] for v in th)
    lam = -(k1 * k1 * ax.abs() ** 2 + 2.0 * k1 * k3 * (ax.conj() * ay).real + (k2 * k2 + k3 * k3) * ay.abs() ** 2) + c1 * ax + c2 * ay
    x, h1, h2 = (torch.fft.fft2(v.T.reshape(-1, nt, nt)) for v in X)
    E = torch.zeros(x.shape, device=x.device, dtype=F64)
    for kind, h, _, _, hp1, hp2 in rows:
        if kind == 1:
            g, mu, r, xp = h, -0.5, x, x + h * lam * x
        else:
            g, r1, r2, p0, p1, p2, mu = _bdf2(h, hp1, hp2)
            r, xp = r1 * x + r2 * h1, p0 * x + p1 * h1 + p2 * h2
        y = r / (1.0 - g * lam)
        E = E + (mu * torch.fft.ifft2(y - xp).real) ** 2
        x, h1, h2 = y, x, h1
    back = lambda z: torch.fft.ifft2(z).real.reshape(-1, w.d).T.contiguous()  # noqa: E731
    return back(x), back(h1), back(h2), E.reshape(-1, w.d).T.contiguous()


def _loglik(w, y, x):
    y = torch.as_tensor(y, device=x.device)[:, None]
    s = torch.as_tensor(w.sigma, device=x.device, dtype=F64)[:, None]
    s = s * y.abs().clamp_min(1e-300) if w.noise == W.NOISE_RELATIVE else s
    return -0.5 * (((y - x[w.obs_idx]) / s) ** 2).sum(0)


class _Plain:
    """One filter's committed state."""

    def __init__(self, w, device):
        self.w, self.n = w, torch.arange(w.N, device=device)
        u = _uniforms(self.n, w.seed, w.stream, 1, 0, w.p)
        phi = []
        for i in range(w.p):
            lo, hi = w.prior_lo[i], w.prior_hi[i]
            if w.prior_kind[i] == W.LOGUNIFORM:
                v = math.log(lo) + u[i] * (math.log(hi) - math.log(lo))
                phi.append(v if w.transform == W.TRANSFORM_LOG else torch.exp(v))
            else:
                v = lo + u[i] * (hi - lo)
                phi.append(torch.log(v) if w.transform == W.TRANSFORM_LOG else v)
        self.phi = torch.stack(phi)
        x0 = torch.as_tensor(np.asarray(w.x0, dtype=np.float64), device=device)[:, None].expand(-1, w.N).contiguous()
        self.X = [x0, x0, x0]
        self.lw = torch.full((w.N,), -math.log(w.N), device=device, dtype=F64)
        self.moments()

    def moments(self):
        e = torch.exp(self.lw)
        live = e > 0
        self.mean = (e * self.phi)[:, live].sum(1)
        dev = (self.phi - self.mean[:, None])[:, live]
        self.C = (e[live] * dev) @ dev.T
        self.xbar = (e * self.X[0])[:, live].sum(1)

    def shrunk(self):
        return self.w.a * self.phi + (1.0 - self.w.a) * self.mean[:, None]


def _theta(w, phi):
    return list(torch.exp(phi) if w.transform == W.TRANSFORM_LOG else phi)


def _cat_propagate(fs, rows, phis, Xs):
    """All filters of one problem and time grid in one propagation."""
    w = fs[0].w
    out = _propagate(w, _theta(w, torch.cat(phis, 1)), rows, [torch.cat(v, 1) for v in zip(*Xs)])
    return list(zip(*(v.split([f.w.N for f in fs], 1) for v in out)))


def _plain_epoch(fs, k, t_prev, hist):
    w = fs[0].w
    rows, after = _table(w, t_prev, float(w.t_obs[k]), hist)
    first = _cat_propagate(fs, rows, [f.shrunk() for f in fs], [f.X for f in fs])
    idx, ll1, phis = [], [], []
    for f, (x, *_) in zip(fs, first):
        ll = _loglik(f.w, f.w.y_obs[k], x)
        lg = f.lw + ll
        lg = torch.where(torch.isfinite(lg), lg, -math.inf)
        c = torch.cumsum(torch.exp(lg - lg.max()), 0)
        c = torch.cummax(c, 0).values
        u = _uniforms(f.n[:1], f.w.seed, f.w.stream, 4, k, 1)[0]
        tau = (f.n.to(F64) + u) / f.w.N * c[-1]
        idx.append(torch.minimum(torch.searchsorted(c, tau, right=True), torch.searchsorted(c, c[-1:])))
        ll1.append(ll[idx[-1]])
        z = torch.stack(_normals(f.n, f.w.seed, f.w.stream, 2, k, f.w.p))
        phis.append(f.shrunk()[:, idx[-1]] + math.sqrt(1.0 - f.w.a ** 2) * (torch.linalg.cholesky(f.C) @ z))
    second = _cat_propagate(fs, rows, phis, [[v[:, i] for v in f.X] for f, i in zip(fs, idx)])
    for f, (x, h1, h2, E), phi, l1 in zip(fs, second, phis, ll1):
        v = torch.sqrt(f.w.kappa * E) * torch.stack(_normals(f.n, f.w.seed, f.w.stream, 3, k, f.w.d))
        f.X, f.phi = [x + v, h1 + v, h2 + v], phi
        lw = _loglik(f.w, f.w.y_obs[k], f.X[0]) - l1
        lw = torch.where(torch.isfinite(lw), lw, -math.inf)
        f.lw = lw - torch.logsumexp(lw, 0)
        f.moments()
    return after


def _plain_runs(ws):
    """All filters' states after every epoch's estimates: [(filter, [(mean, C, xbar), ...])] in the order of ws."""
    device = "cuda" if torch.cuda.is_available() else "cpu"
    fs = [_Plain(w, device) for w in ws]
    est = [[] for _ in fs]
    for ode in {w.ode for w in ws}:
        group = [i for i, w in enumerate(ws) if w.ode == ode]
        t, hist = ws[group[0]].t0, (0, 0.0, 0.0)
        for k in range(len(ws[group[0]].t_obs)):
            hist = _plain_epoch([fs[i] for i in group], k, t, hist)
            t = float(ws[group[0]].t_obs[k])
            for i in group:
                est[i].append((fs[i].mean, fs[i].C, fs[i].xbar))
    return list(zip(fs, est))


def exact(case, seed):
    kind = case["kind"]
    if kind == "resample":
        lw = _log_weights(case["N"], seed)
        return dict(c=torch.cumsum(torch.exp(lw - lw.max()), 0), idx=None)
    ws = _members(case, seed) if kind in ("batch", "server") else [_workload(case["problem"], case["lmm"], case["N"], case["epochs"], seed)]
    runs = _plain_runs(ws)
    if kind in ("filter", "series"):
        f, est = runs[0]
        out = {k: torch.stack([e[i] for e in est]) if kind == "filter" else est[-1][i] for i, k in enumerate(("theta", "C", "xbar"))}
        return out | {k: v.T.contiguous() for k, v in zip(("x", "h1", "h2", "phi"), f.X + [f.phi])} | dict(lw=f.lw)
    out = {k: torch.cat([est[-1][i].reshape(-1) for _, est in runs]) for i, k in enumerate(("theta", "C", "xbar"))}
    cols = {k: torch.cat([f.X[i].T.reshape(-1) for f, _ in runs]) for i, k in enumerate(("x", "h1", "h2"))}
    out |= cols | dict(phi=torch.cat([f.phi.T.reshape(-1) for f, _ in runs]), lw=torch.cat([f.lw for f, _ in runs]))
    return out | (dict(status=None) if kind == "batch" else {})
