"""The fixed-point exp and sqrt of csrc/pf_math.cuh: a host build against mpmath
(CPU), and the device build against the host build and the library (GPU)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1411_1702_gb300", "csrc")
EDGES = [0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, 5e-324, 2.0 ** -1022, np.finfo(float).max, 709.0, 709.8, 710.0, 704.0,
         -704.0, -708.5, -745.0, -745.2, -746.5, -1e10, 63.999, 64.0, -64.0, 1e-300, 2.0 ** -53, 1 - 2.0 ** -53, 2 - 2.0 ** -52]


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fixedshim") / "libfixed_shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-fPIC", "-shared", "-I", CSRC,
                    os.path.join(ROOT, "tests", "fixed_shim.cpp"), "-o", out], check=True)
    L = C.CDLL(out)
    for f in (L.shim_exp, L.shim_sqrt):
        f.argtypes = [C.c_void_p, C.c_void_p, C.c_long]
    return L


def _run(f, x):
    x = np.ascontiguousarray(x, dtype=np.float64)
    y = np.empty_like(x)
    f(x.ctypes.data, y.ctypes.data, len(x))
    return y


def _inputs(rng, n):
    """exp's arguments of every size, around the table's steps and the edges of its ranges."""
    k = rng.integers(-130000, 130000, n)
    step = k * (np.log(2) / 128) + rng.uniform(-1e-9, 1e-9, n)
    half = (k + 0.5) * (np.log(2) / 128) + rng.uniform(-1e-7, 1e-7, n)
    return np.concatenate([rng.uniform(-18, 18, n), rng.uniform(-703, 703, n), step, half,
                           rng.standard_normal(n) * 2.0 ** rng.uniform(-70, 0, n)])


def test_exp_and_sqrt_within_their_bounds(shim):
    mpmath = pytest.importorskip("mpmath")
    mpmath.mp.dps = 40
    rng = np.random.default_rng(3)
    x = _inputs(rng, 1500)
    x = x[np.abs(x) < 704]
    y = _run(shim.shim_exp, x)
    err = [abs(mpmath.mpf(float(b)) - mpmath.exp(mpmath.mpf(float(a)))) / mpmath.mpf(float(np.spacing(b))) for a, b in zip(x, y)]
    assert max(err) <= 0.6
    # just under, at and above powers of two and squares, where the result's last bit turns
    m = np.concatenate([1 + rng.random(3000), 1 + 2.0 ** -rng.integers(1, 53, 500).astype(float),
                        2 - 2.0 ** -rng.integers(1, 52, 500).astype(float), (1 + rng.integers(0, 2 ** 20, 500) / 2.0 ** 20) ** 2])
    x = np.concatenate([m * 2.0 ** rng.integers(-1000, 1000, len(m)).astype(float), m, 2 * m])
    y = _run(shim.shim_sqrt, x)
    err = [abs(mpmath.mpf(float(b)) - mpmath.sqrt(mpmath.mpf(float(a)))) / mpmath.mpf(float(np.spacing(b))) for a, b in zip(x, y)]
    assert max(err) <= 0.51


def test_edges_are_the_library_s(shim):
    x = np.array(EDGES)
    with np.errstate(all="ignore"):
        assert np.allclose(_run(shim.shim_exp, x), np.exp(x), rtol=2.0 ** -52, atol=0, equal_nan=True)
        assert np.allclose(_run(shim.shim_sqrt, x), np.sqrt(x), rtol=2.0 ** -52, atol=0, equal_nan=True)


@pytest.mark.gpu
def test_device_build(shim):
    import torch
    from paper_1411_1702_gb300 import build as B
    B.build()
    P = C.CDLL(B.PROBE_LIB)
    P.pf_probe_fixed.argtypes = [C.c_void_p, C.c_int64, C.c_void_p, C.c_void_p]
    x = np.concatenate([_inputs(np.random.default_rng(4), 1 << 14), EDGES])
    d = torch.from_numpy(x).cuda()
    e, r = torch.empty_like(d), torch.empty_like(d)
    assert P.pf_probe_fixed(d.data_ptr(), len(x), e.data_ptr(), r.data_ptr()) == 0
    he, hr = _run(shim.shim_exp, x), _run(shim.shim_sqrt, x)
    inside = np.abs(x) < 704
    assert np.array_equal(e.cpu().numpy()[inside], he[inside])
    assert np.allclose(e.cpu().numpy(), he, rtol=2.0 ** -51, atol=5e-324, equal_nan=True)
    assert np.allclose(r.cpu().numpy(), hr, rtol=2.0 ** -52, atol=0, equal_nan=True)
