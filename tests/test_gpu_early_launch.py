"""Resampling whose launches overlap the kernels that write what they read
(pf_resample_systematic_noalloc): buffers that start 8 bytes off a cache line, so that
a line of the cumulative weights is written by two blocks, at sizes with one and
with two resampling launches; weights and indices against numpy and the oracle, each
size twice in a row with other weights in the same buffers."""
import numpy as np
import pytest

import oracle
from paper_1411_1702_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 257, 4097, 131071, 311296, 312321, 1000003])
@pytest.mark.parametrize("off", [0, 1, 15])
def test_offset_buffers(N, off):
    import torch
    B.build()
    oracle.build()
    from paper_1411_1702_gb300 import pf
    lw = torch.empty(N + 32, dtype=torch.float64, device="cuda")
    c = torch.empty(N + 32, dtype=torch.float64, device="cuda")
    idx = torch.empty(N + 32, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream or None
    rng = np.random.default_rng([N, off])
    for u in (0.0, 0.73):
        lg = rng.standard_normal(N) * 3.0
        lg[rng.random(N) < 0.1] = -np.inf
        lg[N // 2] = 1.0
        c.fill_(-1.0)
        idx.fill_(-7)
        lw[off:off + N] = torch.tensor(lg, device="cuda")
        pf.pf_resample_systematic_noalloc(lw[off:].data_ptr(), N, u, c[off:].data_ptr(), idx[off:].data_ptr(), stream)
        torch.cuda.synchronize()
        cn, ix = c.cpu().numpy(), idx.cpu().numpy()
        g = np.where(np.isfinite(lg), np.exp(np.where(np.isfinite(lg), lg, 0.0) - lg[np.isfinite(lg)].max()), 0.0)
        ref = np.cumsum(g.astype(np.longdouble))
        # the reference's sums in order: at most N 2^-64 (an 80-bit long double); the kernel's go through
        # fewer than 80 additions each: 80 2^-53; the exponentials: an ulp on each side
        tol = N * 2.0 ** -64 + 82 * 2.0 ** -53
        assert np.all(np.abs(cn[off:off + N] - ref) <= tol * ref)
        assert np.all(np.diff(cn[off:off + N]) >= 0.0)
        assert np.array_equal(ix[off:off + N], oracle.resample_systematic(cn[off:off + N], u))
        # nothing outside the buffers
        assert np.all(cn[:off] == -1.0) and np.all(cn[off + N:] == -1.0)
        assert np.all(ix[:off] == -7) and np.all(ix[off + N:] == -7)
