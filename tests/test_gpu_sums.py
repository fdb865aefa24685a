"""The residual / conservation sums' fixed-point accumulation against the exactly rounded sums (math.fsum): sizes
around a warp, a block and the full grid, exponents spread over the window and beyond it, cancellation, subnormals,
zeros and non-finite values."""
import math

import numpy as np
import pytest

from paper_2212_12365_gb300 import les

pytestmark = pytest.mark.gpu
FILL = {
    "plain": lambda g, n: g.normal(1.0, 0.3, n),
    "spread": lambda g, n: g.normal(size=n) * 2.0 ** g.integers(-300, 300, n),
    # growing values: the window moves at almost every block of points
    "growing": lambda g, n: g.normal(size=n) * 2.0 ** np.linspace(-60, 60, n),
    # pairs that cancel to a remainder 2^-40 of the terms
    "cancel": lambda g, n: (lambda v: np.where(np.arange(n) % 2, -np.roll(v, 1), v) + 2.0 ** -40 * g.normal(size=n))(
        g.normal(size=n)),
    "tiny": lambda g, n: g.normal(size=n) * 1e-310,
}


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1025, 155648 + 1, 700001])
def test_sums_exactly_rounded(n):
    import torch
    g = np.random.default_rng(n)
    q = np.stack([f(g, n) for f in FILL.values()])
    r = g.normal(0.0, 1e-2, (5, n))
    dq, dr = torch.from_numpy(q).cuda(), torch.from_numpy(r).cuda()
    out = torch.empty(12, dtype=torch.float64, device="cuda")
    assert les.les_diag_sums_noalloc(dq.data_ptr(), dr.data_ptr(), n, out.data_ptr()) == les.LES_OK
    o = out.cpu().numpy()
    assert o[0] == np.abs(r[0]).max() and o[11] == 0
    np.testing.assert_allclose(o[1:6], np.sqrt((r ** 2).sum(axis=1)), rtol=1e-12)
    for f, name in enumerate(FILL):
        exact, big = math.fsum(q[f]), np.abs(q[f]).max()
        # s + c rounded once, and the truncated tails: 2^-96 of the largest value each, plus the merges of the
        # compensations (2^-104 of the magnitude sum)
        tol = np.spacing(abs(exact)) + n * big * 2.0 ** -96 + np.abs(q[f]).sum() * 2.0 ** -100
        assert abs(o[6 + f] - exact) <= tol, (name, o[6 + f], exact)
    q[3, n // 2] = np.inf
    r[1, n - 1] = np.nan
    dq.copy_(torch.from_numpy(q))
    dr.copy_(torch.from_numpy(r))
    assert les.les_diag_sums_noalloc(dq.data_ptr(), dr.data_ptr(), n, out.data_ptr()) == les.LES_OK
    o = out.cpu().numpy()
    assert o[11] == 2 and np.isnan(o[9]) and np.isnan(o[2]) and np.isfinite(o[6])
