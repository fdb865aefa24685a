"""Conservation sums in which large values cancel and leave what lies far below their last bits: as close to the
exactly rounded sum as sums of two doubles are, whatever the largest value met on the way."""
import math

import numpy as np
import pytest

from paper_2212_12365_gb300 import les

pytestmark = pytest.mark.gpu


def _planted(big, where):
    def fill(g, n):
        v = g.normal(1.0, 0.3, n)
        i, j = where(n)
        v[i], v[j] = big, -big
        return v
    return fill


FILL = {
    "2^45 first and last": _planted(2.0 ** 45, lambda n: (0, n - 1)),
    "2^70 first and last": _planted(2.0 ** 70, lambda n: (0, n - 1)),
    # the window moves up with values in it, in one warp and across the grid
    "2^70 next to each other": _planted(2.0 ** 70, lambda n: (n // 2, n // 2 + 1)),
    "2^300 last": _planted(2.0 ** 300, lambda n: (n - 1, n - 2)),
    # negative values wholly below the window of an earlier one
    "below": lambda g, n: np.where(np.arange(n) == 3, 2.0 ** 60, np.where(np.arange(n) == n - 1, -2.0 ** 60,
                                                                         -g.random(n) * 2.0 ** -46)),
}


@pytest.mark.parametrize("n", [33, 256, 1025, 155649, 700001])
def test_large_values_cancel_without_a_trace(n):
    import torch
    g = np.random.default_rng(n)
    q = np.stack([f(g, n) for f in FILL.values()])
    dq = torch.from_numpy(q).cuda()
    dr = torch.zeros_like(dq)
    out = torch.empty(12, dtype=torch.float64, device="cuda")
    assert les.les_diag_sums_noalloc(dq.data_ptr(), dr.data_ptr(), n, out.data_ptr()) == les.LES_OK
    o = out.cpu().numpy()
    for f, name in enumerate(FILL):
        exact = math.fsum(q[f])
        # the result's rounding, and those of the compensations where warps and blocks are merged
        tol = np.spacing(abs(exact)) + np.abs(q[f]).sum() * 2.0 ** -100
        assert abs(o[6 + f] - exact) <= tol, (name, o[6 + f], exact, tol)
