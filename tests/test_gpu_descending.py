"""A product grid with two descending axes (positive volumes, negative spacings): LES_FP32_SEPARABLE runs the
product-grid kernel there and LES_FP32 the general one, so that the two kernels meet on one grid; each against the
oracle, and one against the other."""
import numpy as np
import pytest

import oracle
from helpers import rel_l2, to_oracle
from paper_2212_12365_gb300 import inputs as I
from paper_2212_12365_gb300 import les

pytestmark = pytest.mark.gpu


def _flipped(dims, axes):
    g = I.jet_grid(*dims, 6.0, 5.0, 4.0, 0.2, 0.25)
    for a in axes:
        v = getattr(g, "xyz"[a])
        setattr(g, "xyz"[a], v.max() - v if a == 0 else -v)
    if 0 in axes:  # the entrance stays at i-
        g.bc = (1, 3, 1, 1, 1, 1)
    return g


@pytest.mark.parametrize("axes", [(1, 2), (0, 1), (0, 2)])
@pytest.mark.parametrize("dims", [(21, 14, 13), (63, 37, 9)])
def test_separable_on_descending_axes(dims, axes):
    spec, fp = _flipped(dims, axes), I.FlowParams(Re=800.0, TR=1.4)
    prim = I.smooth_random_primitives(spec, 17, amp=0.08)
    g, p = to_oracle(spec, fp)
    m = oracle.metrics(g)
    q = oracle.apply_bc(g, p, m, oracle.qhat_from(g, p, m, prim, True), 0)
    r_or = oracle.rhs(g, p, m, q)
    ref = oracle.state_out(g, p, m, oracle.step(g, p, m, q, 10, 0, oracle.dt_cfl(g, p, m, q)), False)
    out = {}
    for prec, form in ((les.LES_FP32, "general"), (les.LES_FP32_SEPARABLE, "product (separable)")):
        s = les.Solver(spec, fp, prec)
        s.set_state(prim)
        s.step(0)
        assert form in les.les_describe(s.h)
        r = s.rhs()
        s.step(10)
        out[prec] = s.get_state(les.LES_STATE_CONSERVED)
        s.close()
        err = np.abs(r - r_or) / (np.abs(r_or).max(axis=1, keepdims=True) + 1e-30)
        assert err.max() < 2e-5, (form, err.max(axis=1))
        assert np.all(rel_l2(out[prec], ref) <= 2e-5), (form, rel_l2(out[prec], ref))
    # the bound that the separable and the general FP32 forms are held to on ascending axes
    err = rel_l2(out[les.LES_FP32_SEPARABLE], out[les.LES_FP32])
    assert np.all(err <= 5e-6), err
