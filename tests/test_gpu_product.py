"""The stage forms that leave out the zeros of a diagonal metric, which a product grid x(i), y(j), z(k) takes by
itself, against the oracle's general metrics: every boundary type, periodic axes, minimum and ragged sizes; and the
product grids that must stay on the general form (descending axes, sheared periods)."""
import numpy as np
import pytest

import oracle
from helpers import rel_l2, to_oracle
from paper_2212_12365_gb300 import inputs as I
from paper_2212_12365_gb300 import les
from test_gpu_separable import CASES as PRODUCT

pytestmark = pytest.mark.gpu


def _descending():
    g = I.jet_grid(21, 14, 13, 6.0, 5.0, 4.0, 0.3, 0.3)
    g.y, g.z = -g.y, -g.z
    return g


def _sheared():
    g = I.periodic_box_grid((9, 12, 7), (0.3, 0.25, 0.3))
    g.shift = g.shift.copy()
    g.shift[1, 0] = 0.05  # one period of j also moves x
    return g


CASES = {**PRODUCT, "descending_y_z": _descending, "sheared_period": _sheared, "wide_65x64x5": lambda: I.jet_grid(65, 64, 5, 6.0, 6.0, 2.0, 0.1, 0.4)}
GENERAL = {"descending_y_z", "sheared_period"}
# residual (of its scale) and state after five steps (relative L2 per field): the bounds that the general forms are
# held to, FP64 1e-12, FP32 2e-5
TOL = {les.LES_FP64: 1e-12, les.LES_FP32: 2e-5}


@pytest.mark.parametrize("prec", sorted(TOL))
@pytest.mark.parametrize("case", sorted(CASES))
def test_product_residual_and_steps(case, prec):
    spec = CASES[case]()
    fp = I.FlowParams(Re=800.0, TR=1.4)
    prim = I.smooth_random_primitives(spec, 17, amp=0.08)
    g, p = to_oracle(spec, fp)
    m = oracle.metrics(g)
    q = oracle.apply_bc(g, p, m, oracle.qhat_from(g, p, m, prim, True), 0)
    r_or = oracle.rhs(g, p, m, q)
    ref = oracle.state_out(g, p, m, oracle.step(g, p, m, q, 5, 0, oracle.dt_cfl(g, p, m, q)), False)
    s = les.Solver(spec, fp, prec)
    s.set_state(prim)
    s.step(0)
    want = "general" if case in GENERAL else "product"
    assert want in les.les_describe(s.h)
    r = s.rhs()
    s.step(5)
    got = s.get_state(les.LES_STATE_CONSERVED)
    s.close()
    if prec == les.LES_FP32:  # the tuned work list and the fixed ones give the same bits
        for ty, kc in ((8, 0), (16, -1), (16, 3)):
            s = les.Solver(spec, fp, prec)
            les.les_set_fused_tiling(s.h, ty, kc)
            s.set_state(prim)
            np.testing.assert_array_equal(s.rhs(), r)
            s.step(5)
            np.testing.assert_array_equal(s.get_state(les.LES_STATE_CONSERVED), got)
            s.close()
    scale = np.abs(r_or).max(axis=1, keepdims=True) + 1e-30
    err = np.abs(r - r_or) / scale
    assert err.max() < TOL[prec], (case, err.max(axis=1))
    assert np.all(rel_l2(got, ref) <= TOL[prec]), (case, rel_l2(got, ref))


@pytest.mark.parametrize("prec", sorted(TOL))
def test_mixed_batch_bit_identical_to_single(prec):
    """Product and curvilinear jets in one batch: each keeps the form, and the bits, of a single handle."""
    specs = [CASES["jet_ragged_70x37x29"](), I.wavy_box_grid((14, 11, 9), amp=0.05), CASES["tiny_jet_4x4x4"](),
             I.polar_jet_grid(20, 9, 12, 6.0, 3.0), CASES["descending_y_z"](), CASES["mixed_periodic_z"]()]
    fps = [I.FlowParams(Re=2e3, TR=1.0 + 0.2 * j, seed=j + 3) for j in range(len(specs))]
    prims = [I.smooth_random_primitives(g, 5 + j, amp=0.04) for j, g in enumerate(specs)]
    b = les.Solver(specs, fps, prec)
    for j, q in enumerate(prims):
        b.set_state(q, jet=j)
    b.step(3)
    for j, (g, f, q) in enumerate(zip(specs, fps, prims)):
        s = les.Solver(g, f, prec)
        s.set_state(q)
        s.step(3)
        np.testing.assert_array_equal(b.get_state(les.LES_STATE_RAW, jet=j), s.get_state(les.LES_STATE_RAW))
        np.testing.assert_array_equal(b.rhs(jet=j), s.rhs())
        s.close()
    b.close()
