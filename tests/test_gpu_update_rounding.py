"""The stage update rounds the state once.  With a time step so small (and no inflow noise) that the residual does not change over a step,
the new state is Q(0) - dt R rounded to FP64, R the residual of Q(0); Q(0) and R come from the library, the reference
from extended precision."""
import numpy as np
import pytest

from paper_2212_12365_gb300 import inputs as I
from paper_2212_12365_gb300 import les

pytestmark = pytest.mark.gpu
DT = 1e-12
GRIDS = {
    "jet": lambda: I.jet_grid(41, 33, 27, 8.0, 6.0, 6.0, 0.15, 0.18),
    "periodic": lambda: I.periodic_box_grid((16, 15, 14), (0.3, 0.25, 0.2)),
    "wavy_box": lambda: I.wavy_box_grid((24, 21, 19), amp=0.05),
    "polar": lambda: I.polar_jet_grid(30, 14, 16, 10.0, 4.0),
}


@pytest.mark.parametrize("name", sorted(GRIDS))
def test_one_rounding_of_the_state(name):
    spec = GRIDS[name]()
    s = les.Solver(spec, I.FlowParams(Re=1e4, TR=1.3, dt=DT, noise_amp=0.0), les.LES_FP64)
    s.set_state(I.smooth_random_primitives(spec, 9, amp=0.08))
    q0, r = s.get_state(les.LES_STATE_RAW), s.rhs()
    s.step(1)
    q1 = s.get_state(les.LES_STATE_RAW)
    s.close()
    # points that the stage updates: inside the ends of the axes that are not periodic
    inner = np.ones(spec.dims[::-1], bool)
    for a, per in enumerate(spec.periodic):
        if not per:
            ix = [slice(None)] * 3
            ix[2 - a] = [0, -1]
            inner[tuple(ix)] = False
    inner = inner.reshape(-1)
    exact = q0.astype(np.longdouble) - np.longdouble(DT) * r.astype(np.longdouble)
    err = np.abs((q1.astype(np.longdouble) - exact)[:, inner]).astype(float) / np.spacing(np.abs(q1[:, inner]))
    moved = np.abs(q1 - q0)[:, inner].max()
    assert moved > 0
    # half a unit, and what the residual changes over the step (relative 1e-10 of dt R)
    assert err.max() <= 0.51, err.max(axis=1)
