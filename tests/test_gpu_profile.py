"""les_profile_step times every kernel launch by itself: per kind as many counts as a step launches kernels, on grids
with a centerline and in batches whose jets take both forms of the stage."""
import pytest

from paper_2212_12365_gb300 import inputs as I
from paper_2212_12365_gb300 import les

pytestmark = pytest.mark.gpu
JET = lambda: I.jet_grid(20, 13, 11, 6.0, 5.0, 4.0, 0.3, 0.3)  # noqa: E731
POLAR = lambda: I.polar_jet_grid(20, 9, 12, 6.0, 3.0)  # noqa: E731
# grids, launches of one part of a stage (forms in use), launches of a boundary pass
CASES = {"jet": ((JET,), 1, 1), "polar": ((POLAR,), 1, 2), "both": ((JET, POLAR), 2, 2),
         "box": ((lambda: I.periodic_box_grid((8, 8, 8), (0.3, 0.3, 0.3)),), 1, 0)}


@pytest.mark.parametrize("prec", [les.LES_FP64, les.LES_FP32])
@pytest.mark.parametrize("case", sorted(CASES))
def test_every_launch_is_counted(case, prec):
    grids, forms, faces = CASES[case]
    specs = [g() for g in grids]
    fps = [I.FlowParams(Re=1e3) for _ in specs]
    s = les.Solver(specs, fps, prec)
    for j, g in enumerate(specs):
        s.set_state(I.smooth_random_primitives(g, 3 + j, amp=0.02), jet=j)
    s.step(1)
    per_step = les.les_last_launch_count(s.h)
    prof = les.les_profile_step(s.h, 2)
    s.close()
    assert sum(c for _, c in prof.values()) == 2 * per_step
    assert prof["bc"][1] == 2 * 5 * faces and prof["other"][1] == 2
    for k in ("point", "grads", "update"):
        assert prof[k][1] == (2 * 5 * forms if prec == les.LES_FP64 else 0)
    assert prof["iface"][1] == 2 * 5 * forms
    assert all((ms > 0) == (c > 0) for ms, c in prof.values())
