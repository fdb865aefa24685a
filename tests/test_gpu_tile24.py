"""Tile height 24 of the product-grid FP32 stage, which the tuner takes on large boxes, set by the caller: the same
bits as tile height 8 on every product grid, at rows around its tiles' edges, in every work decomposition, after a
staging wait that gave up, in a batch with curvilinear jets, and without an index out of range.

Run as a script under the index-bounds-checked build: prints the violation word of every case's handle."""
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
for d in (os.path.dirname(HERE), HERE):
    if d not in sys.path:
        sys.path.insert(0, d)

from paper_2212_12365_gb300 import inputs as I  # noqa: E402
from paper_2212_12365_gb300 import les  # noqa: E402
from test_gpu_separable import CASES as PRODUCT  # noqa: E402

pytestmark = pytest.mark.gpu

# 22 output rows per tile: the last tile full, one row short and with one row, on bounded and periodic j axes
GRIDS = dict(PRODUCT)
GRIDS.update({f"rows_{nj}": (lambda nj=nj: I.jet_grid(34, nj, 9, 6.0, 5.0, 4.0, 0.05, 0.3)) for nj in (23, 24, 25, 46, 47)})
GRIDS.update({f"periodic_rows_{nj}": (lambda nj=nj: I.periodic_box_grid((33, nj, 6), (0.3, 0.2, 0.25))) for nj in (21, 22, 23, 45)})
TILINGS = ((24, 0), (24, -1), (24, 3), (24, 1), (24, 100000))


def _run(specs, fps, prec, tiling, polls=None, steps=3):
    s = les.Solver(specs, fps, prec)
    les.les_set_fused_tiling(s.h, *tiling)
    if polls is not None:
        les.les_debug_stage_wait(s.h, polls)
    for j, g in enumerate(specs):
        s.set_state(I.smooth_random_primitives(g, 70 + j, amp=0.05), jet=j)
    s.step(steps)
    out = [les.les_get_state_rc(s.h, g.N, les.LES_STATE_RAW, j) for j, g in enumerate(specs)]
    rhs = [s.rhs(j) for j in range(len(specs))] if polls is None else None
    info = les.les_describe(s.h), les.les_bounds_violation(s.h)
    s.close()
    return out, rhs, info


@pytest.mark.parametrize("name", sorted(GRIDS))
def test_bits_of_every_decomposition(name):
    g, fp = GRIDS[name](), I.FlowParams(Re=800.0)
    ref, rhs, _ = _run([g], [fp], les.LES_FP32, (8, 0))
    assert np.isfinite(ref[0][0]).all()
    for prec in (les.LES_FP32, les.LES_FP32_SEPARABLE):
        for t in TILINGS:
            got, r, info = _run([g], [fp], prec, t)
            assert "ty=24" in info[0] and info[1] == 0
            np.testing.assert_array_equal(got[0][0], ref[0][0], err_msg=str(t))
            np.testing.assert_array_equal(r[0], rhs[0], err_msg=str(t))


def test_more_tiles_than_ctas():
    """A grid whose whole-column waves of tiles of 24 rows are followed by shared-out planes."""
    import torch
    g, fp = I.jet_grid(640, 180, 12, 30.0, 10.0, 10.0, 0.05, 0.1), I.FlowParams(Re=1e4)
    assert -(-638 // 30) * -(-178 // 22) > torch.cuda.get_device_properties(0).multi_processor_count
    ref, _, _ = _run([g], [fp], les.LES_FP32, (8, 100000), steps=2)
    for t in ((24, -1), (24, 0), (24, 4)):
        got, _, info = _run([g], [fp], les.LES_FP32, t, steps=2)
        assert "ty=24" in info[0]
        np.testing.assert_array_equal(got[0][0], ref[0][0])


@pytest.mark.parametrize("tiling", [(24, 0), (24, 5), (24, -1)])
def test_wait_that_gives_up(tiling):
    """Single jet, and a batch of enough jets that the lockstep form has more tiles than CTAs."""
    import torch
    spec, fp = I.jet_small()
    ref, _, _ = _run([spec], [fp], les.LES_FP32, tiling)
    got, _, info = _run([spec], [fp], les.LES_FP32, tiling, 0)
    assert got[0][1] == les.LES_ERR_TIMEOUT and info[1] >> 48 == 8
    np.testing.assert_array_equal(got[0][0], ref[0][0])
    if tiling == (24, -1):
        n = torch.cuda.get_device_properties(0).multi_processor_count // 4 + 2
        specs = [spec] * n
        ref, _, _ = _run(specs, [fp] * n, les.LES_FP32, tiling, steps=2)
        got, _, info = _run(specs, [fp] * n, les.LES_FP32, tiling, 0, steps=2)
        assert info[1] >> 48 == 8
        for (a, rca), (b, rcb) in zip(ref, got):
            assert rca == les.LES_OK and rcb == les.LES_ERR_TIMEOUT
            np.testing.assert_array_equal(b, a)


def test_a_batch_with_curvilinear_jets_takes_16_rows_for_those():
    specs = [GRIDS["rows_47"](), I.wavy_box_grid((14, 27, 9), amp=0.05), GRIDS["tiny_jet_4x4x4"]()]
    fps = [I.FlowParams(Re=900.0)] * 3
    ref, rhs, _ = _run(specs, fps, les.LES_FP32, (8, 0))
    got, r, info = _run(specs, fps, les.LES_FP32, (24, -1))
    assert "product ty=24" in info[0] and "general ty=16" in info[0]
    for j in range(3):
        np.testing.assert_array_equal(got[j][0], ref[j][0])
        np.testing.assert_array_equal(r[j], rhs[j])


def test_refused_without_a_product_grid():
    s = les.Solver(I.wavy_box_grid((12, 10, 9), amp=0.05), I.FlowParams(), les.LES_FP32)
    with pytest.raises(les.LesError) as e:
        les.les_set_fused_tiling(s.h, 24, 0)
    assert e.value.code == les.LES_ERR_ARG
    s.close()


def test_no_index_out_of_range():
    from paper_2212_12365_gb300 import build
    build.build(bounds=True)
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=dict(os.environ, LES_LIBRARY=build.BOUNDS_LIB),
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    words = dict(line.rsplit(" ", 1) for line in r.stdout.split("\n") if line.startswith("case "))
    assert len(words) == len(GRIDS) * 3 and set(words.values()) == {"0x0"}, words


if __name__ == "__main__":
    assert les.les_bounds_checking()
    for name, make in sorted(GRIDS.items()):
        for t in ((24, 0), (24, -1), (24, 1)):
            print("case", name, t, hex(_run([make()], [I.FlowParams(Re=800.0)], les.LES_FP32, t, steps=2)[2][1]))
