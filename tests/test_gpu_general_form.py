"""The general-metrics stage kernels on curvilinear grids, in the conditions that the tests on jet boxes meet with the
product-grid kernels: every work decomposition of the fused FP32 stage (whole-column waves with more tiles than CTAs
among them), the staging wait that gives up, the residual monitor of a long run, full-size grids, and the
index-bounds-checked build.  Each case asserts that the handle runs the general form.

Run as a script under the bounds-checked build: prints the violation word of every case's handle."""
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
for d in (os.path.dirname(HERE), HERE):
    if d not in sys.path:
        sys.path.insert(0, d)

import oracle  # noqa: E402
from helpers import to_oracle  # noqa: E402
from paper_2212_12365_gb300 import inputs as I  # noqa: E402
from paper_2212_12365_gb300 import les  # noqa: E402

pytestmark = pytest.mark.gpu

BOX = (48, 32, 32)
GRIDS = {
    "wavy_box": lambda: (I.wavy_box_grid(BOX, amp=0.05, bc=(1, 3, 1, 1, 1, 1)), I.FlowParams(Re=1e4)),
    "polar": lambda: (I.polar_jet_grid(48, 27, 32, 10.0, 4.0), I.FlowParams(Re=1e4, TR=1.2, seed=5)),
    # periodic in i and j: no TMA map
    "wavy_periodic": lambda: (I.wavy_periodic_grid((37, 19, 10), amp=0.2), I.FlowParams(Re=800.0)),
    # 378 tiles of 32 x 8, 168 of 32 x 16: more than CTAs
    "wide_box": lambda: (I.wavy_box_grid((400, 160, 12), L=(20.0, 10.0, 2.0), amp=0.03), I.FlowParams(Re=1e4)),
    "wide_polar": lambda: (I.polar_jet_grid(400, 160, 12, 20.0, 6.0), I.FlowParams(Re=1e4, seed=3)),
}


def _run(specs, fps, tiling, polls=None, steps=3, rhs=False):
    s = les.Solver(specs, fps, les.LES_FP32)
    les.les_set_fused_tiling(s.h, *tiling)
    if polls is not None:
        les.les_debug_stage_wait(s.h, polls)
    for j, g in enumerate(specs):
        s.set_state(I.smooth_random_primitives(g, 70 + j, amp=0.04), jet=j)
    s.step(steps)
    assert "general" in les.les_describe(s.h) and "product" not in les.les_describe(s.h)
    out = [les.les_get_state_rc(s.h, g.N, les.LES_STATE_RAW, j) for j, g in enumerate(specs)]
    res = [s.rhs(j) for j in range(len(specs))] if rhs else None
    word = les.les_bounds_violation(s.h)
    rc = les.les_get_diagnostics(s.h, 0, check=False)["rc"]
    s.close()
    return out, res, word, rc


@pytest.mark.parametrize("name", sorted(GRIDS))
def test_bits_of_every_decomposition(name):
    g, fp = GRIDS[name]()
    ref, rhs, _, _ = _run([g], [fp], (8, 100000), rhs=True)
    assert np.isfinite(ref[0][0]).all()
    for t in ((16, 100000), (8, 1), (16, 5), (8, 0), (16, 0), (8, -1), (16, -1)):
        got, r, _, _ = _run([g], [fp], t, rhs=True)
        np.testing.assert_array_equal(got[0][0], ref[0][0], err_msg=str(t))
        np.testing.assert_array_equal(r[0], rhs[0], err_msg=str(t))


def test_batch_of_uneven_grids_independent_of_tiling():
    jets = [GRIDS[n]() for n in ("wavy_box", "polar", "wavy_periodic")]
    jets.append((I.wavy_box_grid((4, 4, 4), amp=0.02), I.FlowParams(Re=100.0)))
    specs, fps = [g for g, _ in jets], [f for _, f in jets]
    ref, _, _, _ = _run(specs, fps, (8, 100000))
    for t in ((16, 100000), (8, 1), (16, 5), (8, 0), (16, 0), (8, -1), (16, -1)):
        got, _, _, _ = _run(specs, fps, t)
        for (a, _), (b, _) in zip(ref, got):
            np.testing.assert_array_equal(b, a, err_msg=str(t))


@pytest.mark.parametrize("name,tiling", [("wavy_box", (8, 0)), ("wavy_box", (16, 5)), ("polar", (16, 0)),
                                         ("polar", (8, 3)), ("wide_box", (8, -1)), ("wide_polar", (16, -1))])
def test_wait_that_gives_up(name, tiling):
    """The first staging wait of every CTA gives up while its copy is in flight: reported as site 8, the rest of the
    launch by direct loads, the same bits."""
    g, fp = GRIDS[name]()
    ref, _, w0, rc0 = _run([g], [fp], tiling, steps=2)
    got, _, w1, rc1 = _run([g], [fp], tiling, polls=0, steps=2)
    assert ref[0][1] == les.LES_OK and w0 == 0 and rc0 == les.LES_OK
    assert got[0][1] == les.LES_ERR_TIMEOUT and rc1 == les.LES_ERR_TIMEOUT and w1 >> 48 == 8
    np.testing.assert_array_equal(got[0][0], ref[0][0])


def test_wait_that_gives_up_in_a_batch():
    """Staged and unstaged grids together; and enough of them that the lockstep form walks waves first."""
    import torch
    jets = [GRIDS[n]() for n in ("wavy_box", "wavy_periodic", "polar")]
    n = torch.cuda.get_device_properties(0).multi_processor_count // 8
    for reps, tiling in ((1, (8, 3)), (n, (16, -1))):
        specs, fps = [g for g, _ in jets] * reps, [f for _, f in jets] * reps
        ref, _, _, _ = _run(specs, fps, tiling, steps=2)
        got, _, word, rc = _run(specs, fps, tiling, polls=0, steps=2)
        assert word >> 48 == 8 and rc == les.LES_ERR_TIMEOUT
        for (a, rca), (b, rcb) in zip(ref, got):
            assert rca == les.LES_OK and rcb == les.LES_ERR_TIMEOUT
            np.testing.assert_array_equal(b, a)


@pytest.mark.slow
def test_residual_monitor_identical_across_decompositions():
    spec, fp = GRIDS["polar"]()
    runs = []
    for t in ((8, 100000), (16, 5), (8, 0), (16, 0)):
        s = les.Solver(spec, fp, les.LES_FP32)
        les.les_set_fused_tiling(s.h, *t)
        s.set_state(I.ambient_primitives(spec.N, fp.TR))
        hist = []
        for _ in range(10):
            s.step(100)
            hist.append(s.diagnostics()["max_abs_rhs_rho"])
        assert "general" in les.les_describe(s.h)
        runs.append((np.array(hist), s.get_state(les.LES_STATE_RAW)))
        s.close()
    h0, q0 = runs[0]
    assert np.all(np.isfinite(h0)) and h0[-1] > 0
    for h, q in runs[1:]:
        np.testing.assert_array_equal(h, h0)
        np.testing.assert_array_equal(q, q0)


@pytest.mark.slow
@pytest.mark.parametrize("prec,tol", [(les.LES_FP64, 1e-12), (les.LES_FP32, 2e-5)])
def test_full_size_sampled_residual(prec, tol):
    """The polar mesh of the paper's topology at 384 x 192 x 192 (14.2 M points): the residual at sampled points
    (next to the axis, faces and edges too) against the oracle's, of each field's scale; the bounds of the
    full-size jets."""
    spec, fp = I.polar_jet_grid(384, 192, 192, 30.0, 12.0), I.FlowParams(Re=1e5)
    prim = I.smooth_random_primitives(spec, seed=31, amp=0.05)
    g, p = to_oracle(spec, fp)
    m = oracle.metrics(g)
    q = oracle.apply_bc(g, p, m, oracle.qhat_from(g, p, m, prim, True), 0)
    ni, nj, nk = spec.dims
    rng = np.random.default_rng(5)
    pts = [np.stack([rng.integers(1, ni - 1, 3000), rng.integers(1, nj - 1, 3000), rng.integers(0, nk, 3000)], 1)]
    pts += [np.array([[i, j, k]]) for i in (1, ni // 2, ni - 2) for j in (1, 2, nj // 2, nj - 2) for k in (0, 1, nk - 1)]
    pq = np.concatenate(pts)
    lin = (pq[:, 2].astype(np.int64) * nj + pq[:, 1]) * ni + pq[:, 0]
    r_or = oracle.rhs_sampled(g, p, m, q, lin)
    del m, q
    s = les.Solver(spec, fp, prec)
    s.set_state(prim)
    s.step(0)
    assert "general" in les.les_describe(s.h)
    r = s.rhs()[:, lin]
    s.close()
    err = np.abs(r - r_or) / (np.abs(r_or).max(axis=1, keepdims=True) + 1e-30)
    print("polar 384x192x192 sampled residual error / scale:", err.max(axis=1))
    assert err.max() < tol, err.max(axis=1)


def test_no_index_out_of_range():
    from paper_2212_12365_gb300 import build
    build.build(bounds=True)
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=dict(os.environ, LES_LIBRARY=build.BOUNDS_LIB),
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    words = dict(line.rsplit(" ", 1) for line in r.stdout.split("\n") if line.startswith("case "))
    assert len(words) == len(GRIDS) * 4 and set(words.values()) == {"0x0"}, words


if __name__ == "__main__":
    assert les.les_bounds_checking()
    for name, make in sorted(GRIDS.items()):
        g, fp = make()
        for t in ((8, -1), (16, -1), (16, 3), (8, 0)):
            print("case", name, t, hex(_run([g], [fp], t, steps=2)[2]))
