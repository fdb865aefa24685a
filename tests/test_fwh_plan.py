"""The sizes that les_fwh takes for an evaluation (csrc/les_fwh_plan.h, plain C++): which calls get the staged
observer pass, that a window holds every frame its block reads, and that it fits the chip."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2212_12365_gb300", "csrc")
SRC = """
#include "les_fwh_plan.h"
extern "C" void plan(int npts, int N, int nobs, int nt, double dt_obs, double dtau, double c0, double spread, int nsm,
                     long long *o)
{
    const les::FwhPlan P = les::fwh_plan(npts, N, nobs, nt, dt_obs, dtau, c0, spread, nsm);
    const long long v[] = {P.MG, P.ngroups, P.staged, P.T, P.tblocks, P.W, P.span, P.nth, P.NB, P.nchunk,
                           (long long)P.b_src, (long long)P.b_rec, (long long)P.b_part,
                           P.staged ? (long long)les::fwh_win_smem(P.W, les::fwh_rows(P.MG)) : 0};
    for (int i = 0; i < 14; ++i) o[i] = v[i];
}
"""
KEYS = "MG ngroups staged T tblocks W span nth NB nchunk b_src b_rec b_part smem".split()


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("fwh_plan")
    (d / "p.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "p.cpp"), "-o",
                    str(d / "p.so")], check=True)
    f = ctypes.CDLL(str(d / "p.so")).plan
    f.argtypes = [ctypes.c_int] * 4 + [ctypes.c_double] * 4 + [ctypes.c_int, ctypes.POINTER(ctypes.c_longlong)]

    def call(npts, N, nobs, nt, ratio, spread, nsm=152):
        o = (ctypes.c_longlong * 14)()
        f(npts, N, nobs, nt, 0.1 * ratio, 0.1, 1.0, 0.1 * spread, nsm, o)  # dtau 0.1, c0 1: spread in frames
        return dict(zip(KEYS, o))
    return call


def _staged_blocks_of_256(nobs, ratio, spread):
    """Whether a staged pass with blocks of 256 times, FP64 accumulators of every microphone and at least four panel
    windows in 100 KB would run: the reach the staged pass must not fall short of."""
    mg = min(16, nobs)
    w = math.ceil(spread) + math.ceil(255 * ratio) + 4
    return (100 * 1024 - mg * 256 * 8) // (32 * (mg + w) + 4) >= 4


def test_windows_that_fit_blocks_of_256_times_are_staged(plan):
    rng = np.random.default_rng(1)
    seen = 0
    for _ in range(4000):
        nobs, nt = int(rng.integers(1, 80)), int(2 ** rng.uniform(0, 12))
        ratio, spread = rng.choice([0.0, 0.3, 0.5, 1.0, rng.uniform(0, 3)]), rng.uniform(0, 800) * (nobs > 1)
        if not _staged_blocks_of_256(nobs, ratio, spread):
            continue
        seen += 1
        assert plan(10000, 1024, nobs, nt, ratio, spread)["staged"], (nobs, nt, ratio, spread)
    assert seen > 1000


@pytest.mark.parametrize("mics,nt,spread", [(24, 512, 180), (32, 512, 180), (20, 512, 175), (4, 512, 340), (8, 320, 340),
                                            (8, 512, 340)])
def test_neighbours_of_the_64_microphone_arc_are_staged(plan, mics, nt, spread):
    """Dense observer times of microphone arcs whose groups spread over hundreds of frames."""
    assert plan(98304, 1024, mics, nt, 1.0, spread)["staged"]


def test_a_window_holds_its_block_and_fits_the_chip(plan):
    rng = np.random.default_rng(2)
    for _ in range(4000):
        nobs, nt = int(rng.integers(1, 200)), int(2 ** rng.uniform(0, 13))
        ratio, spread = rng.uniform(0, 4), rng.uniform(0, 900) * (nobs > 1)
        p = plan(int(2 ** rng.uniform(0, 17)), int(rng.integers(3, 3000)), nobs, nt, ratio, spread)
        assert p["MG"] <= 16 and p["MG"] * p["ngroups"] >= nobs and p["T"] * p["tblocks"] >= nt
        assert p["nchunk"] >= 1 and 1 <= p["NB"]
        if not p["staged"]:
            continue
        # entries off - 1 .. off + span, off from 1 to 1 + the spread in frames: the last index is read as ix + 1
        last = 1 + math.floor(spread) + 1 + math.floor((p["T"] - 1) * ratio + 1 + 1) + 1
        assert p["W"] % 32 == 0 and p["W"] <= 1024 and last <= p["W"] - 1 and p["span"] < p["W"]
        assert p["smem"] <= 110 * 1024 and p["nth"] >= (p["T"] + 1) // 2 and p["nth"] in (64, 128, 256)


def test_scratch_is_bounded_by_the_records_of_a_batch(plan):
    """Source records and panel records take at most 256 MB each, save where the source records of 1024 panels alone
    take more; the records of the panels in hand are never more than those of all panels."""
    rng = np.random.default_rng(3)
    cases = [(98304, 64, 2048, 512, 1.0, 20.0), (98304, 3, 100000, 16, 1.0, 0.0), (2000000, 3, 64, 8, 1.0, 0.0)]
    cases += [(int(2 ** rng.uniform(0, 21)), int(2 ** rng.uniform(1.6, 20)), int(2 ** rng.uniform(0, 18)),
               int(2 ** rng.uniform(0, 12)), rng.uniform(0, 2), rng.uniform(0, 300)) for _ in range(4000)]
    for npts, N, nobs, nt, ratio, spread in cases:
        p = plan(npts, N, nobs, nt, ratio, spread * (nobs > 1))
        assert p["b_src"] <= min(32 * npts * N, max(256 << 20, 32 * 1024 * N)), (npts, N, nobs)
        assert p["b_rec"] <= max(256 << 20, 32 * nobs), (npts, N, nobs)
        assert p["b_part"] <= 8 * nobs * nt * 1217


def test_the_default_batch_keeps_its_panels(plan):
    """Up to as many microphones as frames the batch is set by the source records alone."""
    assert plan(98304, 1024, 64, 512, 1.0, 90)["NB"] == 8192
