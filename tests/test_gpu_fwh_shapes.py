"""The staged observer pass at the sizes where its tiling can go wrong: microphone groups that are short, odd or
uneven, observer times around the block sizes, sparse and dense times, several panel batches, against the oracle."""
import numpy as np
import pytest

from oracle import fwh
from paper_2212_12365_gb300 import les
from test_gpu_fwh import C0, P0, RHO0, _frames, _ring, _sphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,mics,nt,ratio", [
    (les.LES_FP32, 1, 1, 1.0), (les.LES_FP32, 2, 63, 1.0), (les.LES_FP64, 15, 129, 0.37), (les.LES_FP32, 17, 257, 0.9),
    (les.LES_FP32, 33, 40, 1.0), (les.LES_FP32, 5, 513, 0.5), (les.LES_FP64, 16, 300, 1.0), (les.LES_FP32, 3, 64, 4.5)])
def test_shapes(prec, mics, nt, ratio):
    import torch
    xyz, nrm, area = _sphere(1.0, 11, 23)
    dtau, nfr = 0.02, 900
    frames = _frames(xyz, nfr, dtau)
    ring = _ring(frames, nfr, torch.float64 if prec == les.LES_FP64 else torch.float32)
    a = np.linspace(0.2, 2.6, mics)
    obs = np.stack([5.0 * np.cos(a), 5.0 * np.sin(a), 0.3 * np.arange(mics) % 1.0])
    t0, dt_obs = 7.9, ratio * dtau
    used = frames.astype(np.float32).astype(np.float64) if prec == les.LES_FP32 else frames
    got = les.les_fwh(ring.data_ptr(), prec, nfr, nfr, xyz, nrm, area, dtau, P0, C0, obs, t0, dt_obs, nt)
    ref = fwh.pressure(used, xyz, nrm, area, dtau, RHO0, P0, C0, obs, t0, dt_obs, nt)
    # FP32 records and products: the bound of the other far-field tests
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()


def test_batches_and_wrapped_ring():
    """More panels than one batch takes (1024 at this frame count), a ring that has wrapped."""
    import torch
    xyz, nrm, area = _sphere(1.0, 30, 71)
    # a long ring of which the last frames matter: 256 MB / (32 bytes x frames) < 1024 panels
    dtau, nfr, cap = 0.001, 8800, 8300
    frames = _frames(xyz, nfr, dtau).astype(np.float32)
    ring = _ring(frames, cap, torch.float32)
    used = frames[nfr - cap:].astype(np.float64)
    obs = np.array([[2.5, 0.3, 0.1], [-1.5, 1.9, 0.4]]).T
    t0, dt_obs, nt = 4.6, 0.0013, 200
    got = les.les_fwh(ring.data_ptr(), les.LES_FP32, cap, nfr, xyz, nrm, area, dtau, P0, C0, obs, t0, dt_obs, nt)
    ref = fwh.pressure(used, xyz, nrm, area, dtau, RHO0, P0, C0, obs, t0, dt_obs, nt)
    # the frames' FP32 rounding (6e-8 of p0) over 2 dtau is noise that both see alike; what differs is FP32 products
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()
