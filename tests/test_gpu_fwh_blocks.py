"""The staged observer pass where a group's emission times spread over hundreds of frames, at the edges of what a
window holds: short groups with a buffer row per microphone, blocks of 512 and of 256 times, full groups, and windows
that leave the direct pass; against the oracle."""
import numpy as np
import pytest

from oracle import fwh
from paper_2212_12365_gb300 import les
from test_gpu_fwh import AMP, C0, P0, RHO0, SRC, _ring, _sphere

pytestmark = pytest.mark.gpu
DTAU, NFR = 0.02, 1700


def _tone(xyz, w=2.5):
    """Frames of a steadily sounding point monopole, which every microphone hears at any time."""
    d = xyz - SRC[:, None]
    R = np.sqrt((d * d).sum(axis=0))
    tr = (DTAU * np.arange(NFR))[:, None] - R / C0
    q, qd = AMP * np.sin(w * tr), AMP * w * np.cos(w * tr)
    p = RHO0 * qd / (4 * np.pi * R)
    u = (qd / (4 * np.pi * C0 * R) + q / (4 * np.pi * R * R))[:, None, :] * (d / R)
    return np.concatenate([(RHO0 + p / C0 ** 2)[:, None], u, (P0 + p)[:, None]], axis=1)


@pytest.fixture(scope="module")
def data():
    import torch
    xyz, nrm, area = _sphere(1.0, 7, 13)
    frames = _tone(xyz).astype(np.float32)
    return xyz, nrm, area, frames.astype(np.float64), _ring(frames, NFR, torch.float32)


# (microphones, times, spread of a group in frames, dt_obs / dtau)
@pytest.mark.parametrize("mics,nt,spread,ratio", [
    (2, 512, 480, 1.0), (3, 512, 640, 0.5), (7, 300, 640, 1.0), (8, 512, 470, 1.0), (9, 513, 380, 1.0),
    (12, 512, 300, 1.0), (14, 512, 150, 1.0), (16, 512, 170, 1.0), (16, 512, 110, 1.0), (16, 257, 360, 1.0),
    (16, 40, 560, 1.0), (16, 40, 700, 1.0), (32, 300, 200, 1.0), (40, 512, 260, 1.0)])
def test_spread_groups(data, mics, nt, spread, ratio):
    xyz, nrm, area, used, ring = data
    # microphones along a ray; those of a group 16 (or fewer) apart cover the spread
    far = 2.5 + C0 * DTAU * spread * np.arange(mics) / max(min(mics, 16) - 1, 1)
    far = 2.5 + (far - 2.5) % (C0 * DTAU * spread + 1e-9)
    obs = np.stack([0.8 * far, 0.5 * far, np.sqrt(1 - 0.89) * far])
    t0 = (far.max() + 1.0) / C0 + 0.01
    assert t0 + nt * ratio * DTAU - (far.min() - 1.0) / C0 < (NFR - 1) * DTAU
    got = les.les_fwh(ring.data_ptr(), les.LES_FP32, NFR, NFR, xyz, nrm, area, DTAU, P0, C0, obs, t0, ratio * DTAU, nt)
    ref = fwh.pressure(used, xyz, nrm, area, DTAU, RHO0, P0, C0, obs, t0, ratio * DTAU, nt)
    # FP32 records and products: the bound of the other far-field tests, per microphone (each has its own distance)
    scale = np.abs(ref).max(axis=1, keepdims=True)
    assert (np.abs(got - ref) <= 2e-5 * scale).all(), (np.abs(got - ref) / scale).max(axis=1)


def test_many_microphones_in_several_batches():
    """More (panel, microphone) records than one batch holds: the first microphones have the same pressure as in a
    call of their own."""
    import torch
    xyz, nrm, area = _sphere(1.0, 23, 61)  # 1403 panels x 8192 microphones x 32 bytes: two batches
    frames = _tone(xyz)[:300].astype(np.float32)
    ring = _ring(frames, 300, torch.float32)
    mics, nt = 8192, 5
    a = np.linspace(0.1, 3.0, mics)
    obs = np.stack([2.5 * np.cos(a), 2.5 * np.sin(a), 0.2 * np.sin(7 * a)])
    t0 = 3.6 / C0 + 0.01
    got = les.les_fwh(ring.data_ptr(), les.LES_FP32, 300, 300, xyz, nrm, area, DTAU, P0, C0, obs, t0, DTAU, nt)
    few = les.les_fwh(ring.data_ptr(), les.LES_FP32, 300, 300, xyz, nrm, area, DTAU, P0, C0, obs[:, :160], t0, DTAU, nt)
    ref = fwh.pressure(frames.astype(np.float64), xyz, nrm, area, DTAU, RHO0, P0, C0, obs[:, ::400], t0, DTAU, nt)
    scale = np.abs(ref).max()
    assert np.abs(got[::400] - ref).max() <= 2e-5 * scale
    assert np.abs(got[:160] - few).max() <= 2e-6 * scale


def _line(n_frames, panels=1):
    """A ring of a slow tone at a panel (or a few), made on the GPU, with a period of 400 frames."""
    import torch
    t = (torch.arange(n_frames, device="cuda") % 400).double() * (2 * np.pi / 400)
    ring = torch.empty((n_frames, 5, panels), dtype=torch.float32, device="cuda")
    for f, (mean, amp, ph) in enumerate(((RHO0, 1e-2, 0.0), (0.0, 2e-2, 0.4), (0.0, 1e-2, 1.1), (0.0, 0.0, 0.0), (P0, 1e-2, 2.0))):
        ring[:, f] = (mean + amp * torch.sin(t + ph)).float()[:, None]
    return ring


def _panel(panels=1):
    xyz = np.zeros((3, panels))
    xyz[0] = 0.01 * np.arange(panels)
    nrm = np.tile(np.array([[1.0], [0.0], [0.0]]), (1, panels))
    return xyz, nrm, np.full(panels, 0.3)


def test_more_frames_than_a_grid_has_rows():
    """4.2 million frames: the source pass covers them all (65,535 segments of 64 frames and more)."""
    n = 65535 * 64 + 1000
    xyz, nrm, area = _panel()
    ring = _line(n)
    obs = np.array([[3.0, 1.0, 0.5]]).T
    # the last 300 observer times that the frames cover; the tone repeats every 400 frames, so the same times of a
    # ring of 2000 frames (a whole number of periods earlier) give the same pressure
    shift = (n - 2000) // 400 * 400
    t_short = 1600 * DTAU
    args = (xyz, nrm, area, DTAU, P0, C0, obs)
    got = les.les_fwh(ring.data_ptr(), les.LES_FP32, n, n, *args, t_short + shift * DTAU, DTAU, 300)
    ref = les.les_fwh(ring.data_ptr(), les.LES_FP32, 2000, 2000, *args, t_short, DTAU, 300)
    assert np.abs(ref).max() > 0 and np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()


def test_more_time_blocks_than_a_grid_has_rows():
    """34 million observer times: more than 65,535 blocks of 512."""
    nt = 65535 * 512 + 700
    xyz, nrm, area = _panel(3)
    ring = _line(2000, 3)
    obs = np.array([[3.0, 1.0, 0.5]]).T
    t0, dt_obs = 5.0, 30.0 / nt
    args = (xyz, nrm, area, DTAU, P0, C0, obs)
    got = les.les_fwh(ring.data_ptr(), les.LES_FP32, 2000, 2000, *args, t0, dt_obs, nt)[0]
    ref = les.les_fwh(ring.data_ptr(), les.LES_FP32, 2000, 2000, *args, t0 + (nt - 500) * dt_obs, dt_obs, 500)[0]
    assert np.abs(got[-500:] - ref).max() <= 1e-5 * np.abs(ref).max()
    every = les.les_fwh(ring.data_ptr(), les.LES_FP32, 2000, 2000, *args, t0, dt_obs * 65536, nt // 65536)[0]
    assert np.abs(got[::65536][:every.size] - every).max() <= 1e-5 * np.abs(every).max()


def test_two_threads_with_windows_of_different_size():
    """Calls from two host threads whose staged passes need different amounts of shared memory."""
    import threading
    import torch
    xyz, nrm, area = _panel(64)
    ring = _line(2000, 64)
    obs = np.array([[3.0, 1.0, 0.5], [2.0, -1.0, 0.5]]).T
    torch.cuda.synchronize()
    errors = []

    def calls(ratio):
        try:
            st = torch.cuda.Stream()
            for _ in range(1500):
                les.les_fwh(ring.data_ptr(), les.LES_FP32, 2000, 2000, xyz, nrm, area, DTAU, P0, C0, obs, 6.0,
                            ratio * DTAU, 512, stream=st.cuda_stream)
        except Exception as e:  # noqa: BLE001 (handed to the test's thread)
            errors.append(e)

    th = [threading.Thread(target=calls, args=(r,)) for r in (0.05, 1.0)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not errors, errors
