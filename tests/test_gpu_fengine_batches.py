"""The F-engine's passes when a CTA runs many frames: the 64-channel pass with runs of 4, 8
and 16 frames per CTA (the runs shrink while the GPU is not filled; the last run is
ragged and odd), the passes of 16 to 256 channels on more points than fill the GPU (fewer
take the 16-antenna pass), and several batches of frames per CTA.

Bars: the FP32 outputs within 1e-5 relative Frobenius error of the CPU FP64 oracle (the
F-engine's bar) on a few antennas of every antenna group; the int8 codes of every
antenna equal to the quantised FP32 outputs bit for bit."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_0909_0001_gb300 import omni

pytestmark = pytest.mark.gpu


def check(F, N, T, P, extra, gains, antennas):
    rng = np.random.default_rng(F + N + T)
    raw = rng.integers(-128, 128, size=(N, (T + P - 1) * 2 * F + extra)).astype(np.int8)
    w = rng.standard_normal(P * 2 * F).astype(np.float32)
    g = (rng.standard_normal((F, N)) + 1j * rng.standard_normal((F, N))).astype(np.complex64) if gains else None
    scale = 0.3 / np.sqrt(P * F)
    kw = dict(window=torch.from_numpy(w), gains=None if g is None else torch.from_numpy(g), scale=scale)
    dev = torch.from_numpy(raw).cuda()
    y = omni.fengine(dev, F, P, dtype="cf32", **kw).cpu().numpy()
    q = omni.fengine(dev, F, P, dtype="ci8", **kw).cpu().numpy()
    assert y.shape == (F, T, N, 2) == q.shape
    np.testing.assert_array_equal(q, oracle.quantize(y))
    sel = np.unique(np.array(antennas) % N)
    ref = oracle.fengine(raw[sel], F, P, window=w.astype(np.float64),
                         gains=None if g is None else g[:, sel].astype(np.complex128), scale=float(np.float32(scale)))
    v = y[:, :, sel, 0] + 1j * y[:, :, sel, 1]
    # frame by frame: a wrong frame would be a small part of a long run's norm
    err = np.linalg.norm(v - ref, axis=(0, 2)) / np.linalg.norm(ref, axis=(0, 2))
    assert err.max() <= 1e-5


@pytest.mark.parametrize("P, gains", [(1, False), (3, True), (4, False), (8, True)])
@pytest.mark.parametrize("N, T", [(300, 70), (600, 71), (1201, 67)])  # runs of 4, 8 and 16 frames
def test_64_channel_frame_runs(N, T, P, gains):
    check(64, N, T, P, 0, gains, list(range(0, N, 37)) + [N - 1])


@pytest.mark.parametrize("N, T, P, gains", [(8, 2101, 1, False), (3, 2099, 4, True), (20, 1303, 8, False), (28, 2500, 3, True),
                                            (40, 1301, 4, False)])
def test_64_channels_of_a_few_antennas(N, T, P, gains):
    check(64, N, T, P, 0, gains, [0, N // 2, N - 1])


@pytest.mark.parametrize("F, N, T, P, extra, gains", [(16, 300, 261, 4, 0, False), (16, 260, 301, 1, 3, True),
                                                      (32, 200, 197, 5, 1, True), (64, 150, 131, 4, 2, False),
                                                      (128, 70, 141, 3, 0, True), (256, 35, 141, 4, 2, True),
                                                      (256, 17, 301, 12, 0, False)])
def test_16_to_256_channels_on_a_filled_gpu(F, N, T, P, extra, gains):
    check(F, N, T, P, extra, gains, list(range(0, N, 13)) + [N - 1])


@pytest.mark.parametrize("F, N, T, P, gains", [(16, 300, 1625, 3, True), (128, 70, 1629, 2, False),
                                               (512, 100, 401, 4, True), (1024, 39, 489, 1, False)])
def test_several_batches_per_cta(F, N, T, P, gains):
    check(F, N, T, P, 0, gains, [0, N // 2, N - 1])


@pytest.mark.parametrize("F, N, T, P, extra, gains", [(512, 20, 101, 5, 3, True), (1024, 9, 103, 2, 0, False),
                                                      (2048, 5, 103, 1, 1, True), (512, 20, 30, 3, 0, False),
                                                      (512, 13, 23, 5, 3, True), (1024, 5, 33, 3, 0, True),  # a quarter
                                                      (2048, 3, 7, 12, 2, False)])                           # each
def test_512_channels_and_more(F, N, T, P, extra, gains):
    check(F, N, T, P, extra, gains, [0, 1, N - 1])
