"""The F-engine's multi-frame passes at the edges of their splits: every transform
length, frame counts that leave part of a batch (2, 4 or 16 frames), antenna groups
that leave part of a group, one tap and many, rows of any alignment, with and
without gains, both output types.

Bars: the FP32 outputs within 1e-5 relative Frobenius error of the CPU FP64 oracle (the
F-engine's bar); the int8 codes equal to the quantised FP32 outputs bit for bit."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_0909_0001_gb300 import omni

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [4, 8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("N, T, P, extra, gains", [(1, 1, 1, 0, False), (5, 3, 2, 1, True), (33, 18, 5, 2, False),
                                                   (67, 5, 12, 4, True)])
def test_fengine_lengths_and_edges(F, N, T, P, extra, gains):
    if F >= 1024:
        N = min(N, 9)
    rng = np.random.default_rng(F + N)
    raw = rng.integers(-128, 128, size=(N, (T + P - 1) * 2 * F + extra)).astype(np.int8)
    T = (raw.shape[1] - (P - 1) * 2 * F) // (2 * F)
    w = rng.standard_normal(P * 2 * F).astype(np.float32)
    g = (rng.standard_normal((F, N)) + 1j * rng.standard_normal((F, N))).astype(np.complex64) if gains else None
    scale = 0.3 / np.sqrt(P * F)
    kw = dict(window=torch.from_numpy(w), gains=None if g is None else torch.from_numpy(g), scale=scale)
    y = omni.fengine(torch.from_numpy(raw).cuda(), F, P, dtype="cf32", **kw).cpu().numpy()
    q = omni.fengine(torch.from_numpy(raw).cuda(), F, P, dtype="ci8", **kw).cpu().numpy()
    ref = oracle.fengine(raw, F, P, window=w.astype(np.float64), gains=None if g is None else g.astype(np.complex128),
                         scale=float(np.float32(scale)))
    assert y.shape == (F, T, N, 2) == q.shape
    assert np.linalg.norm(y[..., 0] + 1j * y[..., 1] - ref) <= 1e-5 * np.linalg.norm(ref)
    np.testing.assert_array_equal(q, oracle.quantize(y))


def test_fengine_64_channels_even_and_odd_frames():
    """The 64-channel pass: a last pair with one frame, two CTAs of frames, a ragged
    antenna group with unaligned output rows, no window."""
    rng = np.random.default_rng(11)
    for N, T, P in ((32, 16, 4), (35, 17, 3), (8, 33, 8), (70, 2, 1)):
        raw = rng.integers(-128, 128, size=(N, (T + P - 1) * 128)).astype(np.int8)
        y = omni.fengine(torch.from_numpy(raw).cuda(), 64, P, scale=0.05, dtype="cf32").cpu().numpy()
        q = omni.fengine(torch.from_numpy(raw).cuda(), 64, P, scale=0.05, dtype="ci8").cpu().numpy()
        ref = oracle.fengine(raw, 64, P, scale=float(np.float32(0.05)))
        assert np.linalg.norm(y[..., 0] + 1j * y[..., 1] - ref) <= 1e-5 * np.linalg.norm(ref)
        np.testing.assert_array_equal(q, oracle.quantize(y))
