"""Unpadded square levels (beam pointings) in one pass, and contiguous axes read and
written in runs, against the CPU FP64 oracle: every square size of the one-pass kernel
and its neighbours, block counts that leave part of a CTA, voltages off the vector
loads' alignment.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1, n2, outer", [(2, 2, (2, 3)), (4, 4, (3, 3)), (8, 8, (3, 2)), (16, 16, (2, 2)), (32, 32, (2, 1)),
                                           (64, 64, (2, 1)), (16, 8, (2, 2))])
@pytest.mark.parametrize("dtype, shift", [("cf32", 0), ("ci8", 0), ("ci8", 1)])
def test_beam_blocks_match_oracle(n1, n2, outer, dtype, shift):
    levels = synth.hierarchy([(n1, n2), outer], [0.1, 0.4], [0.0, 0.1])
    dims = synth.lattice_dims(levels)
    x = synth.random_complex(dims, 2, 3, seed=900 + n1, dtype=dtype, sigma=30.0 if dtype == "ci8" else 1.0)
    xd = x.cuda()
    if shift:  # the same values one complex int8 (2 bytes) further on
        flat = torch.zeros(xd.numel() + 2, dtype=xd.dtype, device="cuda")
        flat[2:] = xd.reshape(-1)
        xd = flat[2:].view(xd.shape)
    with omni.BeamPlan(levels, 2, dtype=dtype) as plan:
        plan.correlate(xd)
        V = plan.visibilities().reshape(2, -1).cpu().numpy()
    ref = oracle.beam_correlate(dims, x).reshape(2, -1)
    assert (np.linalg.norm(V - ref, axis=1) <= 1e-5 * np.linalg.norm(ref, axis=1)).all()


@pytest.mark.parametrize("n1, n2", [(2, 70), (4, 33), (8, 3), (16, 9), (32, 5), (5, 129)])
def test_contiguous_axes_match_oracle(n1, n2):
    levels = [synth.Level(n1, n2, (1.0, 0.2, 0.0, 1.0))]
    x = synth.random_complex([n1, n2], 3, 4, seed=950 + n1)
    with omni.Plan(levels, 3) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy()
    ref = oracle.correlate([n1, n2], x)
    assert (np.linalg.norm(V - ref, axis=1) <= 1e-5 * np.linalg.norm(ref, axis=1)).all()
