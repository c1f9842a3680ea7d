"""LAST passes of axes beyond the tiled DFT forms (one thread per output): whole and in
slices of the samples, with terms that leave part of a group of four, onto the sums of an
earlier call, against the CPU FP64 oracle.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar."""
import numpy as np
import pytest

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1, n2, C, T", [(4, 100, 1, 70), (4, 100, 9, 3), (3, 150, 2, 20), (1, 250, 3, 40), (2, 131, 1, 33),
                                          (8, 98, 60, 2)])
@pytest.mark.parametrize("dtype", ["cf32", "ci8"])
def test_longer_axes_match_oracle(n1, n2, C, T, dtype):
    levels = [synth.Level(n1, n2, (1.0, 0.2, 0.1, 1.0))]
    x = synth.random_complex([n1, n2], C, T, seed=1500 + T, dtype=dtype, sigma=30.0 if dtype == "ci8" else 1.0)
    with omni.Plan(levels, C, dtype=dtype) as plan:
        plan.correlate(x.cuda())
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy()
    ref = 2 * oracle.correlate([n1, n2], x)
    assert (np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() <= 1e-5
