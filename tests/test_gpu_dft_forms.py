"""Axes whose length is no power of two in both forms of their passes: the tiles of lines
in shared memory, which take passes of several million terms (padded lines forward, whole
lines inverse, unpadded beam axes of odd and even length; contiguous and strided axes;
first, middle and last passes), and the thread per output that takes smaller ones.  Against
the CPU FP64 oracle, the sums of several calls included.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar."""
import numpy as np
import pytest

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


def err(V, ref):
    V, ref = V.reshape(V.shape[0], -1), ref.reshape(ref.shape[0], -1)
    return float((np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)).max())


def levels_of(shape):
    return synth.hierarchy(shape, [0.2 + 0.3 * k for k in range(len(shape))], [0.1 * k for k in range(len(shape))])


# forward MID and both inverse passes of 4 and 8 million terms, per tile axis
@pytest.mark.parametrize("n1, n2, nt, C, T", [(3, 1, 130, 18, 110), (5, 1, 100, 12, 90), (1, 7, 90, 9, 60), (13, 1, 40, 9, 40),
                                              (30, 1, 24, 5, 24), (73, 1, 20, 2, 20), (96, 1, 17, 2, 15),
                                              (5, 7, 33, 7, 60), (12, 9, 24, 3, 24), (11, 3, 41, 4, 75)])
def test_tile_axes_match_oracle(n1, n2, nt, C, T):
    x = synth.random_complex([n1, n2, nt], C, T, seed=1200 + n1)
    offs = np.random.default_rng(nt).uniform(-4000.0, 4000.0, size=(nt, 2))
    with omni.TilePlan(synth.Level(n1, n2), offs, C) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy().reshape(C, -1)
    assert err(V, oracle.tile_correlate(n1, n2, nt, x).reshape(C, -1)) <= 1e-5


# LAST passes of 3 million terms and more (the first call) and of fewer (the second)
@pytest.mark.parametrize("shape, C, T", [([(2, 3)], 150, 400), ([(2, 12)], 28, 110), ([(4, 13)], 20, 60), ([(8, 7)], 40, 55),
                                         ([(16, 33)], 3, 17), ([(2, 73)], 4, 20), ([(2, 96)], 3, 17), ([(3, 95)], 5, 6)])
@pytest.mark.parametrize("dtype", ["cf32", "ci8"])
def test_last_axes_match_oracle(shape, C, T, dtype):
    levels = levels_of(shape)
    dims = synth.lattice_dims(levels)
    x = synth.random_complex(dims, C, T, seed=1300 + T, dtype=dtype, sigma=30.0 if dtype == "ci8" else 1.0)
    short = x[:, : max(1, T // 7)].contiguous()
    with omni.Plan(levels, C, dtype=dtype) as plan:
        plan.correlate(x.cuda())
        plan.correlate(short.cuda())
        V = plan.visibilities().cpu().numpy()
    assert err(V, oracle.correlate(dims, x) + oracle.correlate(dims, short)) <= 1e-5


@pytest.mark.parametrize("block", [(11, 9), (10, 6)])
def test_unpadded_axes_match_oracle(block):
    levels = levels_of([block, (6, 6)])
    x = synth.random_complex(synth.lattice_dims(levels), 6, 40, seed=1400)
    with omni.BeamPlan(levels, 6) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy()
    assert err(V, oracle.beam_correlate(synth.lattice_dims(levels), x)) <= 1e-5
