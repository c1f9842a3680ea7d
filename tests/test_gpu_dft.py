"""Axes whose length is no power of two: the tiled DFT passes (padded, whole and
unpadded lines; odd and even n; contiguous and strided axes; first, middle and last
passes; several bin groups) and the lengths beyond them, against the CPU FP64 oracle.

Bars: 1e-5 relative Frobenius error per channel (FP32 paths), 1e-4 (mixed)."""
import numpy as np
import pytest

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


def levels_of(shape):
    return synth.hierarchy(shape, [0.2 + 0.3 * k for k in range(len(shape))], [0.1 * k for k in range(len(shape))])


def err(V, ref):
    return float((np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)).max())


@pytest.mark.parametrize("shape, T", [([(3, 1)], 3), ([(1, 5)], 2), ([(5, 7)], 9), ([(6, 6)], 5), ([(14, 3)], 4),
                                      ([(30, 31)], 3), ([(33, 2)], 3), ([(95, 3)], 3), ([(3, 96)], 2), ([(2, 97)], 2),
                                      ([(120, 2)], 2), ([(3, 5), (7, 2)], 4), ([(8, 8), (5, 6)], 3),
                                      ([(3, 3), (3, 2), (2, 3)], 6)])
@pytest.mark.parametrize("dtype", ["cf32", "ci8"])
def test_odd_axes_match_oracle(shape, T, dtype):
    levels = levels_of(shape)
    x = synth.random_complex(synth.lattice_dims(levels), 3, T, seed=40 + T, dtype=dtype,
                             sigma=30.0 if dtype == "ci8" else 1.0)
    with omni.Plan(levels, 3, dtype=dtype) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy()
    assert err(V, oracle.correlate(synth.lattice_dims(levels), x)) <= 1e-5


@pytest.mark.parametrize("shape", [[(5, 3), (4, 4)], [(2, 6), (3, 2)], [(9, 9), (2, 5)], [(1, 7), (3, 3)]])
def test_odd_beam_axes_match_oracle(shape):
    levels = levels_of(shape)
    x = synth.random_complex(synth.lattice_dims(levels), 2, 5, seed=60)
    with omni.BeamPlan(levels, 2) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().reshape(2, -1).cpu().numpy()
    ref = oracle.beam_correlate(synth.lattice_dims(levels), x).reshape(2, -1)
    assert err(V, ref) <= 1e-5


@pytest.mark.parametrize("n1, n2, nt, precision", [(12, 12, 9, "mixed"), (6, 10, 17, "fp32"), (3, 5, 70, "fp32")])
def test_odd_tiles_match_oracle(n1, n2, nt, precision):
    x = synth.random_complex([n1, n2, nt], 2, 20, seed=61)
    offs = np.random.default_rng(nt).uniform(-400.0, 400.0, size=(nt, 2))
    with omni.TilePlan(synth.Level(n1, n2), offs, 2, precision=precision) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().reshape(2, -1).cpu().numpy()
    assert err(V, oracle.tile_correlate(n1, n2, nt, x).reshape(2, -1)) <= (1e-5 if precision == "fp32" else 1e-4)
