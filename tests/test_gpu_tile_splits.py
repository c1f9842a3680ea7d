"""The FP32 cross-spectrum kernel's three ways to split the tile pairs: the grid that
fills the GPU (up to 64 tiles in one CTA; 24 x 32 rectangles beyond), and the rectangles
of 2 x 2 groups of 8 tiles and the single pairs of groups that few channels take; and
tiles of one antenna, whose stages are not tensor-map boxes.  Tile counts at the edges of
groups and rectangles, full and part stages, against the CPU FP64 oracle.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar."""
import numpy as np
import pytest

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1, n2, nt, C, T", [
    (4, 4, 64, 26, 29), (2, 4, 72, 20, 29), (4, 4, 89, 9, 7), (2, 2, 17, 152, 9), (4, 4, 41, 26, 6),  # a CTA per SM
    (3, 5, 9, 1, 66), (2, 2, 8, 1, 1),                                                                # few warps
    (2, 4, 57, 8, 13), (4, 2, 90, 4, 21), (2, 2, 66, 9, 5), (4, 4, 64, 1, 33), (1, 2, 130, 1, 10),    # 2 x 2 groups
    (2, 2, 64, 16, 30), (8, 8, 64, 2, 9),                                                             # single pairs
    (1, 1, 1, 3, 40), (1, 1, 8, 1, 1), (1, 1, 9, 2, 5), (1, 1, 64, 4, 1030), (1, 1, 65, 3, 31), (1, 1, 200, 2, 17),
    (1, 1, 60, 60, 14), (1, 1, 100, 20, 21)])
def test_splits_match_oracle(n1, n2, nt, C, T):
    x = synth.random_complex([n1, n2, nt], C, T, seed=1000 + nt + C)
    offs = np.random.default_rng(nt).uniform(-900.0, 900.0, size=(nt, 2))
    with omni.TilePlan(synth.Level(n1, n2, (1.0, 0.3, 0.0, 1.0)), offs, C) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().reshape(C, -1).cpu().numpy()
    ref = oracle.tile_correlate(n1, n2, nt, x).reshape(C, -1)
    assert (np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() <= 1e-5


@pytest.mark.parametrize("n1, n2, nt, C", [(4, 4, 64, 26), (3, 5, 9, 1), (2, 4, 57, 8), (2, 2, 64, 16), (1, 1, 65, 3)])
def test_calls_add_up(n1, n2, nt, C):
    """Each split folds into the sums of the calls before."""
    x = synth.random_complex([n1, n2, nt], C, 9, seed=1100 + nt)
    offs = np.random.default_rng(nt).uniform(-900.0, 900.0, size=(nt, 2))
    with omni.TilePlan(synth.Level(n1, n2, (1.0, 0.3, 0.0, 1.0)), offs, C) as plan:
        plan.correlate(x[:, :5].contiguous().cuda())
        plan.correlate(x[:, 5:].contiguous().cuda())
        V = plan.visibilities().reshape(C, -1).cpu().numpy()
    ref = oracle.tile_correlate(n1, n2, nt, x).reshape(C, -1)
    assert (np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() <= 1e-5
