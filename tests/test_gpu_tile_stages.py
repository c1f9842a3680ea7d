"""The FP32 cross-spectrum kernel over many stages: its ring of three four-sample stages
is filled again behind the loads that read it, so a box that landed too early would
replace samples of some pairs.  Both splits (every tile in one CTA; 24 x 32 rectangles),
full and part stages, one and several CTAs per channel, against the CPU FP64 oracle.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar (one sample of 97
replaced is an error of about 0.1)."""
import numpy as np
import pytest

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1, n2, nt, T", [(4, 4, 64, 97), (4, 4, 33, 64), (2, 4, 72, 50), (2, 2, 130, 97)])
def test_stage_ring_matches_oracle(n1, n2, nt, T):
    x = synth.random_complex([n1, n2, nt], 3, T, seed=900 + nt)
    offs = np.random.default_rng(nt).uniform(-400.0, 400.0, size=(nt, 2))
    with omni.TilePlan(synth.Level(n1, n2, (1.0, 0.3, 0.0, 1.0)), offs, 3) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().reshape(3, -1).cpu().numpy()
    ref = oracle.tile_correlate(n1, n2, nt, x).reshape(3, -1)
    assert (np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() <= 1e-5
