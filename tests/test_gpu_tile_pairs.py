"""The FP32 cross-spectrum kernel of the tile hybrid at the edges of its splits
(groups of 8 tiles; up to 64 tiles one CTA reads them all, beyond in 24 x 32
rectangles; 32 frequencies; 4 samples a stage) against the CPU FP64 oracle.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar."""
import numpy as np
import pytest

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


def run(n1, n2, nt, x):
    offs = np.random.default_rng(nt).uniform(-400.0, 400.0, size=(nt, 2))
    with omni.TilePlan(synth.Level(n1, n2, (1.0, 0.3, 0.0, 1.0)), offs, x.shape[0]) as plan:
        plan.correlate(x.cuda())
        return plan.visibilities().reshape(x.shape[0], -1).cpu().numpy()


@pytest.mark.parametrize("n1, n2, nt, T", [(2, 2, 8, 4), (3, 2, 9, 7), (8, 8, 40, 13), (4, 4, 63, 5), (8, 8, 64, 12),
                                           (4, 2, 65, 9), (2, 3, 130, 6), (1, 1, 70, 5), (16, 16, 16, 1)])
def test_tile_pairs_match_oracle(n1, n2, nt, T):
    x = synth.random_complex([n1, n2, nt], 2, T, seed=600 + nt)
    V = run(n1, n2, nt, x)
    ref = oracle.tile_correlate(n1, n2, nt, x).reshape(2, -1)
    err = np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= 1e-5


def test_expired_wait_is_reported(monkeypatch):
    """The test hook makes every CTA's first wait run out (~0.5 ms): the host reports
    OMNI_ERR_TIMEOUT and the next plan on the same context is correct."""
    x = synth.random_complex([4, 4, 20], 1, 21, seed=700)
    monkeypatch.setenv("OMNI_TEST_FORCE_TIMEOUT", "1")
    with pytest.raises(omni.OmniError) as e:
        run(4, 4, 20, x)
    assert e.value.status == 6
    monkeypatch.delenv("OMNI_TEST_FORCE_TIMEOUT")
    ref = oracle.tile_correlate(4, 4, 20, x).reshape(1, -1)
    assert np.linalg.norm(run(4, 4, 20, x) - ref) <= 1e-5 * np.linalg.norm(ref)
