"""Selection where the candidates' keys crowd: residuals of a long run pile up
just below the level at which they are sent, so that all the sent values lie
within a narrow band above the k-th. The candidates' relative histogram has to
follow them (no worker may fall back to the dense select), and the selection
stays exact. Bit for bit against the oracle."""
import numpy as np
import pytest

from parity_util import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,ratio,width", [
    (1_300_001, 3, 0.02, 1e-3),    # bulk pass: 26,000 sent within 0.1% (the deep pipeline)
    (1_300_001, 6, 0.02, 1e-2),    # and the one-tile pipeline
    (1_300_001, 2, 0.02, 3e-5),    # narrower than the sampled threshold's own step of 2^10 keys
    (1_300_001, 20, 0.012, 1e-3),  # more workers
    (400_003, 20, 0.05, 1e-3),     # load/store pass
])
def test_crowded_candidates_stay_on_the_fast_path(d, K, ratio, width):
    rng = np.random.default_rng(d + K)
    p = Pair(d, K, 0.9, 0.05, ratio=ratio, seed=3)
    for t in range(3):
        g = (rng.standard_normal((K, d)) * 0.05).astype(np.float32)
        crowd = rng.random((K, d)) < 1.5 * ratio  # more values in the band than are sent
        band = (1.0 + width * rng.random((K, d))) * np.where(rng.random((K, d)) < 0.5, -1.0, 1.0)
        g = np.where(crowd, band * (2.0 ** t), g).astype(np.float32)
        p.compare(p.step(g), workers=[0, K - 1])
    assert p.compare_stats()["fallbacks"] == 0
