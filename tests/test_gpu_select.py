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
    (5_100_001, 3, 0.01, 1e-3),    # bulk pass: 51,000 sent within 0.1% (the deep pipeline)
    (5_100_001, 6, 0.005, 1e-2),   # and the one-tile pipeline
    (5_100_001, 2, 0.005, 3e-5),   # narrower than the sampled threshold's own step of 2^10 keys
    (1_300_001, 20, 0.012, 1e-3),  # load/store pass
    (400_003, 20, 0.05, 1e-3),
])
def test_crowded_candidates_stay_on_the_fast_path(d, K, ratio, width):
    rng = np.random.default_rng(d + K)
    p = Pair(d, K, 0.9, 0.05, ratio=ratio, seed=3)
    for t in range(3):
        g = (rng.standard_normal((K, d)) * 0.05).astype(np.float32)
        crowd = rng.random((K, d)) < 2.5 * ratio  # more values in the band than the sampled threshold lets through
        band = (1.0 + width * rng.random((K, d))) * np.where(rng.random((K, d)) < 0.5, -1.0, 1.0)
        g = np.where(crowd, band * (2.0 ** t), g).astype(np.float32)
        p.compare(p.step(g), workers=[0, K - 1])
    assert p.compare_stats()["fallbacks"] == 0


def test_candidates_of_one_layer_do_not_overflow_the_bulk_parts():
    """A layer of 1/64 of the coordinates that holds every sent value: few tiles,
    so few CTAs' parts take all the candidates."""
    d, K = 5_100_001, 2
    rng = np.random.default_rng(1)
    p = Pair(d, K, 0.9, 0.05, ratio=0.01, seed=3)
    for t in range(2):
        g = (rng.standard_normal((K, d)) * 1e-3).astype(np.float32)
        g[:, 2_000_000:2_080_000] *= 1e3
        p.compare(p.step(g))
    assert p.compare_stats()["fallbacks"] == 0


@pytest.mark.parametrize("ratio,most", [(1.0, 0.6e9), (0.1, 0.25e9), (0.01, 0.2e9)])
def test_candidate_memory_at_large_ratios(ratio, most):
    """Bulk pass, d = 5.1 M, K = 2: e, w and the like take 0.12 GB; the candidates'
    parts at most twice the expected candidates, or what one layer can bring."""
    import torch
    from paper_1905_12948_gb300 import GMC
    GMC(5_100_001, 2, 0.9, 0.1, compressor="topk", ratio=0.001).close()  # the library's kernels are loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = GMC(5_100_001, 2, 0.9, 0.1, compressor="topk", ratio=ratio)
    used = before - torch.cuda.mem_get_info()[0]
    h.close()
    assert used <= most, f"{used / 1e9:.2f} GB"
