"""RBGS block choice decided draw by draw in parallel, and the detached rows
written by the step's own pass: edges of both, bit for bit against the oracle."""
import numpy as np
import pytest

from parity_util import Pair, assert_fp32_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,B,ratio,per_worker", [
    (100, 100, 1.0, False),        # one block
    (5_000, 1, 1.0, True),         # every block: each draw after the first few collides
    (40_003, 2, 0.9, False),       # long chains; first-draw table in global memory
    (16_384, 1, 0.5, True),        # the largest table in shared memory
    (500_003, 1, 0.3, False),      # bitmap in global memory, flags cleared by a memset
    (70_000, 1, 0.02, True),       # more blocks than one warp clears flags of
])
def test_pick(d, B, ratio, per_worker):
    K = 2
    rng = np.random.default_rng(d)
    p = Pair(d, K, 0.9, 0.1, compressor="rbgs", ratio=ratio, block=B, lam=0.5, seed=5, per_worker=per_worker)
    for t in range(3):
        p.compare(p.step(rng.standard_normal((K, d)).astype(np.float32)))
    p.compare_stats()


@pytest.mark.parametrize("d,K,B,ratio,per_worker", [
    (1_024, 2, 1, 1.0, False), (1_025, 2, 1, 1.0, False),       # the most draws a step makes itself, one more
    (10_600, 1, 1, 0.05, False), (10_601, 1, 1, 0.05, False),   # its largest table, one more
    (6_174, 12, 7, 0.09, True), (6_181, 12, 7, 0.09, True),     # the same with a stream per worker
    (130, 12, 1, 0.1, True), (130, 13, 1, 0.1, True), (129, 32, 1, 0.1, False),  # the most streams
    (590_000, 17, 4096, 0.05, False), (590_000, 18, 4096, 0.05, False),          # the most values
    (272_474, 8, 256, 0.05, True), (33, 3, 1, 0.04, True),
])
def test_choice_within_the_step(d, K, B, ratio, per_worker):
    rng = np.random.default_rng(d)
    p = Pair(d, K, 0.9, 0.1, compressor="rbgs", ratio=ratio, block=B, lam=0.5, seed=6, per_worker=per_worker)
    for t in range(3):
        p.compare(p.step(rng.standard_normal((K, d)).astype(np.float32)))
    p.compare_stats()


def test_choice_within_and_before_the_step_in_turn():
    """One handle whose shared choice is made in the step and whose per-worker
    choice (too many draws) by a kernel of its own."""
    d, K = 9_000, 4
    rng = np.random.default_rng(77)
    p = Pair(d, K, 0.9, 0.1, compressor="rbgs", ratio=0.5, block=10, lam=0.5, seed=7)
    for t in range(6):
        assert p.gpu.lib.gmc_set_rbgs_mode(p.gpu.h, t & 1) == 0
        p.ref.per_worker = bool(t & 1)
        p.compare(p.step(rng.standard_normal((K, d)).astype(np.float32)))
    p.compare_stats()


@pytest.mark.parametrize("d,K,B,offset,pad", [
    (127, 1, 10, 0, 0), (128, 5, 128, 1, 1), (1_025, 9, 100, 2, 3), (50_001, 32, 333, 3, 0),  # load/store pass
    (4096 * 160 + 130, 3, 1000, 1, 2), (4096 * 152 + 4095, 2, 4096, 3, 1),                     # bulk pass
])
@pytest.mark.parametrize("per_worker", [False, True])
@pytest.mark.parametrize("bf16", [False, True])
def test_detached_rows_at_any_alignment(d, K, B, offset, pad, per_worker, bf16):
    import torch
    rng = np.random.default_rng(d + K)
    p = Pair(d, K, 0.9, 0.1, compressor="rbgs", ratio=0.2, block=B, lam=0.5, seed=8, per_worker=per_worker)
    ld = d + pad
    buf = torch.full((offset + K * ld + 4,), 7.0, dtype=torch.float32, device=p.dev)
    lib, h = p.gpu.lib, p.gpu.h
    assert lib.gmc_set_detach_output(h, buf.data_ptr() + 4 * offset, ld) == 0
    for t in range(2):
        g = torch.from_numpy(rng.standard_normal((K, d)).astype(np.float32))
        if bf16:
            g = g.to(torch.bfloat16)
        p.step(g.float().numpy(), g.to(p.dev))
    host = buf.cpu().numpy()
    rows = host[offset: offset + K * ld].reshape(K, ld)
    for k in range(K):
        assert_fp32_state(rows[k, :d], p.ref.worker_params(k), f"detached row {k}")
        assert_fp32_state(p.gpu.worker_params(k).cpu().numpy(), p.ref.worker_params(k), "gmc_get_worker_params")
    assert (rows[:, d:] == 7.0).all() and (host[:offset] == 7.0).all() and (host[offset + K * ld:] == 7.0).all()
