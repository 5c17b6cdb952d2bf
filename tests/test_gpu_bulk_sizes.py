"""The bulk top-k pass (2 to 16 workers, d >= 8 * 4096 * SMs: about 5 M), and the
load/store pass (what lies between that and the one-launch step of small
problems: K x d up to about 7 M), under the tests that other files run at sizes
where the other passes take the step."""
import numpy as np
import pytest

import test_gpu_approx
import test_gpu_bf16
import test_gpu_checkpoint
import test_gpu_deferred
import test_gpu_failure
import test_gpu_parity
import test_gpu_variants
from parity_util import Pair

pytestmark = pytest.mark.gpu

D = 5_100_001
D_LS, K_LS = 1_300_001, 7  # load/store pass
D_LS1 = 8_000_001          # and with one worker


@pytest.mark.parametrize("d,K,want", [(D, 2, "bulk"), (D, 16, "bulk"), (D, 1, "one launch"), (D, 17, "load/store"),
                                      (D_LS, K_LS, "load/store"), (D_LS, 3, "one launch"), (D_LS1, 1, "load/store")])
@pytest.mark.parametrize("compressor", ["topk", "topk_approx"])
def test_routes(d, K, want, compressor):
    p = Pair(d, K, 0.9, 0.1, compressor=compressor, ratio=0.001)
    assert p.route() == want


@pytest.mark.parametrize("name", ["test_deferred_steps_in_a_row_with_eta_schedule",
                                  "test_state_read_on_another_stream_between_deferred_steps",
                                  "test_deferred_steps_mixed_with_host_steps_and_detach",
                                  "test_dense_sub_tiles_and_ties_on_the_bulk_pass",
                                  "test_bulk_pass_reports_non_finite_values"])
def test_deferral(name, monkeypatch):
    monkeypatch.setattr(test_gpu_deferred, "D_BULK", D)
    getattr(test_gpu_deferred, name)()


@pytest.mark.parametrize("variant,compressor,K", [
    ("server_momentum", "topk", 3), ("lr_in_residual", "topk_approx", 2), ("local_momentum", "topk", 7),
    ("local_momentum_mfm", "topk_approx", 2)])
def test_variants(variant, compressor, K):
    test_gpu_variants.test_variant_parity(variant, compressor, D, K)


@pytest.mark.parametrize("variant", test_gpu_variants.VARIANTS)
@pytest.mark.parametrize("compressor", ["topk", "topk_approx"])
def test_variants_load_store(variant, compressor):
    test_gpu_variants.test_variant_parity(variant, compressor, D_LS, K_LS)


@pytest.mark.parametrize("variant,compressor", [("lr_in_residual", "topk"), ("local_momentum", "topk_approx")])
def test_variants_load_store_one_worker(variant, compressor):
    test_gpu_variants.test_variant_parity(variant, compressor, D_LS1, 1)


@pytest.mark.parametrize("d,K", [(D, 8), (D, 3), (D_LS1, 1)])
def test_approximate(d, K):
    test_gpu_approx.test_approx_bulk_pass_deferred(d, K)


@pytest.mark.parametrize("offset", [0, 1])
def test_copies_at_every_alignment(offset):
    test_gpu_parity.test_topk_bulk_copy_path(offset, D, 3)


@pytest.mark.parametrize("pinned", [True, False])
def test_host_steps(pinned, monkeypatch):
    monkeypatch.setattr(test_gpu_deferred, "D_BULK", D)
    test_gpu_deferred.test_host_steps_pinned_and_pageable(pinned)
    test_gpu_bf16.test_bf16_host_steps(pinned, D)


def test_approximate_limit_ties_and_host_steps():
    test_gpu_approx.test_approx_limit_takes_exact_top(D)
    test_gpu_approx.test_approx_ties_all_sent(D)
    test_gpu_approx.test_approx_host_steps_and_gmcplus_detach(D)


@pytest.mark.parametrize("d,K", [(D, 3), (D_LS, K_LS)])
def test_allocation_failures(d, K):
    test_gpu_failure.test_create_allocation_failures_leak_nothing(d, K, 0)


@pytest.mark.parametrize("case", [
    dict(compressor="topk", d=D, K=4, ratio=0.002), dict(compressor="topk", d=D, K=6, ratio=0.002),
    dict(compressor="topk", d=D, K=3, ratio=0.002, offset=1), dict(compressor="topk", d=D_LS1, K=1, ratio=0.002),
    dict(compressor="topk", d=D_LS, K=K_LS, ratio=0.002, offset=3),
    dict(compressor="topk_approx", d=D, K=2, ratio=1 / 1024),
    dict(compressor="topk", d=D, K=3, ratio=0.002, variant="local_momentum")], ids=str)
def test_bf16(case):
    test_gpu_bf16.test_bf16_step_parity(case)


@pytest.mark.parametrize("case", [
    dict(compressor="topk", d=D, K=4, ratio=0.002), dict(compressor="topk", d=D, K=6, ratio=0.002),
    dict(compressor="topk", d=2_500_001, K=4, ratio=0.002),  # load/store pass
    dict(compressor="topk", d=D_LS, K=K_LS, ratio=0.002, variant="server_momentum"),
    dict(compressor="topk_approx", d=D_LS, K=K_LS, ratio=0.002, variant="local_momentum_mfm"),
    dict(compressor="topk_approx", d=D, K=2, ratio=1 / 1024),
    dict(compressor="topk", d=D, K=2, ratio=0.002, variant="local_momentum")], ids=str)
def test_checkpoint(case):
    test_gpu_checkpoint.test_resume_continues_the_trajectory(case)


@pytest.mark.parametrize("read_between", [False, True])
@pytest.mark.parametrize("K", [2, 5, 16])
def test_sent_pairs_concentrated_in_one_region(K, read_between):
    """Gradients whose scale falls along the coordinates: sub-tiles of 512 hold
    every number of sent pairs from none to some hundreds, so the counts cross 32
    (one round) and 64 (two rounds), for a pending aggregation and an applied one."""
    rng = np.random.default_rng(60 + K)
    p = Pair(D, K, 0.9, 0.1, ratio=0.004, seed=11)
    scale = np.exp(-np.arange(D) / (0.05 * D)).astype(np.float32)
    for t in range(3):
        r = p.step(rng.standard_normal((K, D), dtype=np.float32) * scale)
        p.compare(r, state=read_between or t == 2)
    per_sub = np.bincount(np.concatenate(r.supports) // 512)
    assert per_sub.min() <= 32 < 64 < per_sub.max()
    p.compare_stats()
    assert p.gpu.check() == 0
    p.gpu.close()
