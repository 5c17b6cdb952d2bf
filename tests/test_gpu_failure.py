"""Failure detection without a GPU fault.

* A bounded wait that runs out: the test hook withholds one item's copy in a
  bulk pass, so the waits on it give up after a short limit; the kernel
  returns, gmc_check reports GMC_ETIMEOUT, and a reset (or a new handle) steps
  exactly as the oracle again. Likewise a block that leaves before a grid
  barrier of gmc_topk_noalloc or of the one-launch top-k step.
* A device allocation that fails: the allocation hook makes the n-th
  allocation of gmc_create / gmc_set_variant fail as cudaMalloc does when
  memory runs out; the call returns GMC_ENOMEM, leaks nothing, and leaves an
  existing handle as it was.
"""
import ctypes
import gc

import numpy as np
import pytest

from parity_util import Pair, bits

pytestmark = pytest.mark.gpu

GMC_OK, GMC_EINVAL, GMC_ENOMEM, GMC_ETIMEOUT = 0, 1, 2, 8
TILE = 4096


def _lib():
    from paper_1905_12948_gb300 import gmc
    return gmc.load()


def _grads(rng, K, d):
    return (rng.standard_normal((K, d)) * 0.1).astype(np.float32)


@pytest.mark.parametrize("compressor,d,K,hold", [
    ("topk", 5_100_001, 6, (1_000, 3)),  # bulk top-k pass, the one-tile pipeline
    ("topk", 1_300_001, 3, (5, 1)),      # moved to the bulk pass by the hook (d >= 4096 * 2 * SMs), an odd worker
    ("topk", 1_300_001, 4, (0, 0)),      # the first fixed tile of CTA 0, the lead warps' worker
    ("topk_approx", 1_300_001, 2, (317, 1)),  # the last tile, ragged
    ("rbgs", 700_001, 3, (40, 2)),       # bulk RBGS pass (d >= 4096 * SMs)
])
def test_withheld_copy_times_out_and_is_reported(compressor, d, K, hold):
    import torch
    lib = _lib()
    rng = np.random.default_rng(11)
    ratio = 0.05 if compressor == "rbgs" else 0.001
    p = Pair(d, K, 0.9, 0.1, compressor=compressor, ratio=ratio, block=4096, seed=3)
    for _ in range(2):
        r = p.step(_grads(rng, K, d))
    p.compare(r)
    assert p.gpu.check() == GMC_OK
    tile, k = hold
    assert lib.gmc_test_withhold_copy(p.gpu.h, tile, k, 50_000_000) == GMC_OK
    g = torch.from_numpy(_grads(rng, K, d)).cuda()
    p.gpu.step(g)
    torch.cuda.synchronize()
    st = p.gpu.check()
    assert st == GMC_ETIMEOUT, lib.gmc_strerror(st)
    assert b"bounded wait" in lib.gmc_strerror(GMC_ETIMEOUT)
    assert p.gpu.check() == GMC_ETIMEOUT  # reading does not clear it

    # the same handle after a reset, and a new handle, step as the oracle does
    p2 = Pair(d, K, 0.9, 0.1, compressor=compressor, ratio=ratio, block=4096, seed=3)
    w0 = (np.random.default_rng(5).standard_normal(d) * 0.01).astype(np.float32)
    p.gpu.set_params(torch.from_numpy(w0).cuda())
    p.ref.set_params(w0)
    p2.gpu.set_params(torch.from_numpy(w0).cuda())
    p2.ref.set_params(w0)
    assert p.gpu.check() == GMC_OK
    for _ in range(3):
        g = _grads(rng, K, d)
        r = p.step(g)
        r2 = p2.step(g)
    p.compare(r)
    p2.compare(r2)
    assert p.gpu.check() == GMC_OK and p2.gpu.check() == GMC_OK
    p.gpu.close()
    p2.gpu.close()


@pytest.mark.parametrize("compressor,d,K", [("topk", 50_003, 4), ("topk", 900_007, 7), ("topk_approx", 300_001, 3)])
def test_one_launch_step_whose_wait_gives_up(compressor, d, K):
    """A block that never comes to the barrier: the step is reported, the steps
    after it leave the state alone, and a reset handle steps as the oracle does."""
    import torch
    lib = _lib()
    rng = np.random.default_rng(d)
    p = Pair(d, K, 0.9, 0.1, compressor=compressor, ratio=0.01, seed=3)
    p.compare(p.step(_grads(rng, K, d)))
    assert lib.gmc_test_leave_barrier(p.gpu.h, 20_000_000) == GMC_OK
    g = torch.from_numpy(_grads(rng, K, d)).cuda()
    p.gpu.step(g)
    assert p.gpu.check() == GMC_ETIMEOUT
    state = [p.gpu.residual(k).clone() for k in range(K)] + [p.gpu.params().clone()]
    for _ in range(3):
        p.gpu.step(g)
    assert p.gpu.check() == GMC_ETIMEOUT
    after = [p.gpu.residual(k) for k in range(K)] + [p.gpu.params()]
    assert all(torch.equal(a, b) for a, b in zip(state, after))
    w0 = (np.random.default_rng(5).standard_normal(d) * 0.01).astype(np.float32)
    p.gpu.set_params(torch.from_numpy(w0).cuda())
    p.ref.set_params(w0)
    assert p.gpu.check() == GMC_OK
    for _ in range(3):
        p.compare(p.step(_grads(rng, K, d)))
    p.compare_stats()
    assert p.gpu.check() == GMC_OK


@pytest.mark.parametrize("compressor,d", [("topk", 5_003), ("rbgs", 5_003)])
def test_getters_leave_other_destinations_to_the_copy_call(compressor, d):
    """Host memory as a getter's destination: copied to or refused by the CUDA
    copy call, as it decides, and never written by a kernel; pinned memory is
    copied to. (The header asks for device memory.)"""
    import torch
    lib = _lib()
    K = 2
    p = Pair(d, K, 0.9, 0.1, compressor=compressor, ratio=0.05, block=64)
    p.step(_grads(np.random.default_rng(2), K, d))
    s = torch.cuda.current_stream().cuda_stream
    for pinned in (True, False):
        for read, want in ((lambda q: lib.gmc_get_params(p.gpu.h, q, s), p.ref.w),
                           (lambda q: lib.gmc_get_residual(p.gpu.h, 1, q, s), p.ref.e[1])):
            out = torch.zeros(d, pin_memory=pinned)
            st = read(out.data_ptr())
            torch.cuda.synchronize()
            assert st == GMC_OK if pinned else st in (GMC_OK, 3)
            if st == GMC_OK:
                assert np.array_equal(bits(out.numpy()), bits(want))
    p.compare(p.step(_grads(np.random.default_rng(3), K, d)))


@pytest.mark.parametrize("compressor,d,K,ratio", [
    ("topk", 1, 1, 1.0), ("topk", 4_099, 3, 0.01), ("topk", 32_768, 8, 0.01), ("topk", 65_537, 4, 0.01),
    ("topk", 900_007, 7, 0.002), ("topk", 1_300_001, 3, 0.01),
    ("topk_approx", 5, 2, 0.5), ("topk_approx", 40_001, 5, 0.01), ("topk_approx", 300_001, 3, 0.01),
])
@pytest.mark.parametrize("variant,lam", [("gmc", 0.5), ("server_momentum", None), ("local_momentum_mfm", 0.3)])
def test_one_launch_step_refused_by_its_context(compressor, d, K, ratio, variant, lam):
    """A context with fewer SMs than the one-launch step's blocks: the step that is
    refused and those after it take the load/store pass and give the same."""
    import torch
    lib = _lib()
    rng = np.random.default_rng(d)
    p = Pair(d, K, 0.9, 0.1, compressor=compressor, ratio=ratio, seed=3, variant=variant, lam=lam)
    out = torch.zeros(K, d, device="cuda")
    if lam is not None:
        assert lib.gmc_set_detach_output(p.gpu.h, out.data_ptr(), d) == GMC_OK
    for t in range(5):
        if t == 2:
            assert lib.gmc_test_refuse_cooperative(1) == GMC_OK
        r = p.step(_grads(rng, K, d))
        p.compare(r, workers=sorted({0, K - 1}))
        if lam is not None:
            assert np.array_equal(bits(out[K - 1].cpu().numpy()), bits(p.ref.worker_params(K - 1)))
    p.compare_stats()
    assert p.gpu.check() == GMC_OK
    p.gpu.profile()
    p.step(_grads(rng, K, d))
    assert "dense_select" in p.gpu.profile_read()  # the load/store pass


@pytest.mark.parametrize("n,k,refused", [(20_000, 300, 1), (3_000_001, 3_000, 2), (3_000_001, 2_000_000, 7),
                                         (30_000_000, 30_000, 7), ((1 << 26) - 3, 60_000, 6)])
def test_noalloc_refused_by_its_context(n, k, refused):
    """Fewer SMs than blocks: the call is repeated with half the blocks, down to one."""
    import oracle
    import torch
    lib = _lib()
    x_np = np.random.default_rng(n).standard_normal(n, dtype=np.float32)
    x = torch.from_numpy(x_np).cuda()
    idx = torch.zeros(k, dtype=torch.int32, device="cuda")
    val = torch.zeros(k, dtype=torch.float32, device="cuda")
    assert lib.gmc_test_refuse_cooperative(refused) == GMC_OK
    assert lib.gmc_topk_noalloc(x.data_ptr(), n, k, idx.data_ptr(), val.data_ptr(),
                                torch.cuda.current_stream().cuda_stream) == GMC_OK
    assert lib.gmc_test_refuse_cooperative(0) == GMC_OK
    torch.cuda.synchronize()
    want = oracle.top_s_support(x_np, k)
    assert np.array_equal(idx.cpu().numpy(), want)
    assert np.array_equal(bits(val.cpu().numpy()), bits(x_np[want]))


def test_leave_barrier_refused_without_a_grid_barrier():
    import torch
    from paper_1905_12948_gb300 import GMC
    lib = _lib()
    for d, K in [(1_000, 2), (1_300_001, 20)]:  # one cluster; load/store pass
        h = GMC(d, K, 0.9, 0.1, compressor="topk", ratio=0.01)
        h.set_params(torch.zeros(d, device="cuda"))
        assert lib.gmc_test_leave_barrier(h.h, 1_000_000) == GMC_EINVAL
        h.close()


@pytest.mark.parametrize("n,k", [(20_000, 300), (3_000_001, 3_000), (100_000, 100_000)])
def test_noalloc_wait_that_gives_up_marks_its_output(n, k):
    """A block that never comes to the barrier: the call returns, its indices say
    that there is no selection, and the next call is as if it had not been."""
    import oracle
    import torch
    lib = _lib()
    x_np = np.random.default_rng(n).standard_normal(n).astype(np.float32)
    x = torch.from_numpy(x_np).cuda()
    idx = torch.zeros(k, dtype=torch.int32, device="cuda")
    val = torch.zeros(k, dtype=torch.float32, device="cuda")

    def call():
        assert lib.gmc_topk_noalloc(x.data_ptr(), n, k, idx.data_ptr(), val.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream) == GMC_OK
        torch.cuda.synchronize()
        return idx.cpu().numpy()

    want = oracle.top_s_support(x_np, k)
    assert np.array_equal(call(), want)
    assert lib.gmc_test_leave_barrier(None, 20_000_000) == GMC_OK
    assert np.all(call() == -1)
    assert np.array_equal(call(), want)


def test_withhold_refused_without_a_bulk_pass():
    import torch
    from paper_1905_12948_gb300 import GMC
    lib = _lib()
    small = GMC(100_000, 2, 0.9, 0.1, compressor="topk", ratio=0.01)  # one launch, too small for the bulk pass
    small.set_params(torch.zeros(100_000, device="cuda"))
    assert lib.gmc_test_withhold_copy(small.h, 0, 0, 1_000_000) == GMC_EINVAL
    small.close()
    big = GMC(1_300_001, 2, 0.9, 0.1, compressor="topk", ratio=0.001)
    assert lib.gmc_test_withhold_copy(big.h, 0, 2, 1_000_000) == GMC_EINVAL   # worker out of range
    assert lib.gmc_test_withhold_copy(big.h, 318, 0, 1_000_000) == GMC_EINVAL  # tile out of range
    assert lib.gmc_test_withhold_copy(big.h, 0, 0, 0) == GMC_EINVAL            # no limit
    assert lib.gmc_test_withhold_copy(big.h, 0, 0, 3_000_000_000) == GMC_EINVAL
    big.close()


@pytest.mark.parametrize("d,K,compressor", [
    (100_000, 4, 0),      # top-k, one-launch step (the other passes: test_gpu_bulk_sizes.py)
    (1_300_001, 3, 0),
    (700_001, 5, 1),      # RBGS
    (300_000, 2, 2),      # approximate top-s
])
def test_create_allocation_failures_leak_nothing(d, K, compressor):
    import torch
    lib = _lib()
    torch.cuda.init()
    gc.collect()  # handles of earlier tests still waiting for the collector
    live0 = lib.gmc_test_fail_alloc(-1)
    failures = 0
    for i in range(64):
        lib.gmc_test_fail_alloc(i)
        h = ctypes.c_void_p()
        st = lib.gmc_create(ctypes.byref(h), d, K, 0.9, 0.1, compressor, 0.01, 4096)
        live = lib.gmc_test_fail_alloc(-1)
        if st == GMC_OK:
            assert live > live0
            lib.gmc_destroy(h)
            break
        assert st == GMC_ENOMEM, (i, st)
        assert h.value is None
        assert live == live0, f"allocation {i} failed and {live - live0} allocations leaked"
        failures += 1
    else:
        pytest.fail("gmc_create never succeeded")
    assert failures >= 8  # every allocation of the handle's state was made to fail once
    assert lib.gmc_test_fail_alloc(-1) == live0


def test_set_variant_allocation_failure_leaves_the_handle_usable():
    import torch
    lib = _lib()
    d, K = 200_003, 3
    rng = np.random.default_rng(4)
    gc.collect()
    p = Pair(d, K, 0.9, 0.1, compressor="topk", ratio=0.01)
    live = lib.gmc_test_fail_alloc(-1)
    for variant in (1, 3):  # Alg. 3's server momentum, the local momentum: one allocation each
        lib.gmc_test_fail_alloc(0)
        assert lib.gmc_set_variant(p.gpu.h, variant) == GMC_ENOMEM
        assert lib.gmc_test_fail_alloc(-1) == live
    for _ in range(3):  # still Alg. 1, still exact
        r = p.step(_grads(rng, K, d))
    p.compare(r)
    p.compare_stats()
    assert p.gpu.check() == GMC_OK
    p.gpu.close()
    assert lib.gmc_test_fail_alloc(-1) == live - _handle_allocations(d, K)


def _handle_allocations(d, K):
    """Device allocations one top-k handle of this size holds (counted with the hook)."""
    lib = _lib()
    before = lib.gmc_test_fail_alloc(-1)
    h = ctypes.c_void_p()
    assert lib.gmc_create(ctypes.byref(h), d, K, 0.9, 0.1, 0, 0.01, 4096) == GMC_OK
    n = lib.gmc_test_fail_alloc(-1) - before
    lib.gmc_destroy(h)
    assert lib.gmc_test_fail_alloc(-1) == before
    return n


@pytest.mark.parametrize("variant", ["gmc", "local_momentum"])
def test_memory_allocated_on_the_way_is_ready_on_any_stream(variant):
    """The staging buffer of pageable host gradients and a variant's momentum are
    allocated by a call and cleared on the default stream: the work of that call
    on another stream comes after, however busy the default stream is."""
    import torch
    d, K = 200_003, 3
    rng = np.random.default_rng(8)
    p = Pair(d, K, 0.9, 0.1, ratio=0.01)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    g = [_grads(rng, K, d) for _ in range(2)]
    torch.cuda._sleep(20_000_000)  # the default stream, about 10 ms
    if variant != "gmc":
        assert _lib().gmc_set_variant(p.gpu.h, 3) == GMC_OK
        p.ref = type(p.ref)(d, K, 0.9, 0.1, compressor="topk", ratio=0.01, variant=variant)
        p.ref.set_params(p.gpu.params().cpu().numpy())
        torch.cuda.synchronize()
        torch.cuda._sleep(20_000_000)
    for x in g:
        p.gpu.step_host(torch.from_numpy(x), stream=s)
        r = p.ref.step(x)
    torch.cuda.synchronize()
    p.compare(r)
