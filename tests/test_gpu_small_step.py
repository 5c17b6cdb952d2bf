"""The top-k step as one cooperative launch (problems that fit in the SMs' shared
memory): edges of its split into groups of 128, its radix rounds, lists and ties,
and steps of the other path before and after it. Bit for bit against the oracle."""
import numpy as np
import pytest

from parity_util import Pair, assert_fp32_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compressor", ["topk", "topk_approx"])
@pytest.mark.parametrize("d,K,ratio", [
    (1, 1, 1.0), (5, 2, 0.5), (127, 3, 0.1), (129, 32, 0.05), (1_000, 9, 1.0),
    (128 * 17, 1, 0.02), (32_768, 4, 0.01), (32_769, 4, 0.01), (4_096, 32, 0.01),  # one cluster, up to its largest
    (128 * 152, 4, 0.01), (128 * 152 + 1, 5, 0.001), (210_001, 32, 0.01), (900_007, 8, 0.002),
    (1_200_003, 1, 0.3), (128 * 152 * 94, 4, 0.001), (128 * 152 * 47 - 1, 8, 0.001),  # all of a block's 376 items
    (128 * 152 * 376 - 3, 1, 0.001),
])
def test_sizes(d, K, ratio, compressor):
    rng = np.random.default_rng(d + K)
    p = Pair(d, K, 0.9, 0.1, compressor=compressor, ratio=ratio, seed=4)
    assert p.route() == "one launch"
    for t in range(3):
        g = (rng.standard_normal((K, d)) * np.exp(rng.uniform(-3, 0, size=d))).astype(np.float32)
        p.compare(p.step(g), workers=sorted({0, K - 1}))
    p.compare_stats()
    assert p.gpu.check() == 0


@pytest.mark.parametrize("d,K", [(128 * 152 * 94 + 1, 4), (128 * 152 * 376 + 1, 1)])
def test_one_coordinate_past_the_largest(d, K):
    p = Pair(d, K, 0.9, 0.1, ratio=0.001)
    assert p.route() == "load/store"
    for t in range(2):
        p.compare(p.step(np.random.default_rng(t).standard_normal((K, d), dtype=np.float32)))
    p.compare_stats()


@pytest.mark.parametrize("levels,ratio", [(1, 0.3), (3, 0.1), (200, 0.01), (200_000, 0.02)])
def test_ties(levels, ratio):
    """Few distinct magnitudes: ties at the k-th key from 64 up to all of d."""
    d, K = 300_003, 3
    rng = np.random.default_rng(levels)
    p = Pair(d, K, 0.0, 0.1, ratio=ratio, w0=np.zeros(d, np.float32))
    for t in range(2):
        g = rng.integers(1, levels + 1, size=(K, d)).astype(np.float32) * rng.choice([-1.0, 1.0], size=(K, d))
        p.compare(p.step(g.astype(np.float32)))
    p.compare_stats()


@pytest.mark.parametrize("variant,lam", [("gmc", 0.5), ("server_momentum", None), ("lr_in_residual", None),
                                         ("local_momentum", 0.3), ("local_momentum_mfm", 0.3)])
@pytest.mark.parametrize("bf16,offset", [(False, 1), (True, 3)])
def test_forms_with_detached_rows_and_misaligned_inputs(variant, lam, bf16, offset):
    import torch
    d, K = 40_003, 5
    rng = np.random.default_rng(7)
    p = Pair(d, K, 0.9, 0.1, ratio=0.01, variant=variant, lam=lam)
    out = torch.zeros(K * (d + 1) + 8, dtype=torch.float32, device=p.dev)
    if lam is not None:
        assert p.gpu.lib.gmc_set_detach_output(p.gpu.h, out.data_ptr() + 4 * offset, d + 1) == 0
    dt = torch.bfloat16 if bf16 else torch.float32
    buf = torch.empty(K * d + offset, dtype=dt, device=p.dev)
    for t in range(3):
        g = torch.from_numpy(rng.standard_normal((K, d)).astype(np.float32)).to(dt)
        view = buf[offset:].view(K, d)
        view.copy_(g)
        p.compare(p.step(g.float().numpy(), view))
        if lam is not None:
            rows = out[offset: offset + K * (d + 1)].view(K, d + 1).cpu().numpy()
            for k in range(K):
                assert_fp32_state(rows[k, :d], p.ref.worker_params(k), f"detached row {k}")
    p.compare_stats()


def test_alternating_with_the_dense_engine():
    """Steps of the one-launch path and of the dense engine continue one another."""
    d, K = 50_001, 4
    rng = np.random.default_rng(3)
    p = Pair(d, K, 0.9, 0.1, ratio=0.01)
    for t in range(6):
        assert p.gpu.lib.gmc_set_select_mode(p.gpu.h, t % 2) == 0
        p.compare(p.step(rng.standard_normal((K, d)).astype(np.float32)))
    p.compare_stats()


def test_captured_in_a_graph():
    import torch
    d, K = 65_536, 4
    rng = np.random.default_rng(5)
    p = Pair(d, K, 0.9, 0.1, ratio=0.01)
    g = [rng.standard_normal((K, d)).astype(np.float32) for _ in range(2)]
    dev = [torch.from_numpy(x).to(p.dev) for x in g]
    p.step(g[0], dev[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        p.gpu.step(dev[1])
    graph.replay()
    torch.cuda.synchronize()
    p.compare(p.ref.step(g[1]))


@pytest.mark.parametrize("d,K", [(65_536, 4), (1_300_001, 3), (1_300_001, 8), (5_100_001, 2)])
def test_step_and_read_captured_after_a_read(d, K):
    """A step and a read of w captured on another stream than the read before them,
    replayed once, and read and stepped on from outside; also at sizes whose reads
    are ordered across streams."""
    import torch
    rng = np.random.default_rng(5)
    p = Pair(d, K, 0.9, 0.1, ratio=0.01)
    g = [torch.from_numpy(rng.standard_normal((K, d)).astype(np.float32)).to(p.dev) for _ in range(3)]
    w = torch.empty(d, device=p.dev)
    p.compare(p.step(g[0].cpu().numpy(), g[0]))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        p.gpu.step(g[1])
        assert p.gpu.lib.gmc_get_params(p.gpu.h, w.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    graph.replay()
    torch.cuda.synchronize()
    r = p.ref.step(g[1].cpu().numpy())
    assert_fp32_state(w.cpu().numpy(), p.ref.w, "w")
    p.compare(r)
    p.compare(p.step(g[2].cpu().numpy(), g[2]))


def test_handles_and_calls_on_streams_of_their_own():
    """Two handles and the bare compressor, each a launch that wants every SM at
    once, on three streams with other work between them: none waits for another
    beyond its turn, and each gives what it gives alone."""
    import torch
    from paper_1905_12948_gb300 import gmc
    import oracle
    steps = 12
    shapes = [(272_474, 8), (900_007, 7)]
    rng = np.random.default_rng(12)
    pairs = [Pair(d, K, 0.9, 0.1, ratio=0.005, seed=2) for d, K in shapes]
    assert all(p.route() == "one launch" for p in pairs)
    grads = [[rng.standard_normal((K, d)).astype(np.float32) for _ in range(steps)] for d, K in shapes]
    dev = [[torch.from_numpy(g).cuda() for g in gs] for gs in grads]
    n, k = 3_000_001, 3_000
    x_np = rng.standard_normal(n).astype(np.float32)
    x = torch.from_numpy(x_np).cuda()
    idx = torch.zeros(k, dtype=torch.int32, device="cuda")
    val = torch.zeros(k, device="cuda")
    a = torch.randn(2048, 2048, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    for t in range(steps):
        for p, gs, s in zip(pairs, dev, streams):
            with torch.cuda.stream(s):
                p.gpu.step(gs[t])
        assert gmc.load().gmc_topk_noalloc(x.data_ptr(), n, k, idx.data_ptr(), val.data_ptr(),
                                           streams[2].cuda_stream) == 0
        with torch.cuda.stream(streams[3]):
            a = torch.tanh(a @ a)
        if t == 0:
            torch.cuda.synchronize()
            assert all(p.gpu.check() == 0 for p in pairs)
    torch.cuda.synchronize()
    for p, gs in zip(pairs, grads):
        for g in gs:
            r = p.ref.step(g)
        p.compare(r)
        p.compare_stats()
        assert p.gpu.check() == 0
    assert np.array_equal(idx.cpu().numpy(), oracle.top_s_support(x_np, k))
