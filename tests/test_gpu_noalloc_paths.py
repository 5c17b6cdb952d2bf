"""gmc_topk_noalloc where its interval of keys misses the k-th, is crowded, or
has to be narrowed to one key, at every alignment of x, against the oracle."""
import numpy as np
import pytest

import oracle
from parity_util import bits

pytestmark = pytest.mark.gpu


def _run(x_np, k, offset=0):
    import torch
    from paper_1905_12948_gb300 import gmc
    n = x_np.size
    buf = torch.full((n + 8,), float("inf"), dtype=torch.float32, device="cuda")
    x = buf[offset: offset + n]
    x.copy_(torch.from_numpy(x_np))
    idx = torch.full((k + 1,), -1, dtype=torch.int32, device="cuda")
    val = torch.full((k + 1,), 7.0, dtype=torch.float32, device="cuda")
    st = gmc.load().gmc_topk_noalloc(x.data_ptr(), n, k, idx.data_ptr(), val.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    got, v = idx.cpu().numpy(), val.cpu().numpy()
    assert got[k] == -1 and v[k] == 7.0, "written past k"
    want = oracle.top_s_support(x_np, k)
    assert np.array_equal(got[:k].astype(np.int64), want)
    assert np.array_equal(bits(v[:k]), bits(x_np[want]))


def _band(rng, n, lo, hi):
    return (rng.uniform(lo, hi, n) * np.where(rng.random(n) < 0.5, -1, 1)).astype(np.float32)


CASES = {
    "one_block": lambda rng: (rng.standard_normal(8_192), 100),
    "two_blocks": lambda rng: (rng.standard_normal(8_193), 8_000),
    "k_1_far_above_the_sample": lambda rng: (np.append(rng.standard_normal(3_000_000), 1e30), 1),
    "few_far_above": lambda rng: (np.concatenate([_band(rng, 40, 1e20, 1e25), rng.standard_normal(2_000_000)]), 17),
    "crowded_in_2_10_keys": lambda rng: (_band(rng, 4_000_000, 1.0, 1.00001), 40_000),
    "list_overflows_then_narrows": lambda rng: (_band(rng, 6_000_000, 1.0, 2.0), 1_500_000),
    "zeros_are_kept": lambda rng: (np.where(rng.random(3_000_000) < 0.001, rng.standard_normal(3_000_000), 0.0), 50_000),
    "ties_in_one_slice": lambda rng: (np.concatenate([rng.standard_normal(2_000_000) * 0.1, np.full(60_000, -3.0)]), 30_000),
    "k_is_n": lambda rng: (rng.standard_normal(2_000_003), 2_000_003),
    "sorted_rising": lambda rng: (np.linspace(0, 1, 3_000_001), 3_000),
}


@pytest.mark.parametrize("case", list(CASES))
def test_narrowing(case):
    rng = np.random.default_rng(sum(map(ord, case)))
    x, k = CASES[case](rng)
    x = np.ascontiguousarray(x, np.float32)
    for _ in range(2):  # the scratch is left as it was found
        _run(x, k)


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("n", [1, 2, 5, 127, 129, 20_001])
def test_alignment(n, offset):
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n).astype(np.float32)
    for k in {1, (n + 1) // 2, n}:
        _run(x, k, offset)


def test_passes_in_quick_succession():
    """A few blocks whose passes last a microsecond or two and are many (more keys in
    the interval than the list takes, so that it is narrowed again): a block's
    counts of one pass stand until every other block has read them."""
    rng = np.random.default_rng(77)
    for n in (24_577, 60_001):
        for width in (1e-5, 3e-4):
            x = np.ascontiguousarray(_band(rng, n, 1.0, 1.0 + width))
            x[rng.integers(0, n, n // 3)] = 1.0
            for k in (n // 3, n // 2, n - 1):
                for _ in range(10):
                    _run(x, k)
