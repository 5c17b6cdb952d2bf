"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is one pass of a training program through the public entry points: it
hands the K workers' gradients to a handle (``GMC.step`` / ``GMC.step_host``)
and takes back what the next iteration needs -- the parameters w_{t+1} that the
next forward pass reads, and under GMC+ the detached points w_{t+1,k} -- or it
compresses one vector (``gmc_topk_noalloc``). ``steps`` is the number of
iterations between two reads of w: 1 in training, more where recorded gradients
are replayed. A handle has taken two steps before the pass, so that residuals
and w_t - w_{t-1} are those of a run under way.

Sizes are the repository's own workloads (65,536 parameters x 4 workers up to
138.4 M x 8), the sizes of its tests, and drawn ones between.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1905_12948_gb300 import GMC, gmc

BETA = 0.9
WARM = 2       # steps taken before the pass
VIEWS = 64     # gradients of consecutive steps are windows of one buffer, each 128 values
               # further on than the one it is numbered after: noise that does not repeat
               # from step to step, as stochastic gradients are
_M64 = (1 << 64) - 1
_GAMMA = 0x9E3779B97F4A7C15


def _step(name, d, K, compressor="topk", ratio=0.001, *, block=4096, per_worker=False, lam=0.0,
          detach=False, variant="gmc", dtype="f32", host=False, steps=1, eta=0.05, layers=32):
    return {"name": name, "kind": "step", "d": d, "K": K, "compressor": compressor, "ratio": ratio,
            "block": block, "per_worker": per_worker, "lam": lam, "detach": detach,
            "variant": variant, "dtype": dtype, "host": host, "steps": steps, "eta": eta,
            "layers": layers}


def listed():
    return [
        # the smallest run: a 65 k-parameter MLP and four workers, where launches count
        _step("topk_mlp65k", 65_536, 4, ratio=0.01, eta=0.1, layers=1),
        # the paper's CIFAR model (ResNet20) with its eight workers
        _step("topk_resnet20", 272_474, 8, ratio=0.01, eta=0.1, layers=20),
        # many workers on a small model, an odd size: every gradient row at another alignment
        _step("topk_20_workers", 1_300_001, 20, ratio=0.002, eta=0.05, layers=20),
        # an ordinary model (ResNet18) trained step by step, w read after each
        _step("topk_resnet18", 11_173_962, 16, layers=62),
        # the largest model (VGG16), gradients replayed: four steps between reads of w
        _step("topk_vgg16_replay", 138_357_544, 8, eta=0.01, steps=4),
        # the same model trained step by step from bfloat16 gradients
        _step("topk_vgg16_bf16", 138_357_544, 8, eta=0.01, dtype="bf16"),
        # approximate top-s (a fresh random sample sets the threshold), ratio 1/1024
        _step("approx_vgg16", 138_357_544, 8, "topk_approx", 1 / 1024, eta=0.01),
        # GMC+ with random blocks: ResNet50, 32 workers, the detached points written each step
        _step("gmcplus_rbgs_resnet50", 25_557_032, 32, "rbgs", 0.01, lam=0.5, detach=True, eta=0.1,
              layers=161),
        # GMC+ on the small model, short blocks chosen by each worker for itself
        _step("gmcplus_rbgs_resnet20", 272_474, 8, "rbgs", 0.05, block=256, per_worker=True, lam=0.5,
              detach=True, eta=0.1, layers=20),
        # the baseline the method is compared with: local momentum with factor masking
        _step("local_mfm_resnet18", 11_173_962, 16, variant="local_momentum_mfm", layers=62),
        # gradients that arrive in page-locked host memory, the step's counters read back
        _step("host_resnet18", 11_173_962, 16, host=True, layers=62),
        # the compressor alone, on one vector of ResNet50's size, in buffers of the caller
        {"name": "noalloc_resnet50", "kind": "noalloc", "d": 25_557_032, "k": 25_557, "layers": 161},
    ]


def _size(rng, lo, hi):
    d = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return d - d % 8 if rng.random() < 0.4 else d


def draw(rng):
    family = rng.choice(["topk", "topk", "topk", "approx", "rbgs", "rbgs", "variant", "host", "noalloc"])
    if family == "noalloc":
        n = _size(rng, 3_000, 1 << 26)
        return {"kind": "noalloc", "d": n, "k": max(1, int(n * math.exp(rng.uniform(math.log(5e-4), math.log(0.02))))),
                "layers": 32}
    K = int(math.exp(rng.uniform(0.0, math.log(32.99))))
    most = 1.5e8 if family == "host" else 1.1e9   # values of one batch of gradients
    d = _size(rng, 3_000, min(138_400_000, most / K))
    c = _step("", d, K, ratio=math.exp(rng.uniform(math.log(5e-4), math.log(0.02))),
              eta=rng.choice([0.01, 0.05, 0.1]), layers=rng.choice([1, 20, 62]),
              dtype=rng.choice(["f32", "f32", "bf16"]))
    if family == "topk":
        c["lam"] = rng.choice([0.0, 0.0, 0.5])
        c["detach"] = c["lam"] > 0
        c["steps"] = rng.choice([1, 1, 1, 4]) if K * d <= 4e8 else 1
    elif family == "approx":
        c["compressor"] = "topk_approx"
    elif family == "rbgs":
        c["compressor"] = "rbgs"
        c["block"] = rng.choice([256, 1000, 4096, 4096] if d < 20_000_000 else [1000, 4096, 4096])
        c["ratio"] = math.exp(rng.uniform(math.log(2e-3), math.log(0.05)))
        c["per_worker"] = rng.choice([False, False, True])
        c["lam"] = rng.choice([0.0, 0.5])
        c["detach"] = c["lam"] > 0
    elif family == "variant":
        c["variant"] = rng.choice(["server_momentum", "lr_in_residual", "local_momentum", "local_momentum_mfm"])
    else:
        c["host"] = True
    del c["name"]
    return c


# -- inputs -------------------------------------------------------------------
def _layer_scale(d, layers, seed):
    """Gradient std per parameter: layers of random sizes, log-uniform on [1e-3, 1e-1]."""
    rng = np.random.default_rng([seed, 1])
    n = min(layers, d)
    cuts = np.sort(rng.choice(d - 1, size=n - 1, replace=False) + 1) if d < 1_000_000 else \
        np.unique(rng.integers(1, d, size=n - 1))
    sizes = np.diff(np.concatenate([[0], cuts, [d]]))
    std = np.exp(rng.uniform(math.log(1e-3), math.log(1e-1), size=sizes.size)).astype(np.float32)
    return torch.repeat_interleave(torch.from_numpy(std).cuda(), torch.from_numpy(sizes).cuda(), output_size=d)


def _inputs(case, seed):
    """w_0 and the buffer of the gradients, or the vector of the bare compressor."""
    d = case["d"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    sigma = _layer_scale(d, case["layers"], seed)
    if case["kind"] == "noalloc":
        return torch.randn(d, generator=gen, device="cuda").mul_(sigma)
    w0 = torch.randn(d, generator=gen, device="cuda").mul_(0.01)
    K = case["K"]
    buf = torch.empty(K * d + VIEWS * 128, device="cuda", dtype=torch.float32)
    buf.normal_(generator=gen)
    rows, rest = buf[: K * d].view(K, d), buf[K * d:]
    rows.mul_(sigma)
    rest.mul_(sigma.repeat(-(-rest.numel() // d))[: rest.numel()])
    # the workers' data are not identically distributed: each has its own offset
    rows.add_(torch.randn((K, 1), generator=gen, device="cuda").mul_(1e-4))
    return w0, buf.to(torch.bfloat16) if case["dtype"] == "bf16" else buf


def _gradients(case, buf, t):
    """The K x d gradients of step t."""
    at = (t * 37 % VIEWS) * 128
    return buf[at: at + case["K"] * case["d"]].view(case["K"], case["d"])


def prepare(case, seed):
    x = _inputs(case, seed)
    if case["kind"] == "noalloc":
        return {"case": case, "x": x, "idx": torch.empty(case["k"], dtype=torch.int32, device="cuda"),
                "val": torch.empty(case["k"], dtype=torch.float32, device="cuda")}
    w0, buf = x
    h = GMC(case["d"], case["K"], BETA, case["eta"], compressor=case["compressor"], ratio=case["ratio"],
            block=case["block"], lam=case["lam"], seed=11, per_worker=case["per_worker"],
            variant=case["variant"])
    h.set_params(w0)
    s = {"case": case, "h": h, "t": 0, "out": None, "stats": None}
    if case["detach"]:
        s["out"] = torch.zeros((case["K"], case["d"]), dtype=torch.float32, device="cuda")
        h.set_detach_output(s["out"])
    if case["host"]:
        s["stats"] = torch.zeros(8, dtype=torch.int64, pin_memory=True)
        pinned = torch.empty(buf.shape, dtype=buf.dtype, pin_memory=True)
        pinned.copy_(buf)
        buf = pinned
    s["g"] = buf
    for _ in range(WARM):
        _one(s)
    torch.cuda.synchronize()
    return s


def _one(s):
    g = _gradients(s["case"], s["g"], s["t"])
    s["t"] += 1
    if s["case"]["host"]:
        s["h"].step_host(g, s["stats"])
    else:
        s["h"].step(g)


def run(state):
    case = state["case"]
    if case["kind"] == "noalloc":
        st = gmc.load().gmc_topk_noalloc(state["x"].data_ptr(), case["d"], case["k"],
                                         state["idx"].data_ptr(), state["val"].data_ptr(),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if st != 0:
            raise RuntimeError(f"gmc_topk_noalloc: {st}")
        return {"idx": state["idx"], "val": state["val"]}
    for _ in range(case["steps"]):
        _one(state)
    r = {"w": state["h"].params()}
    if state["out"] is not None:
        r["detached"] = state["out"]
    if state["stats"] is not None:
        r["stats"] = state["stats"]
    return r


def work(case):
    d = case["d"]
    if case["kind"] == "noalloc":
        return {"bytes": 4 * d + 8 * case["k"], "flops": 0}
    n = case["K"] * d
    local = case["variant"].startswith("local")
    # a step: g, and e read and written (the local momentum too); w, and w as it is taken back
    per = (2 if case["dtype"] == "bf16" else 4) + 8 + (8 if local else 0) + (4 if case["detach"] else 0)
    dense = 16 * d if case["variant"] == "server_momentum" else 4 * d if case["detach"] else 0
    return {"bytes": case["steps"] * (per * n + dense) + 8 * d, "flops": 3 * case["steps"] * n}


def tolerance(case):
    # every operation of a step is fixed to one fp32 rounding in a stated order,
    # and the selections are exact: there is one right answer
    return "exact"


# -- the same in 64 bits --------------------------------------------------------
def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _stream(seed, t, stream):
    return _mix((_mix((seed + _GAMMA * (t + 1)) & _M64) + _GAMMA * (stream + 1)) & _M64)


def _blocks(seed, t, stream, nb, m):
    """Floyd's sampling of m of nb blocks from the counter stream of (seed, t, stream)."""
    key, chosen = _stream(seed, t, stream), set()
    for i in range(m):
        top = nb - m + i
        r = ((_mix((key + _GAMMA * (i + 1)) & _M64) >> 32) * (top + 1)) >> 32
        chosen.add(top if r in chosen else r)
    return sorted(chosen)


def _sample(seed, t, d):
    """Positions of the approximate top-s sample: runs of 8, one per stratum."""
    n = max(1, d // 800)
    key = _stream(seed, t, 0)
    at = []
    for r in range(n):
        lo, hi = r * d // n, (r + 1) * d // n
        a = (lo + 7) & ~7
        at.append(a + 8 * (((_mix((key + _GAMMA * (r + 1)) & _M64) >> 32) * ((hi - a) >> 3)) >> 32))
    at = torch.tensor(at, dtype=torch.int64, device="cuda")
    return (at[:, None] + torch.arange(8, device="cuda")).reshape(-1)


def _top(v, k):
    """Mask of the k largest |v|, ties to the lower index."""
    a = v.abs()
    T = torch.topk(a, k, sorted=False).values.min()
    keep = a > T
    ties = torch.nonzero(a == T).reshape(-1)[: k - int(keep.sum())]
    keep[ties] = True
    return keep


def exact(case, seed):
    x = _inputs(case, seed)
    d = case["d"]
    if case["kind"] == "noalloc":
        return {"idx": None, "val": x[_top(x, case["k"])].double()}
    w, buf = x
    w = w.double()
    K, eta, ratio = case["K"], float(np.float32(case["eta"])), case["ratio"]
    beta = float(np.float32(BETA))
    variant, comp = case["variant"], case["compressor"]
    local = variant.startswith("local")
    scaled = local or variant == "lr_in_residual"   # eta is in the residual
    c = 0.0 if local or variant == "server_momentum" else beta if scaled else beta / eta
    a = (1.0 if scaled else eta) / K
    e = torch.zeros((K, d), dtype=torch.float64, device="cuda")
    m = torch.zeros((K, d), dtype=torch.float64, device="cuda") if local else None
    dw = torch.zeros_like(w)
    nb = (d + case["block"] - 1) // case["block"]
    for t in range(WARM + case["steps"]):
        chosen = None
        if comp == "rbgs":
            kept = max(1, int(math.floor(ratio * nb)))
            chosen = [_blocks(11, t, k + 1 if case["per_worker"] else 0, nb, kept)
                      for k in range(K if case["per_worker"] else 1)]
        elif comp == "topk_approx":
            at = _sample(11, t, d)
        total = torch.zeros_like(w)
        for k in range(K):
            g = _gradients(case, buf, t)[k].double()
            if scaled:
                g = eta * g
            if local:
                m[k].mul_(beta).add_(g)
                g = m[k]
            v = (e[k] + g).sub_(dw, alpha=c)
            if comp == "rbgs":
                flag = torch.zeros(nb, dtype=torch.bool, device="cuda")
                flag[torch.tensor(chosen[k if case["per_worker"] else 0], device="cuda")] = True
                keep = torch.repeat_interleave(flag, case["block"])[:d]
            elif comp == "topk":
                keep = _top(v, max(1, int(math.floor(ratio * d))))
            else:
                s = v[at].abs()
                theta = torch.topk(s, max(1, int(math.floor(ratio * s.numel())))).values.min()
                keep = v.abs() >= theta
                limit = min(d, 4 * max(1, int(math.floor(ratio * d))) + 4096)
                if int(keep.sum()) > limit:
                    keep = _top(v, limit)
            total += torch.where(keep, v, 0.0)
            e[k] = v.masked_fill_(keep, 0.0)
            if variant == "local_momentum_mfm":
                m[k].masked_fill_(keep, 0.0)
        wn = w - a * total
        if variant == "server_momentum":
            wn = wn + beta * dw
        dw, w = wn - w, wn
    r = {"w": w}
    if case["detach"]:
        b = case["lam"] * (1.0 if local else eta)
        r["detached"] = e.mul_(-b).add_(w)
    if case["host"]:
        r["stats"] = None
    return r
