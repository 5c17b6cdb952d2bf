// One top-k step (Alg. 1 with the exact or the approximate top-s, and the
// appendix variants) as ONE cooperative launch, for problems whose K x d
// accumulator fits in the SMs' shared memory (about 7 M values).
//
// A block owns the groups of 128 coordinates g with g mod grid its index, for all
// K workers, and keeps their accumulators v in shared memory from the moment they
// are formed until the residuals are written:
//   form     v = (e + g) - c*(w_t - w_{t-1}); e, g and w_t - w_{t-1} read once
//   select   radix rounds over all blocks: each round a histogram of 2,048 bins
//            per worker of the digit in question, a grid barrier, and every
//            block finds the bin that holds the k-th key (a warp per worker).
//            Two digits of 11 bits leave a few elements; up to kListCap of them
//            are listed (key, index) and ranked directly. Crowded keys go on to
//            the last 9 bits and, if tied, to digits of the index.
//   apply    a coordinate's K values are all here: sent values summed in
//            ascending worker order, w and w_{t+1} - w_t updated, residuals
//            written, the sent pairs appended to their sub-chunks in index order
// The approximate top-s ranks the sampled coordinates' keys the same way, then
// counts what reaches theta, and ranks all keys when that exceeds its limit.
//
// Bound by latency and issue: three grid barriers, a dozen dependent L2 accesses,
// a few passes over shared memory. Step and read of w, where the step took nine
// launches: d = 65,536, K = 4: 53 -> 22 us; d = 272 k, K = 8: 70 -> 36 us (steps
// alone, back to back: 21.3 and 35.0; 21.7 and 37.5 when a barrier's arrival was
// an atomic whose answer its block waited for). 768 threads, 80 registers (28 to
// 68 bytes of spills): with 512 the passes over shared memory are short of warps,
// with 1,024 more is spilled; either took 2 us more at d = 272 k, K = 8.
#include <algorithm>

#include "gmc_internal.h"

namespace gmc {
namespace {

constexpr int kSmThreads = 768;
constexpr int kSmWarps = kSmThreads / 32;
constexpr int kMaxK = 32;
constexpr int kItemMax = kSmallItems;       // (group, worker) items of a block
constexpr int kListCap = 64;                // listed elements per worker
constexpr int kCoarse = kHistBins / 32;     // sums of 32 bins
constexpr int kHistWords = kHistBins + kCoarse;
constexpr uint32_t kDirect = 65536;         // keys of a bin that go straight to the global histogram
constexpr int kIdxBits = 23;                // an index digit's range: d < 2^23
constexpr int kClusterMax = 16;             // blocks of a cluster launch (above the portable 8)
constexpr int kClusterItems = 1024;          // items up to which the step runs as one cluster
constexpr int kMaxRounds = 16;
static_assert(kItemMax * 512 + 8 * (kHistBins / 2) * 4 <= 232448 - 6 * 1024, "accumulators and eight histograms");

// The launch's global scratch (words; zero when the state is reset).
struct Scratch {
  uint32_t arrivals, base;    // GridBarrier's count, and its value when a launch begins
  uint32_t start;             // the first round's histogram of the three
  uint32_t dead;              // a launch's wait gave up: later launches do nothing until the state is reset
  uint32_t pad[28];
  uint32_t listed[kMaxK];     // elements listed
  uint32_t reach[kMaxK];      // approximate top-s: elements that reach theta
  uint2 list[kMaxK][kListCap];
  uint32_t hist[1];                      // three of K * kHistWords, used in turn
};

// The search for the k-th element of one worker, the same in every block.
struct Search {
  uint32_t prefix;   // digits fixed so far: of the key, then of the inverted index
  int left;          // bits of the key (or, by_index, of the index) not fixed yet
  uint32_t rank;     // the element's 1-based rank among those with the prefix
  uint32_t count;    // elements with the prefix
  uint32_t T, t_idx; // the result: sent iff selected(key, j, T, t_idx)
  int mode;          // kDigit, kList or kDone
  int by_index;      // the key is fixed (T) and its ties are ranked by index
};
enum { kDigit = 0, kList = 1, kDone = 2 };

__device__ __forceinline__ int digit_width(int left) { return left < 11 ? left : 11; }
__device__ __forceinline__ uint32_t inv_index(uint32_t j) { return ((1u << kIdxBits) - 1) - j; }

// Sampled coordinates of the approximate top-s among a block of 8 from j (a
// multiple of 8): run r, one per stratum, starts at the multiple of 8 its draw picks.
__device__ __forceinline__ bool sampled_block(const TopkArgs& A, uint64_t key, uint32_t j) {
  if (A.d < 8) return true;
  const uint64_t n = A.n_sample >> 3, d = (uint64_t)A.d;
  const int64_t r0 = (int64_t)((uint64_t)j * n / d);
  for (int64_t r = r0 - 1; r <= r0 + 1; ++r) {
    if (r < 0 || r >= (int64_t)n) continue;
    const uint64_t lo = (uint64_t)r * d / n, hi = (uint64_t)(r + 1) * d / n;
    const uint64_t a = (lo + 7) & ~uint64_t(7);
    if (a + 8 * (uint64_t)below(draw(key, (uint64_t)r), (hi - a) >> 3) == j) return true;
  }
  return false;
}

// kCluster: the grid is one thread-block cluster (co-scheduled by the hardware),
// whose barrier takes the grid barrier's place and whose launch overlaps the end
// of the kernel before it, as a cooperative one does not: steps of up to
// kClusterItems items. Step and read of w, cluster against cooperative, us, at
// 256 items (K = 4) 21.2 / 24.6, 512 21.2 / 24.0, 1,024 20.9 / 24.2, 1,536 22.4 /
// 23.1 (K = 8: 24.5 / 23.8), 2,048 28.1 / 23.8, 4,096 41.2 / 24.7: past the line a
// cluster's 16 blocks have too much each.
template <bool kBf16, bool kCluster>
__global__ void __launch_bounds__(kSmThreads, 1) k_topk_step(TopkArgs A, DetachArgs D, Scratch* S, int hist_k) {
  if (kCluster) griddep_wait();
  const uint32_t dead = S->dead;
  if (A.hold_tile >= 0 && blockIdx.x == gridDim.x - 1) return;  // test hook: the other blocks' waits give up
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Search sr[kMaxK];
  __shared__ uint32_t cnt[kItemMax];            // per item: sent elements, then its pairs' first slot
  __shared__ uint32_t imax[kItemMax];           // per item: its largest key
  __shared__ uint16_t smask[kItemMax];          // approximate: sampled blocks of 8 of each own group
  __shared__ unsigned long long red[kSmWarps][5];
  __shared__ uint32_t s_ok, s_active, s_pairs;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int G = gridDim.x, me = blockIdx.x, K = A.K;
  const int n_groups = (int)((A.d + 127) >> 7);
  const int own = n_groups > me ? (n_groups - 1 - me) / G + 1 : 0;  // groups of this block
  const int items = own * K;
  float* vs = reinterpret_cast<float*>(smem);                       // items x 128
  // histograms of hist_k workers at a time, 16-bit counts (a block has under 2^16 values of a worker)
  uint32_t* hs = reinterpret_cast<uint32_t*>(smem + (size_t)kItemMaxBytes(n_groups, G, K));
  auto group_of = [&](int gi) { return me + gi * G; };
  const uint32_t lt = lanemask_lt();

  uint32_t buf = S->start;  // 0, 1 or 2
  GridBarrier grid{&S->arrivals, S->base, A.wait_ns, &s_ok};
  // every block's writes so far are seen by every block (false: a wait gave up)
  auto barrier = [&]() -> bool {
    if (!kCluster) return grid.wait();
    __syncwarp();  // (.aligned: a whole warp at once)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  };

  if (A.approx) {
    const uint64_t key = stream_key(A.seed, A.t, 0);
    for (int q = threadIdx.x; q < own * 16; q += kSmThreads) {
      const int gi = q >> 4, b = q & 15;
      const uint32_t j = (uint32_t)group_of(gi) * 128u + b * 8u;
      const bool in = j < (uint64_t)A.d && sampled_block(A, key, j);
      const uint32_t m = __ballot_sync(0xffffu << (lane & 16), in);  // a group's 16 lanes
      if (b == 0) smask[gi] = (uint16_t)((m >> (lane & 16)) & 0xffffu);
    }
  }
  // the first digit's histogram is counted while v is formed, when all the workers' fit
  const bool fused = hist_k >= K;
  if (fused)
    for (int q = threadIdx.x; q < K * (kHistBins / 2); q += kSmThreads) hs[q] = 0;
  __syncthreads();
  if (dead) return;  // (every block: set by a launch before, or by this one, whose waits then give up)
  if (me == 0 && threadIdx.x < kMaxK) {  // used after the first barrier
    if (threadIdx.x < 8) A.step_ctr->v[threadIdx.x] = 0ull;
    S->listed[threadIdx.x] = 0;
    S->reach[threadIdx.x] = 0;
    if ((int)threadIdx.x < K) A.sel[threadIdx.x].count = 0;
  }

  // ---- form v ----
  unsigned long long nonfinite = 0;
  constexpr int kU = 4;  // items a warp loads together
  for (int i0 = warp; i0 < items; i0 += kU * kSmWarps) {
    float4 ev[kU], gv[kU], dv[kU], mv[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = i0 + u * kSmWarps;
      if (i >= items) continue;
      const int gi = i / K, k = i - gi * K;
      const int64_t j = (int64_t)group_of(gi) * 128 + lane * 4;
      ev[u] = __ldcs(reinterpret_cast<const float4*>(A.e + (int64_t)k * A.ld + j));
      const float* gk = A.grads + (int64_t)k * A.d;
      gv[u] = kBf16 ? load_g4_bf16(A.grads16 + (int64_t)k * A.d, j, A.d) : load_g4(gk, j, A.d, g_mode(gk));
      dv[u] = *reinterpret_cast<const float4*>(A.dlt + j);
      if (A.local_mom) mv[u] = __ldcs(reinterpret_cast<const float4*>(A.lm + (int64_t)k * A.ld + j));
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = i0 + u * kSmWarps;
      if (i >= items) continue;
      const int gi = i / K, k = i - gi * K;
      const int64_t j = (int64_t)group_of(gi) * 128 + lane * 4;
      float4 g = gv[u];
      if (A.local_mom) {
        g.x = __fadd_rn(__fmul_rn(A.beta, mv[u].x), __fmul_rn(A.gs, g.x));
        g.y = __fadd_rn(__fmul_rn(A.beta, mv[u].y), __fmul_rn(A.gs, g.y));
        g.z = __fadd_rn(__fmul_rn(A.beta, mv[u].z), __fmul_rn(A.gs, g.z));
        g.w = __fadd_rn(__fmul_rn(A.beta, mv[u].w), __fmul_rn(A.gs, g.w));
        *reinterpret_cast<float4*>(A.lm + (int64_t)k * A.ld + j) = g;
      } else if (A.gscale) {
        g.x = __fmul_rn(A.gs, g.x);
        g.y = __fmul_rn(A.gs, g.y);
        g.z = __fmul_rn(A.gs, g.z);
        g.w = __fmul_rn(A.gs, g.w);
      }
      const float4 v = make_float4(accumulate(ev[u].x, g.x, A.c, dv[u].x), accumulate(ev[u].y, g.y, A.c, dv[u].y),
                                   accumulate(ev[u].z, g.z, A.c, dv[u].z), accumulate(ev[u].w, g.w, A.c, dv[u].w));
      *reinterpret_cast<float4*>(vs + (size_t)i * 128 + lane * 4) = v;
      const float x[4] = {v.x, v.y, v.z, v.w};
      const bool in = !A.approx || ((smask[gi] >> (lane >> 1)) & 1u);
      uint32_t most = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (j + c >= A.d) continue;
        nonfinite += is_nonfinite(x[c]) ? 1u : 0u;
        most = max(most, mag_key(x[c]));
        const uint32_t bin = mag_key(x[c]) >> 20;
        if (fused && in) atomicAdd(&hs[k * (kHistBins / 2) + (bin >> 1)], (bin & 1) ? 0x10000u : 1u);
      }
      most = __reduce_max_sync(0xffffffffu, most);
      if (lane == 0) imax[i] = most;
    }
  }
  // start of a search: the rank-th largest of all keys (or of the sampled ones)
  auto begin = [&](int k, uint32_t rank, uint32_t count) {
    Search& s = sr[k];
    s.prefix = 0;
    s.left = 31;
    s.rank = rank;
    s.count = count;
    s.T = s.t_idx = 0;
    s.mode = kDigit;
    s.by_index = 0;
  };
  if ((int)threadIdx.x < K) {
    if (A.approx) begin(threadIdx.x, min(A.sample_rank, A.n_sample), A.n_sample);
    else begin(threadIdx.x, A.ksel, (uint32_t)A.d);
  }

  bool ok = true;
  uint32_t fallbacks = 0;  // thread k: worker k's ties went to index digits, or it exceeded the limit
  // For the items of workers [k_lo, k_hi) that pass `want`: f(k, search, m, key, j)
  // with bit c of m set where value c belongs to the search and has its prefix.
  // Items whose largest key lies below the prefix are passed over: most, where
  // layers differ in scale.
  auto each_match = [&](int k_lo, int k_hi, bool sampled, auto&& want, auto&& f) {
    const int nk = k_hi - k_lo, dg = kSmWarps / nk, dk = kSmWarps - dg * nk;
    int gi = warp / nk, k = k_lo + warp % nk;
    while (gi < own) {
      const Search s = sr[k];
      if (want(s) && imax[gi * K + k] >= (s.by_index ? s.T : s.prefix << s.left)) {
        const float4 v = *reinterpret_cast<const float4*>(vs + (size_t)(gi * K + k) * 128 + lane * 4);
        const uint32_t key[4] = {mag_key(v.x), mag_key(v.y), mag_key(v.z), mag_key(v.w)};
        const uint32_t j = (uint32_t)group_of(gi) * 128u + lane * 4;
        uint32_t m = A.d - j >= 4 ? 0xfu : (A.d <= (int64_t)j ? 0u : (1u << (A.d - j)) - 1u);  // values below d
        if (sampled && !((smask[gi] >> (lane >> 1)) & 1u)) m = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const bool in = s.by_index ? key[c] == s.T && (inv_index(j + c) >> s.left) == s.prefix
                                     : (key[c] >> s.left) == s.prefix;
          if (!in) m &= ~(1u << c);
        }
        f(k, s, m, key, j);
      }
      gi += dg;
      k += dk;
      if (k >= k_hi) {
        k -= nk;
        ++gi;
      }
    }
  };
  // one batch of shared histograms into the global ones
  auto flush = [&](uint32_t* gh, int k_lo, int k_hi) {
    const int nw = (k_hi - k_lo) * (kHistBins / 2);
    __syncthreads();
    for (int q = threadIdx.x; q < nw; q += kSmThreads) {  // whole warps: nw is a multiple of 32
      const uint32_t word = hs[q];
      if (!__any_sync(0xffffffffu, word != 0)) continue;
      const int k = k_lo + q / (kHistBins / 2), bin = (q & (kHistBins / 2 - 1)) * 2;
      uint32_t sum = (word & 0xffffu) + (word >> 16);
      if (word & 0xffffu) atomicAdd(&gh[k * kHistWords + bin], word & 0xffffu);
      if (word >> 16) atomicAdd(&gh[k * kHistWords + bin + 1], word >> 16);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o, 16);  // 16 words: 32 bins
      if ((lane & 15) == 0 && sum) atomicAdd(&gh[k * kHistWords + kHistBins + (bin >> 5)], sum);
    }
  };
  // Run every worker's search (those not done yet) to its end.
  int round = 0;
  bool first = true;
  auto search = [&](bool sampled) {
    for (; round < kMaxRounds; ++round) {
      __syncthreads();
      uint32_t* gh = S->hist + buf * (uint32_t)(K * kHistWords);
      uint32_t* gz = S->hist + (buf + 1) % 3 * (uint32_t)(K * kHistWords);  // last read two rounds ago
      for (int q = me * kSmThreads + threadIdx.x; q < K * kHistWords; q += G * kSmThreads) gz[q] = 0;
      // elements with the prefix: into the list, or counted by the next digit --
      // straight into the global histogram when they are few
      const bool counted = round == 0 && fused && first;  // while v was formed
      const bool opening = round == 0;
      auto direct = [&](const Search& s) { return s.mode == kList || (s.mode == kDigit && s.count <= kDirect); };
      auto crowded = [&](const Search& s) { return s.mode == kDigit && (opening || s.count > kDirect); };
      if (counted) {
        flush(gh, 0, K);
      } else if (!opening) {
        each_match(0, K, sampled, direct, [&](int k, const Search& s, uint32_t m, const uint32_t (&key)[4], uint32_t j) {
          if (s.mode == kList) {
            if (!m) return;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              if (!((m >> c) & 1u)) continue;
              const uint32_t at = atomicAdd(&S->listed[k], 1u);
              if (at < (uint32_t)kListCap) S->list[k][at] = make_uint2(key[c], j + c);
            }
            return;
          }
          const int w = digit_width(s.left), sh = s.left - w;
          uint32_t* hk = gh + k * kHistWords;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t bin = ((s.by_index ? inv_index(j + c) : key[c]) >> sh) & ((1u << w) - 1);
            if ((m >> c) & 1u) {
              atomicAdd(hk + bin, 1u);
              atomicAdd(hk + kHistBins + (bin >> 5), 1u);
            }
          }
        });
      }
      for (int k_lo = 0; k_lo < K && !counted; k_lo += hist_k) {
        const int k_hi = min(K, k_lo + hist_k);
        bool any = false;
        for (int k = k_lo; k < k_hi; ++k) any |= crowded(sr[k]);
        if (!any) continue;
        __syncthreads();
        for (int q = threadIdx.x; q < (k_hi - k_lo) * (kHistBins / 2); q += kSmThreads) hs[q] = 0;
        __syncthreads();
        each_match(k_lo, k_hi, sampled, crowded, [&](int k, const Search& s, uint32_t m, const uint32_t (&key)[4], uint32_t j) {
          const int w = digit_width(s.left), sh = s.left - w;
          uint32_t* hk = hs + (k - k_lo) * (kHistBins / 2);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t bin = ((s.by_index ? inv_index(j + c) : key[c]) >> sh) & ((1u << w) - 1);
            if ((m >> c) & 1u) atomicAdd(hk + (bin >> 1), (bin & 1) ? 0x10000u : 1u);
          }
        });
        flush(gh, k_lo, k_hi);
      }
      ok = barrier();
      if (threadIdx.x == 0) s_active = 0;
      __syncthreads();
      if (!ok) return;
      // every block the same: a warp per worker
      for (int k = warp; k < K; k += kSmWarps) {
        Search s = sr[k];
        if (s.mode == kDone) continue;
        __syncwarp();
        if (s.mode == kList) {
          // at most kListCap elements, two a lane; the wanted one has rank - 1 before it
          uint2 a = make_uint2(0u, 0u), b = a;
          if ((uint32_t)lane < s.count) a = __ldcg(&S->list[k][lane]);
          if ((uint32_t)lane + 32 < s.count) b = __ldcg(&S->list[k][lane + 32]);
          uint32_t ra = 0, rb = 0;
          for (uint32_t q = 0; q < s.count; ++q) {
            const uint32_t ox = __shfl_sync(0xffffffffu, q < 32 ? a.x : b.x, q & 31);
            const uint32_t oy = __shfl_sync(0xffffffffu, q < 32 ? a.y : b.y, q & 31);
            ra += ox > a.x || (ox == a.x && oy < a.y);
            rb += ox > b.x || (ox == b.x && oy < b.y);
          }
          const uint32_t ma = __ballot_sync(0xffffffffu, (uint32_t)lane < s.count && ra == s.rank - 1);
          const uint32_t mb = __ballot_sync(0xffffffffu, (uint32_t)lane + 32 < s.count && rb == s.rank - 1);
          const int src = __ffs(ma ? ma : mb) - 1;
          s.T = __shfl_sync(0xffffffffu, ma ? a.x : b.x, src < 0 ? 0 : src);
          s.t_idx = __shfl_sync(0xffffffffu, ma ? a.y : b.y, src < 0 ? 0 : src);
          if (src < 0 && lane == 0) atomicOr(A.status, kStatusInternal);
          s.mode = kDone;
        } else {
          // from the top: the 32-bin sum that holds the rank, then the bin
          const uint32_t* hk = gh + k * kHistWords;
          const int w = digit_width(s.left);
          const uint32_t c1 = __ldcg(hk + kHistBins + 63 - lane), c2 = __ldcg(hk + kHistBins + 31 - lane);
          uint32_t i1 = c1, i2 = c2;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y1 = __shfl_up_sync(0xffffffffu, i1, o), y2 = __shfl_up_sync(0xffffffffu, i2, o);
            if (lane >= o) {
              i1 += y1;
              i2 += y2;
            }
          }
          const uint32_t t1 = __shfl_sync(0xffffffffu, i1, 31);
          i2 += t1;
          const uint32_t h1 = __ballot_sync(0xffffffffu, i1 >= s.rank), h2 = __ballot_sync(0xffffffffu, i2 >= s.rank);
          const int l1 = h1 ? __ffs(h1) - 1 : (h2 ? __ffs(h2) - 1 : 31);
          const int coarse = h1 ? 63 - l1 : 31 - l1;
          const uint32_t above1 = __shfl_sync(0xffffffffu, h1 ? i1 - c1 : i2 - c2, l1);
          const uint32_t f = __ldcg(hk + coarse * 32 + 31 - lane);
          uint32_t fi = f;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, fi, o);
            if (lane >= o) fi += y;
          }
          fi += above1;
          const uint32_t hf = __ballot_sync(0xffffffffu, fi >= s.rank);
          const int lf = hf ? __ffs(hf) - 1 : 31;
          if ((!hf || (!h1 && !h2)) && lane == 0) atomicOr(A.status, kStatusInternal);
          const uint32_t in_bin = __shfl_sync(0xffffffffu, f, lf), above = __shfl_sync(0xffffffffu, fi - f, lf);
          s.prefix = (uint32_t)(((uint64_t)s.prefix << w) | (uint32_t)(coarse * 32 + 31 - lf));
          s.left -= w;
          s.rank -= above;
          s.count = in_bin;
          if (sampled && s.left == 0) {  // theta: its whole key, every tie reaches it
            s.T = s.prefix;
            s.mode = kDone;
          } else if (!sampled && s.count <= s.rank) {  // every element with the prefix is sent
            if (s.by_index) s.t_idx = inv_index(s.prefix << s.left);
            else {
              s.T = s.prefix << s.left;
              s.t_idx = 0xffffffffu;
            }
            s.mode = kDone;
          } else if (s.count <= (uint32_t)kListCap) {
            s.mode = kList;
          } else if (s.left == 0 && !s.by_index) {  // the key is fixed: its ties by index
            s.T = s.prefix;
            s.prefix = 0;
            s.left = kIdxBits;
            s.by_index = 1;
          }
        }
        if (lane == 0) {
          sr[k] = s;
          if (s.mode != kDone) s_active = 1;
        }
      }
      __syncthreads();
      const bool active = s_active != 0;
      buf = (buf + 1) % 3;
      if (!active) {
        ++round;
        return;
      }
    }
    ok = false;  // not reached: a search ends within 3 key and 3 index digits and a list
    if (threadIdx.x == 0) atomicOr(A.status, kStatusInternal);
  };
  search(A.approx != 0);
  if (ok && A.approx) {
    // theta is known: count what reaches it
    __syncthreads();
    if ((int)threadIdx.x < K) sr[threadIdx.x].T = min(sr[threadIdx.x].T, 0x7f800000u);
    if ((int)threadIdx.x < K) cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int i = warp; i < items; i += kSmWarps) {
      const int gi = i / K, k = i - gi * K;
      const float4 v = *reinterpret_cast<const float4*>(vs + (size_t)i * 128 + lane * 4);
      const float x[4] = {v.x, v.y, v.z, v.w};
      const uint32_t j = (uint32_t)group_of(gi) * 128u + lane * 4;
      uint32_t n = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) n += (j + c < (uint64_t)A.d && mag_key(x[c]) >= sr[k].T) ? 1u : 0u;
      n = __reduce_add_sync(0xffffffffu, n);
      if (lane == 0 && n) atomicAdd(&cnt[k], n);
    }
    __syncthreads();
    if ((int)threadIdx.x < K && cnt[threadIdx.x]) atomicAdd(&S->reach[threadIdx.x], cnt[threadIdx.x]);
    ok = barrier();
    if (threadIdx.x == 0) s_active = 0;
    __syncthreads();
    if (ok) {
      if ((int)threadIdx.x < K) {
        sr[threadIdx.x].t_idx = 0xffffffffu;  // every tie is sent
        if (__ldcg(&S->reach[threadIdx.x]) > A.limit) {
          begin(threadIdx.x, A.limit, (uint32_t)A.d);
          fallbacks = 1;
          s_active = 1;
        }
      }
      if (me == 0 && threadIdx.x < kMaxK) S->listed[threadIdx.x] = 0;  // read by all before the barrier
      __syncthreads();
      if (s_active) {  // (as a step's first round: the lists are used after another barrier)
        round = 0;
        first = false;
        search(false);
      }
    }
  }
  if (!ok) {
    if (threadIdx.x == 0) {
      atomicOr(A.status, kStatusTimeout);
      S->dead = 1;
    }
    return;
  }
  if (me == 0) {
    if (threadIdx.x == 0) {
      S->start = buf;
      if (!kCluster) S->base = grid.reached;
    }
    if ((int)threadIdx.x < K) {
      WorkerSel& W = A.sel[threadIdx.x];
      const Search& s = sr[threadIdx.x];
      W.T = s.T;
      W.t_idx = s.t_idx;
      W.dense = 0;
      W.nsel = A.approx ? min(__ldcg(&S->reach[threadIdx.x]), A.limit) : A.ksel;
      fallbacks |= s.by_index;
      if (fallbacks) {
        atomicAdd(&A.step_ctr->v[kFallbacks], 1ull);
        atomicAdd(&A.total_ctr->v[kFallbacks], 1ull);
      }
    }
  }

  // ---- apply: a warp per group ----
  unsigned long long nnz = 0, uni = 0, changed = 0;
  for (int gi = warp; gi < own; gi += kSmWarps) {
    const int64_t g0 = (int64_t)group_of(gi) * 128, j = g0 + lane * 4;
    const int lim = A.d - g0 < 128 ? (int)(A.d - g0) : 128;
    const float4 w4 = *reinterpret_cast<const float4*>(A.w + j), d4 = *reinterpret_cast<const float4*>(A.dlt + j);
    float4 m4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (A.server_mom) m4 = *reinterpret_cast<const float4*>(A.mom + j);
    float sum[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t inU = 0;
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      float* vk = vs + (size_t)(gi * K + k) * 128 + lane * 4;
      const float4 v = *reinterpret_cast<const float4*>(vk);
      float en[4] = {v.x, v.y, v.z, v.w};
      const uint32_t T = sr[k].T, ti = sr[k].t_idx;
      if (imax[gi * K + k] < T) {  // nothing sent
        __stcs(reinterpret_cast<float4*>(A.e + (int64_t)k * A.ld + j), v);
        if (lane == 0) cnt[gi * K + k] = 0;
        continue;
      }
      uint32_t n = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (lane * 4 + c < lim && selected(mag_key(en[c]), (uint32_t)j + c, T, ti)) {
          sum[c] = __fadd_rn(sum[c], en[c]);
          nnz += en[c] != 0.f;
          inU |= 1u << c;
          en[c] = 0.f;
          ++n;
          if (A.mfm) A.lm[(int64_t)k * A.ld + j + c] = 0.f;  // momentum factor masking
        }
      }
      __stcs(reinterpret_cast<float4*>(A.e + (int64_t)k * A.ld + j), make_float4(en[0], en[1], en[2], en[3]));
      n = __reduce_add_sync(0xffffffffu, n);
      if (lane == 0) cnt[gi * K + k] = n;
    }
    float wo[4] = {w4.x, w4.y, w4.z, w4.w}, dd[4] = {0.f, 0.f, 0.f, 0.f};
    uni += __popc(inU);
    if (A.server_mom) {  // Alg. 3: w_{t+1} = (w_t - a*s) + beta*(w_t - w_{t-1}) everywhere
      const float mo[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (lane * 4 + c >= lim) continue;
        const float wn = __fadd_rn(__fsub_rn(wo[c], __fmul_rn(A.a, sum[c])), __fmul_rn(A.beta, mo[c]));
        dd[c] = __fsub_rn(wn, wo[c]);
        wo[c] = wn;
        changed += dd[c] != 0.f;
      }
      *reinterpret_cast<float4*>(A.w + j) = make_float4(wo[0], wo[1], wo[2], wo[3]);
      *reinterpret_cast<float4*>(A.mom + j) = make_float4(dd[0], dd[1], dd[2], dd[3]);
    } else {
      bool touch = (__float_as_uint(d4.x) | __float_as_uint(d4.y) | __float_as_uint(d4.z) | __float_as_uint(d4.w)) != 0u;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if ((inU >> c) & 1u) {
          const float wn = __fsub_rn(wo[c], __fmul_rn(A.a, sum[c]));
          A.w[j + c] = wn;
          dd[c] = __fsub_rn(wn, wo[c]);
          wo[c] = wn;
          changed += dd[c] != 0.f;
          touch = true;
        }
      }
      if (touch) *reinterpret_cast<float4*>(A.dlt + j) = make_float4(dd[0], dd[1], dd[2], dd[3]);
    }
    if (D.out) {  // GMC+ detach (Alg. 2): w_{t+1} - b*e_{t+1,k}
      for (int k = 0; k < K; ++k) {
        const float4 v = *reinterpret_cast<const float4*>(vs + (size_t)(gi * K + k) * 128 + lane * 4);
        const float en[4] = {v.x, v.y, v.z, v.w};
        float o[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          o[c] = __fsub_rn(wo[c], __fmul_rn(D.b, selected(mag_key(en[c]), (uint32_t)j + c, sr[k].T, sr[k].t_idx) ? 0.f : en[c]));
        store_row(D.out + (int64_t)k * D.out_ld + g0, lane * 4, lim, make_float4(o[0], o[1], o[2], o[3]), lane);
      }
    }
  }
  nnz = warp_sum(nnz);
  uni = warp_sum(uni);
  changed = warp_sum(changed);
  nonfinite = warp_sum(nonfinite);
  if (lane == 0) {
    red[warp][0] = nnz;
    red[warp][1] = uni;
    red[warp][2] = changed;
    red[warp][3] = nonfinite;
  }
  if (threadIdx.x == 0) s_pairs = 0;
  __syncthreads();

  // ---- the sent pairs: slots for this block's items, worker by worker ----
  for (int k = warp; k < K; k += kSmWarps) {
    uint32_t total = 0;
    for (int g = 0; g < own; g += 32) total += __reduce_add_sync(0xffffffffu, g + lane < own ? cnt[(g + lane) * K + k] : 0u);
    uint32_t base = 0;
    if (lane == 0 && total) {
      base = atomicAdd(&A.sel[k].count, total);
      atomicAdd(&s_pairs, total);
    }
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int g = 0; g < own; g += 32) {
      const uint32_t n = g + lane < own ? cnt[(g + lane) * K + k] : 0u;
      uint32_t incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (g + lane < own) {
        const int i = (g + lane) * K + k;
        // sub-chunk (worker, group): tiles are 8 groups
        A.chunk[(int64_t)group_of(g + lane) * K + k] = make_uint2(base + incl - n, n);
        cnt[i] = n ? base + incl - n : 0xffffffffu;
      }
      base += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
  __syncthreads();
  for (int i = warp; i < items; i += kSmWarps) {
    if (cnt[i] == 0xffffffffu) continue;
    const int gi = i / K, k = i - gi * K;
    const float4 v = *reinterpret_cast<const float4*>(vs + (size_t)i * 128 + lane * 4);
    const float x[4] = {v.x, v.y, v.z, v.w};
    const uint32_t j = (uint32_t)group_of(gi) * 128u + lane * 4;
    uint32_t m = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      m |= (j + c < (uint64_t)A.d && selected(mag_key(x[c]), j + c, sr[k].T, sr[k].t_idx) ? 1u : 0u) << c;
    uint32_t at = 0, n = __popc(m);
    // rank in index order: lanes before, then this lane's values
#pragma unroll
    for (int b = 0; b < 3; ++b) at += __popc(__ballot_sync(0xffffffffu, (n >> b) & 1u) & lt) << b;
    at += cnt[i];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (((m >> c) & 1u) && at < A.cap) {
        A.cand_idx[(int64_t)k * A.cap + at] = j + c;
        A.cand_val[(int64_t)k * A.cap + at] = x[c];
        ++at;
      }
    }
  }
  // ---- the step's counts, into its counters and the totals ----
  if (warp == 0) {
    unsigned long long c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) c[q] = warp_sum(lane < kSmWarps ? red[lane][q] : 0ull);
    if (lane < 2) {
      Counters* to = lane ? A.total_ctr : A.step_ctr;
      if (s_pairs) atomicAdd(&to->v[kPairs], (unsigned long long)s_pairs);
      if (c[0]) atomicAdd(&to->v[kNnz], c[0]);
      if (c[1]) atomicAdd(&to->v[kUnion], c[1]);
      if (c[2]) atomicAdd(&to->v[kChanged], c[2]);
      if (c[3]) {
        atomicAdd(&to->v[kNonfinite], c[3]);
        atomicOr(A.status, kStatusNonfinite);
      }
      if (me == 0) atomicAdd(&to->v[kSteps], 1ull);
    }
  }
}

// Shared memory: the accumulators, and as many workers' histograms as fit.
constexpr int kSmemMost = 232448 - 6 * 1024;  // 227 KB less the static part
int small_hist_k(int64_t d, int K, int grid) {
  const int room = kSmemMost - kItemMaxBytes((int)((d + 127) >> 7), grid, K);
  return std::min(K, room / (kHistBins / 2 * 4));
}

}  // namespace

// The one-launch step takes the problem: its accumulators fit in `grid` blocks.
// Returns the grid (0: it does not); *cluster: as one cluster.
int small_grid(int64_t d, int K, int num_sms, bool* cluster) {
  *cluster = false;
  if (d >= (int64_t(1) << kIdxBits)) return 0;
  const int64_t groups = (d + 127) / 128;
  if (groups * K <= kClusterItems) {
    int grid = 1;
    while (grid < kClusterMax && grid < groups) grid *= 2;
    *cluster = true;
    return grid;
  }
  const int grid = (int)std::min<int64_t>(groups, num_sms);
  const int64_t items = (groups + grid - 1) / grid * K;
  if (items > kItemMax) return 0;
  return grid;
}
size_t small_scratch_words(int K) {
  return sizeof(Scratch) / 4 + 3 * (size_t)K * kHistWords;
}
cudaError_t configure_small_kernels() {
  cudaError_t err = cudaSuccess;
  auto set = [&](const void* f, cudaFuncAttribute a, int v) {
    const cudaError_t e2 = cudaFuncSetAttribute(f, a, v);
    if (err == cudaSuccess) err = e2;
  };
  set((const void*)k_topk_step<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMost);
  set((const void*)k_topk_step<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMost);
  for (const void* f : {(const void*)k_topk_step<false, true>, (const void*)k_topk_step<true, true>}) {
    set(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMost);
    set(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  return err;
}
cudaError_t launch_topk_step(const TopkArgs& A, const DetachArgs& D, int grid, bool cluster, uint32_t* scratch,
                             cudaStream_t s) {
  if (refuse_cooperative()) return cudaErrorCooperativeLaunchTooLarge;
  const int hist_k = small_hist_k(A.d, A.K, grid);  // at least 8: kSmallItems leaves them room
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kSmThreads);
  cfg.dynamicSmemBytes = (size_t)kItemMaxBytes((int)((A.d + 127) >> 7), grid, A.K) + hist_k * (kHistBins / 2) * 4;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  cfg.attrs = at;
  Scratch* S = reinterpret_cast<Scratch*>(scratch);
  if (cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)grid;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, A.bf16 ? k_topk_step<true, true> : k_topk_step<false, true>, A, D, S, hist_k);
  }
  at[0].id = cudaLaunchAttributeCooperative;  // its blocks meet at grid barriers
  at[0].val.cooperative = 1;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, A.bf16 ? k_topk_step<true, false> : k_topk_step<false, false>, A, D, S, hist_k);
}

}  // namespace gmc
