// gmc_topk_noalloc: the top-k compressor of one vector, for callers that must
// not allocate device memory. Its scratch (histograms, the keys near the k-th,
// per-block counts) lives in one file-scope __device__ array of a fixed size
// instead of memory the library or the caller allocates. Every GPU that loads
// the library holds that array until the process exits.
//
// One cooperative launch, a block per SM. x is cut into chunks of 512 to 2,048
// values (up to 32,768 where only a few blocks may run), dealt to the blocks in turn (the selected values of a layered
// gradient lie close together: with a contiguous slice a block, one block wrote
// most of them), and within a block taken by the warps as they come:
//   sample   8,192 values a block (all of x up to 1.2 M): two radix digits of
//            the sampled keys give an interval of keys [L, U] that holds the
//            k-th largest key T but for about 1e-9 of inputs
//   collect  one pass over x: keys above U counted per chunk, keys inside listed
//            (key, index) and counted into a histogram over the interval; T is
//            the (k - above)-th largest of the list, found in its bin
//   write    a second pass, over the groups of 128 values that hold a key of the
//            interval or above it: the k pairs in index order, each chunk's
//            first position from the counts and the list
// An interval that missed T, or holds more keys than the list, is narrowed by
// histogram passes (2,048 bins each) until it holds T in a list or is one key
// (ties are then counted per warp). The selection is the library's top-k: the
// first k elements under (|x| bit pattern descending, index ascending).
//
// Bound by memory at the largest sizes (x is read once, and a fifth of it again
// at k = n/1000), by its four grid barriers below a few million values (n =
// 100,000: 40 us in seven launches -> 30). n = 25.6 M, k = n/1000: 304 us with five
// passes of 4-byte loads in seven launches -> 70 us (14 for the sample, 24 the
// pass over x, 15 ranking the list and the chunks' offsets in every block, 6 the
// write). Narrowing: all zeros or ties 299 -> 198 us, k = n 450 -> 182.
#include <atomic>
#include <cstddef>
#include <mutex>

#include "gmc.h"
#include "gmc_internal.h"

namespace gmc {
namespace {

constexpr int64_t kNoallocMaxN = int64_t(1) << 26;  // largest n accepted
constexpr int kNaThreads = 1024;
constexpr int kNaMaxDevices = 64;
constexpr int kNaMaxBlocks = 1024;
constexpr int kNaCap = 20480;    // listed keys (80 KB of shared memory to rank them)
constexpr int kNaChunks = 32768; // chunks of x at most
constexpr int kNaOwn = 1024;     // chunks of one block at most
constexpr int kNaStage = 2048;   // listed keys a block stages before it reserves their slots
constexpr int kNaRounds = 16;    // passes at most: a collect, then three histograms and a collect, with slack
constexpr int kNaUnroll = 4;     // groups of 128 values a warp loads together
constexpr int kNaQuads = 2;      // quads a thread samples
constexpr int kNaFew = 512;      // keys of T's histogram bin up to which each is compared with all
constexpr int kNaBatch = 8;      // listed keys a thread loads together
static_assert(kNaChunks * 2 <= kNaCap * 4, "the chunk counts fit in the keys' shared memory");
static_assert(kNaOwn == kNaThreads, "one thread per own chunk");
constexpr int64_t kNaBlockMin = 8192;  // values per block below which fewer blocks run

// The shared scratch, about 280 KB per device. A call begins with a memset of
// what comes before `above`, so that nothing an earlier call left behind (one
// whose waits gave up, or that overlapped another) reaches it; the rest is
// written before it is read.
struct NaScratch {
  uint32_t arrivals;                    // GridBarrier
  uint32_t pad[31];
  uint32_t count[kNaRounds];            // keys listed by each collect pass
  uint32_t hist[5][kHistBins];          // the sample's two digits; three in turn for the narrowing passes
  // per block: keys above the interval, and inside it. Two of each, used in turn:
  // a pass is separated from the one before by a single barrier, after which
  // some blocks still read that pass's counts while others write this one's
  uint32_t above[2][kNaMaxBlocks];
  uint32_t equal[2][kNaMaxBlocks];
  uint16_t above_c[kNaChunks];          // per chunk: keys above the interval
  union {
    struct {                            // the keys inside, and their indices
      uint32_t key[kNaCap], idx[kNaCap];
    } list;
    uint16_t equal_c[kNaChunks];        // per chunk: keys inside, when the interval is one key
  };
};
static __device__ __align__(256) NaScratch g_noalloc_scratch;

// Warp w's 128-value groups of x, lane l the values 4l .. 4l+3 of a group:
// magnitude keys, -1 outside [0, n). Groups start on 16 bytes: xa is x moved
// back to a 16-byte boundary by `off` values.
struct NaX {
  const float* xa;
  int64_t end;  // n + off
  int off;
  __device__ __forceinline__ float4 load(int64_t e) const {
    if (e >= off && e + 3 < end) return *reinterpret_cast<const float4*>(xa + e);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e >= off && e < end) v.x = xa[e];
    if (e + 1 >= off && e + 1 < end) v.y = xa[e + 1];
    if (e + 2 >= off && e + 2 < end) v.z = xa[e + 2];
    if (e + 3 >= off && e + 3 < end) v.w = xa[e + 3];
    return v;
  }
  __device__ __forceinline__ void keys(float4 v, int64_t e, int32_t (&k)[4]) const {
    k[0] = (int32_t)mag_key(v.x);
    k[1] = (int32_t)mag_key(v.y);
    k[2] = (int32_t)mag_key(v.z);
    k[3] = (int32_t)mag_key(v.w);
    if (e < off || e + 3 >= end) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (e + i < off || e + i >= end) k[i] = -1;
    }
  }
};

// The chunks of one block, taken by its warps as they come.
struct NaChunks {
  int64_t NG;      // groups of x
  int cg;          // groups per chunk: a power of two from 4
  int n_chunks, n_own;
  uint32_t me, G;
  uint32_t* claim;  // shared memory: own chunks taken
  // f(key[4], e, unit) for every group of the block's chunks (unit: the group's
  // sixteenth of its chunk), end(own, chunk) after each chunk.
  template <typename F, typename E>
  __device__ __forceinline__ void each(const NaX& X, int lane, F&& f, E&& end) const {
    __syncthreads();
    if (threadIdx.x == 0) *claim = 0;
    __syncthreads();
    const int ush = cg > 16 ? 31 - __clz(cg / 16) : 0;
    for (;;) {
      uint32_t o = 0;
      if (lane == 0) o = atomicAdd(claim, 1u);
      o = __shfl_sync(0xffffffffu, o, 0);
      if (o >= (uint32_t)n_own) break;
      const int c = (int)(me + o * G);
      const int64_t g0 = (int64_t)c * cg;
      const int gn = NG - g0 < cg ? (int)(NG - g0) : cg;
      for (int g = 0; g < gn; g += kNaUnroll) {
        float4 v[kNaUnroll];
#pragma unroll
        for (int u = 0; u < kNaUnroll; ++u)
          v[u] = g + u < gn ? X.load((g0 + g + u) * 128 + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kNaUnroll; ++u) {
          if (g + u < gn) {
            int32_t k[4];
            X.keys(v[u], (g0 + g + u) * 128 + lane * 4, k);
            f(k, (g0 + g + u) * 128 + lane * 4, (g + u) >> ush);
          }
        }
      }
      end((int)o, c);
    }
  }
};

__global__ void __launch_bounds__(kNaThreads, 1)
    k_na_topk(const float* __restrict__ x, int64_t n, uint32_t k, NaScratch* S, uint32_t* idx_out, float* val_out,
              uint64_t wait_ns, int leave) {
  if (leave && blockIdx.x == gridDim.x - 1) return;  // test hook: the others' waits give up
  extern __shared__ __align__(16) uint32_t na_keys[];  // kNaCap
  __shared__ uint32_t h[kHistBins];
  __shared__ uint2 stage[kNaStage];
  __shared__ uint32_t ws[32];
  __shared__ unsigned long long ws64[32];
  __shared__ uint32_t find[4];
  __shared__ uint16_t flag[kNaOwn];                    // own chunk: sixteenths with a key in or above the interval
  __shared__ uint32_t base_gt[kNaOwn], base_eq[kNaOwn];  // own chunk: keys above T, equal to T before it
  __shared__ uint32_t s_n, s_base, s_ok, s_bin, s_rank, s_claim;
  const int lane = threadIdx.x & 31;
  const uint32_t G = gridDim.x, me = blockIdx.x;
  NaX X;
  X.off = (int)((reinterpret_cast<uintptr_t>(x) >> 2) & 3u);
  X.xa = x - X.off;
  X.end = n + X.off;
  NaChunks C;
  C.NG = (X.end + 127) / 128;
  C.cg = 4;
  while ((C.NG + C.cg - 1) / C.cg > min((int64_t)kNaChunks, (int64_t)kNaOwn * G)) C.cg *= 2;
  C.n_chunks = (int)((C.NG + C.cg - 1) / C.cg);
  C.me = me;
  C.G = G;
  C.n_own = (uint32_t)C.n_chunks > me ? (int)((C.n_chunks - 1 - me) / G) + 1 : 0;
  C.claim = &s_claim;
  bool ok = true;
  GridBarrier grid{&S->arrivals, 0u, wait_ns, &s_ok};

  // A histogram in shared memory added to a global one, and read back after a barrier.
  auto share_hist = [&](uint32_t* gh) {
    __syncthreads();
    for (int b = threadIdx.x; b < kHistBins; b += kNaThreads)
      if (h[b]) atomicAdd(&gh[b], h[b]);
    const bool good = grid.wait();
    for (int b = threadIdx.x; b < kHistBins; b += kNaThreads) h[b] = __ldcg(&gh[b]);
    if (threadIdx.x < 4) find[threadIdx.x] = 0;
    __syncthreads();
    return good;
  };
  auto clear_hist = [&]() {
    __syncthreads();
    for (int b = threadIdx.x; b < kHistBins; b += kNaThreads) h[b] = 0;
    __syncthreads();
  };
  auto block_total = [&](uint32_t v) {
    uint32_t tot;
    block_inclusive_scan<uint32_t>(v, ws, &tot);
    return tot;
  };

  // ---- sample: kNaQuads quads a thread, evenly over x ----
  int32_t L = 0, U = 0x7fffffff;  // the interval: keys in [L, U]
  bool hist_next = false;
  {
    const int64_t nq = C.NG * 32, slots = (int64_t)G * kNaQuads * kNaThreads;
    int32_t sk[kNaQuads][4];
#pragma unroll
    for (int u = 0; u < kNaQuads; ++u) {
      const int64_t t = ((int64_t)u * G + me) * kNaThreads + threadIdx.x;
#pragma unroll
      for (int i = 0; i < 4; ++i) sk[u][i] = -1;
      if (t < nq) {
        const int64_t e = (nq <= slots ? t : (int64_t)((uint64_t)(t * nq) / (uint64_t)slots)) * 4;
        X.keys(X.load(e), e, sk[u]);
      }
    }
    clear_hist();
#pragma unroll
    for (int u = 0; u < kNaQuads; ++u)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (sk[u][i] >= 0) atomicAdd(&h[sk[u][i] >> 20], 1u);
    ok = share_hist(S->hist[0]);
    uint32_t mine = 0;
    for (int b = threadIdx.x; b < kHistBins; b += kNaThreads) mine += h[b];
    const uint32_t ns = block_total(mine);
    // the k-th key's expected rank in the sample, six standard deviations to
    // either side (exact when the sample is all of x)
    uint32_t r_lo = k, r_hi = k;
    if ((int64_t)ns < n) {
      // (in fp32: it only steers, and fp64 by every thread took 10 us)
      const float per = (float)n / (float)ns, r = (float)k / per;
      const float dev = 6.f * sqrtf(fmaxf(r * (1.f - r / (float)ns), 0.f)) + 8.f;
      r_lo = (uint32_t)fminf((float)ns, ceilf(r + dev));
      r_hi = r - dev >= 1.f ? min(r_lo, (uint32_t)(r - dev)) : 0u;
      hist_next = 2.f * dev * per > 0.95f * (float)kNaCap;  // more keys than the list takes
    }
    block_find2_from_top(h, kHistBins, r_lo, r_hi ? r_hi : r_lo, ws, find);
    const uint32_t b1 = find[0], rr1 = find[1], bh = find[2], rrh = find[3];
    const uint32_t n_h = bh != b1 ? h[bh] : 0u;
    clear_hist();
    // second digits: bin b1's in the lower half, bin bh's (when it is another) in the upper
#pragma unroll
    for (int u = 0; u < kNaQuads; ++u) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (sk[u][i] < 0) continue;
        const uint32_t bin = (uint32_t)sk[u][i] >> 20, dig = ((uint32_t)sk[u][i] >> 10) & 1023u;
        if (bin == b1) atomicAdd(&h[dig], 1u);
        else if (bin == bh) atomicAdd(&h[1024u + dig], 1u);
      }
    }
    ok = share_hist(S->hist[1]) && ok;
    block_find2_from_top(h, kHistBins, n_h + rr1, rrh, ws, find);
    L = (int32_t)((b1 << 20) | ((find[0] & 1023u) << 10));
    if (r_lo == ns && (int64_t)ns < n) L = 0;  // below every sampled key
    if (r_hi) U = (int32_t)((bh << 20) | ((find[2] & 1023u) << 10) | 1023u);
    else U = L < 0x7fffffff - (1 << 26) ? L + (1 << 26) : 0x7fffffff;  // eight octaves up
  }

  // ---- narrow the interval until T is known ----
  int32_t T = 0;
  uint32_t n_tie = 0;
  bool listed = false, found = false;
  uint32_t above = 0, in_list = 0;  // keys above the interval; keys listed
  bool know_above = false;          // `above` is that of [L, U]
  int hist_round = 0, sh = 0;       // histograms so far; log2 of the last one's bin width in keys
  for (int round = 0; ok && !found && round < kNaRounds; ++round) {
    uint32_t gt = 0, eq = 0;  // this warp's keys above and inside (collect: lane 0, per chunk in gc / ec)
    if (!hist_next) {
      // collect: count above, list inside (or count, when the interval is one key)
      const bool one = L == U;
      uint32_t gc = 0, ec = 0, units = 0;
      // the listed keys' histogram over the interval, for ranking them
      sh = 0;
      while (((uint32_t)(U - L) >> sh) >= (uint32_t)kHistBins) ++sh;
      uint32_t* gh = S->hist[2 + hist_round % 3];
      uint32_t* gz = S->hist[2 + (hist_round + 1) % 3];  // last read two histograms ago
      if (hist_round > 0)
        for (int b = me * kNaThreads + threadIdx.x; b < kHistBins; b += G * kNaThreads) gz[b] = 0;
      ++hist_round;
      clear_hist();
      if (threadIdx.x == 0) s_n = 0;
      C.each(
          X, lane,
          [&](const int32_t (&key)[4], int64_t e, int unit) {
            uint32_t in = 0, up = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              up += key[i] > U ? 1u : 0u;
              in |= (key[i] >= L && key[i] <= U ? 1u : 0u) << i;
            }
            if (!__any_sync(0xffffffffu, (up | in) != 0)) return;
            units |= 1u << unit;  // the write pass visits these groups
            gc += up;
            ec += __popc(in);
            if (one || !__any_sync(0xffffffffu, in != 0)) return;
            // slots for the warp's listed keys: staged; past the stage straight in
            // the list, unless that is full already (many ties: no slot matters then)
            uint32_t incl = __popc(in);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
              if (lane >= o) incl += y;
            }
            const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
            uint32_t at = 0, to = 0;
            if (lane == 0) {
              at = atomicAdd(&s_n, tot);
              if (at + tot > (uint32_t)kNaStage && __ldcg(&S->count[round]) < (uint32_t)kNaCap)
                to = atomicAdd(&S->count[round], min(tot, at + tot - (uint32_t)kNaStage));
              else
                to = (uint32_t)kNaCap;
            }
            const uint32_t first = __shfl_sync(0xffffffffu, at, 0);  // the warp's first slot
            to = __shfl_sync(0xffffffffu, to, 0);
            const uint32_t over = first > (uint32_t)kNaStage ? first : (uint32_t)kNaStage;  // slot of list entry `to`
            at = first + incl - __popc(in);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (!((in >> i) & 1u)) continue;
              if (at < (uint32_t)kNaCap) atomicAdd(&h[(uint32_t)(key[i] - L) >> sh], 1u);  // (past it the list is not used)
              const uint2 p = make_uint2((uint32_t)key[i], (uint32_t)(e + i - X.off));
              if (at < (uint32_t)kNaStage) {
                stage[at] = p;
              } else if (to + (at - over) < (uint32_t)kNaCap) {
                S->list.key[to + (at - over)] = p.x;
                S->list.idx[to + (at - over)] = p.y;
              }
              ++at;
            }
          },
          [&](int own, int c) {
            if (units) {
              gc = warp_sum(gc);
              ec = warp_sum(ec);
            }
            if (lane == 0) {
              S->above_c[c] = (uint16_t)gc;
              if (one) S->equal_c[c] = (uint16_t)ec;
              flag[own] = (uint16_t)units;
              gt += gc;
              eq += ec;
            }
            gc = ec = units = 0;
          });
      gt = block_total(gt);
      eq = block_total(eq);
      const uint32_t staged = min(s_n, (uint32_t)kNaStage);
      if (threadIdx.x == 0) {
        S->above[round & 1][me] = gt;
        S->equal[round & 1][me] = eq;
        s_base = (!one && staged) ? atomicAdd(&S->count[round], staged) : 0u;
      }
      __syncthreads();
      if (!one)
        for (uint32_t i = threadIdx.x; i < staged; i += kNaThreads) {
          if (s_base + i < (uint32_t)kNaCap) {
            S->list.key[s_base + i] = stage[i].x;
            S->list.idx[s_base + i] = stage[i].y;
          }
        }
      ok = share_hist(gh);
      know_above = true;
      const uint32_t a_all = block_total(threadIdx.x < G ? __ldcg(&S->above[round & 1][threadIdx.x]) : 0u);
      const uint32_t q_all = block_total(threadIdx.x < G ? __ldcg(&S->equal[round & 1][threadIdx.x]) : 0u);
      above = a_all;
      if (a_all >= k) {  // T lies above the interval
        L = U + 1;       // U < 2^31 - 1, since keys lie above it
        U = 0x7fffffff;
        above = 0;
        hist_next = true;
      } else if (a_all + q_all < k) {  // below it
        U = L - 1;
        L = 0;
        above = a_all + q_all;
        hist_next = true;
      } else if (one) {
        T = L;
        n_tie = k - a_all;
        found = true;
      } else if (q_all <= (uint32_t)kNaCap) {
        in_list = q_all;
        listed = found = true;
      } else {
        hist_next = true;
      }
      continue;
    }
    // histogram of the keys of [L, U] in bins of 2^sh keys (the first, on the
    // sampled interval, also counts the keys above it)
    uint32_t* gh = S->hist[2 + hist_round % 3];
    uint32_t* gz = S->hist[2 + (hist_round + 1) % 3];  // last read two histograms ago
    sh = 0;
    while (((uint32_t)(U - L) >> sh) >= (uint32_t)kHistBins) ++sh;
    clear_hist();
    C.each(
        X, lane,
        [&](const int32_t (&key)[4], int64_t, int) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            gt += key[i] > U ? 1u : 0u;
            const bool in = key[i] >= L && key[i] <= U;
            const uint32_t any = __ballot_sync(0xffffffffu, in);
            if (!any) continue;
            // the first lane's bin in one add (ties: the whole warp's), the others their own
            const int bin = in ? (int)((uint32_t)(key[i] - L) >> sh) : -1;
            const int lead = __ffs(any) - 1, b0 = __shfl_sync(0xffffffffu, bin, lead);
            const uint32_t same = __ballot_sync(0xffffffffu, bin == b0);
            if (lane == lead) atomicAdd(&h[b0], (uint32_t)__popc(same));
            else if (in && bin != b0) atomicAdd(&h[bin], 1u);
          }
        },
        [](int, int) {});
    if (hist_round > 0)
      for (int b = me * kNaThreads + threadIdx.x; b < kHistBins; b += G * kNaThreads) gz[b] = 0;
    ++hist_round;
    gt = block_total(gt);
    if (threadIdx.x == 0) S->above[round & 1][me] = gt;
    ok = share_hist(gh);
    if (!know_above) {
      know_above = true;
      above = block_total(threadIdx.x < G ? __ldcg(&S->above[round & 1][threadIdx.x]) : 0u);
      for (int b = threadIdx.x; b < kHistBins; b += kNaThreads) eq += h[b];
      eq = block_total(eq);
      if (above >= k) {  // T lies above the interval
        L = U + 1;
        U = 0x7fffffff;
        above = 0;
        continue;
      }
      if (above + eq < k) {  // below it
        U = L - 1;
        L = 0;
        above += eq;
        continue;
      }
    }
    block_find2_from_top(h, kHistBins, k - above, k - above, ws, find);
    const uint32_t bin = find[0], in_bin = h[bin];
    above = k - find[1];  // keys above the bin
    const int64_t lo = (int64_t)L + ((int64_t)bin << sh), hi = lo + (int64_t(1) << sh) - 1;
    L = (int32_t)lo;
    U = hi < U ? (int32_t)hi : U;
    hist_next = in_bin > (uint32_t)kNaCap && L != U;
    __syncthreads();
  }
  ok = ok && found;

  if (!ok) {
    // a wait gave up: no selection, and every index says so. (Blocks whose waits
    // all ended write their pairs meanwhile: what ends up with an index is one of
    // theirs, and valid; this block's pairs keep the mark.)
    for (uint32_t i = threadIdx.x; i < k; i += kNaThreads) idx_out[i] = kNone;
  } else {
    // ---- T from the list ----
    for (int o = threadIdx.x; o < kNaOwn; o += kNaThreads) base_gt[o] = base_eq[o] = 0;
    if (listed) {
      // h: the listed keys' histogram. The bin that holds T, and T's rank there
      block_find2_from_top(h, kHistBins, k - above, k - above, ws, find);
      const uint32_t bin = find[0], rank = find[1], in_bin = h[bin];
      const bool few = in_bin <= (uint32_t)kNaFew;
      if (threadIdx.x == 0) s_n = 0;
      if (!few) {
        // too many to compare with each other: all the listed keys ranked by radix digits
        for (uint32_t i0 = threadIdx.x; i0 < in_list; i0 += kNaBatch * kNaThreads) {
          uint32_t key[kNaBatch];
#pragma unroll
          for (int q = 0; q < kNaBatch; ++q) {
            const uint32_t i = i0 + q * kNaThreads;
            key[q] = i < in_list ? __ldcg(&S->list.key[i]) : 0u;
          }
#pragma unroll
          for (int q = 0; q < kNaBatch; ++q)
            if (i0 + q * kNaThreads < in_list) na_keys[i0 + q * kNaThreads] = key[q];
        }
        int bits = 0;
        while (bits < 31 && ((uint32_t)(U - L) >> bits) != 0) ++bits;
        __syncthreads();
        T = (int32_t)smem_select_bits(na_keys, in_list, k - above, bits, (uint32_t)L, h, ws, &s_bin, &s_rank, &n_tie);
      }
      __syncthreads();
      // one pass over the list: the keys known to be sent counted at the first own
      // chunk after theirs; those of T's bin set aside (kNaBatch loads in flight a thread)
      // (x / G as a product: exact, x < 2^15 and G <= 2^10)
      const uint32_t inv_G = (uint32_t)((0x100000000ull + G - 1) / G);
      const int cg_sh = 31 - __clz(C.cg);
      auto own_after = [&](uint32_t idx) {
        const uint32_t c = (idx + X.off) >> (7 + cg_sh);
        const int j = c < me ? 0 : (G > 1 ? (int)__umulhi(c - me, inv_G) : (int)(c - me)) + 1;
        return j < C.n_own ? j : -1;
      };
      for (uint32_t i0 = threadIdx.x & ~31u; i0 < in_list; i0 += kNaBatch * kNaThreads) {
        uint32_t key[kNaBatch], idx[kNaBatch];
#pragma unroll
        for (int q = 0; q < kNaBatch; ++q) {
          const uint32_t i = i0 + lane + q * kNaThreads;
          key[q] = i < in_list ? __ldcg(&S->list.key[i]) : 0u;
          idx[q] = i < in_list ? __ldcg(&S->list.idx[i]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < kNaBatch; ++q) {
          if (i0 + q * kNaThreads >= in_list) break;  // (uniform over the warp)
          const bool in = i0 + lane + q * kNaThreads < in_list;
          const uint32_t b = in ? (key[q] - (uint32_t)L) >> sh : 0u;
          const bool up = in && (few ? b > bin : (int32_t)key[q] > T);
          const bool aside = in && (few ? b == bin : (int32_t)key[q] == T);
          const int j = up ? own_after(idx[q]) : -1;
          // (most of a warp's keys often fall before one chunk: added at once)
          const uint32_t any = __ballot_sync(0xffffffffu, j >= 0);
          if (any) {
            const int lead = __ffs(any) - 1, j0 = __shfl_sync(0xffffffffu, j, lead);
            const uint32_t same = __ballot_sync(0xffffffffu, j == j0);
            if (lane == lead) atomicAdd(&base_gt[j0], (uint32_t)__popc(same));
            else if (j >= 0 && j != j0) atomicAdd(&base_gt[j], 1u);
          }
          if (aside) {
            if (few) {
              stage[atomicAdd(&s_n, 1u)] = make_uint2(key[q], idx[q]);
            } else {
              const int t = own_after(idx[q]);
              if (t >= 0) atomicAdd(&base_eq[t], 1u);
            }
          }
        }
      }
      __syncthreads();
      if (few) {  // T among its bin's few keys, each compared with all
        uint2 mine = make_uint2(0u, 0u);
        if (threadIdx.x < in_bin) {
          mine = stage[threadIdx.x];
          uint32_t gt = 0, eq = 0;
          for (uint32_t i = 0; i < in_bin; ++i) {
            gt += stage[i].x > mine.x ? 1u : 0u;
            eq += stage[i].x == mine.x ? 1u : 0u;
          }
          if (gt < rank && rank <= gt + eq) {  // (every key equal to T writes the same)
            s_bin = mine.x;
            s_rank = rank - gt;
          }
        }
        __syncthreads();
        T = (int32_t)s_bin;
        n_tie = s_rank;
        if (threadIdx.x < in_bin && (int32_t)mine.x >= T) {
          const int t = own_after(mine.y);
          if (t >= 0) atomicAdd((int32_t)mine.x > T ? &base_gt[t] : &base_eq[t], 1u);
        }
      }
    }
    __syncthreads();
    {  // sums over the own chunks before (one thread each): keys sent of the list
      unsigned long long tot;
      const int o = threadIdx.x;  // kNaOwn == kNaThreads
      const unsigned long long v = ((unsigned long long)base_gt[o] << 32) | base_eq[o];
      const unsigned long long p = block_inclusive_scan<unsigned long long>(v, ws64, &tot);
      base_gt[o] = (uint32_t)(p >> 32);
      base_eq[o] = (uint32_t)p;
    }
    __syncthreads();
    // and over all chunks before: a thread's run of chunks, then its own chunks in it
    for (int pass = 0; pass < (listed ? 1 : 2); ++pass) {
      const uint16_t* cnt = pass ? S->equal_c : S->above_c;
      uint32_t* base = pass ? base_eq : base_gt;
      constexpr int kPer = kNaChunks / kNaThreads;
      const int per = (C.n_chunks + kNaThreads - 1) / kNaThreads;  // at most kPer
      const int c0 = (int)threadIdx.x * per;
      // through shared memory (the keys' is free now), so that the lines are read once, whole
      uint16_t* cs = reinterpret_cast<uint16_t*>(na_keys);
      for (int i = threadIdx.x; i < (C.n_chunks + 7) / 8; i += kNaThreads)
        reinterpret_cast<uint4*>(cs)[i] = __ldcg(reinterpret_cast<const uint4*>(cnt) + i);
      __syncthreads();
      uint32_t v[kPer], mine = 0, tot;
#pragma unroll
      for (int i = 0; i < kPer; ++i) v[i] = i < per && c0 + i < C.n_chunks ? cs[c0 + i] : 0u;
#pragma unroll
      for (int i = 0; i < kPer; ++i) mine += v[i];
      uint32_t before = block_inclusive_scan<uint32_t>(mine, ws, &tot) - mine;
      // the first own chunk from c0 on
      uint32_t o = c0 <= (int)me ? 0u : ((uint32_t)c0 - me + G - 1) / G;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        if (i < per && c0 + i < C.n_chunks && (uint32_t)(c0 + i) == me + o * G) base[o++] += before;
        before += v[i];
      }
      __syncthreads();
    }
    // ---- write ----
    if (threadIdx.x == 0) s_claim = 0;
    __syncthreads();
    const int ush = C.cg > 16 ? 31 - __clz(C.cg / 16) : 0;
    for (;;) {
      uint32_t o = 0;
      if (lane == 0) o = atomicAdd(&s_claim, 1u);
      o = __shfl_sync(0xffffffffu, o, 0);
      if (o >= (uint32_t)C.n_own) break;
      const uint32_t units = flag[o];
      if (!units) continue;
      const int64_t g0 = (int64_t)(me + o * G) * C.cg;
      const int gn = C.NG - g0 < C.cg ? (int)(C.NG - g0) : C.cg;
      uint32_t gt_at = base_gt[o], eq_at = base_eq[o];  // sent keys above T, keys equal to T before the group
      int g = 0;
      while (g < gn) {
        float4 v[kNaUnroll];
        int gi[kNaUnroll];
#pragma unroll
        for (int u = 0; u < kNaUnroll; ++u) {  // the next groups of flagged sixteenths
          while (g < gn && !((units >> (g >> ush)) & 1u)) ++g;
          gi[u] = g < gn ? g++ : -1;
          v[u] = gi[u] >= 0 ? X.load((g0 + gi[u]) * 128 + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < kNaUnroll; ++u) {
          if (gi[u] < 0) continue;
          const int64_t e = (g0 + gi[u]) * 128 + lane * 4;
          int32_t key[4];
          X.keys(v[u], e, key);
          uint32_t cnt = 0;  // above T << 16 | equal to it
#pragma unroll
          for (int i = 0; i < 4; ++i) cnt += key[i] > T ? 0x10000u : (key[i] == T ? 1u : 0u);
          if (!__any_sync(0xffffffffu, cnt != 0)) continue;
          uint32_t incl = cnt;
#pragma unroll
          for (int s = 1; s < 32; s <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += y;
          }
          const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
          const uint32_t exc = incl - cnt;
          uint32_t ga = gt_at + (exc >> 16), ea = eq_at + (exc & 0xffffu);
          const float xv[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const bool tie = key[i] == T;
            if (key[i] > T || (tie && ea < n_tie)) {
              const uint32_t to = ga + min(ea, n_tie);
              if (to < k) {
                idx_out[to] = (uint32_t)(e + i - X.off);
                val_out[to] = xv[i];
              }
            }
            ga += key[i] > T ? 1u : 0u;
            ea += tie ? 1u : 0u;
          }
          gt_at += tot >> 16;
          eq_at += tot & 0xffffu;
        }
      }
    }
  }
}

// Set-up of one device: the scratch array's device address and the grid,
// valid for the CUDA context they were taken in.
struct DeviceSetup {
  unsigned long long ctx_id = 0;  // 0: not set up
  NaScratch* scratch = nullptr;
  int blocks = 1;                 // resident blocks of k_na_topk
};
// Test hook (gmc_test_leave_barrier): the next call's wait limit, 0 = off.
std::atomic<uint64_t> g_leave_ns{0};
std::mutex g_setup_mutex;
DeviceSetup g_setup[kNaMaxDevices];

using CtxGetCurrentFn = int (*)(void** ctx);
using CtxGetIdFn = int (*)(void* ctx, unsigned long long* id);

// Id of the current thread's CUDA context on the current device (the
// runtime's primary context, made current if it was not), through the driver
// entry points the runtime exposes. 0 on failure.
unsigned long long current_context_id(int dev) {
  static CtxGetCurrentFn get_current = nullptr;
  static CtxGetIdFn get_id = nullptr;
  if (!get_current || !get_id) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !f)
      return 0;
    get_current = reinterpret_cast<CtxGetCurrentFn>(f);
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !f)
      return 0;
    get_id = reinterpret_cast<CtxGetIdFn>(f);
  }
  void* ctx = nullptr;
  if (get_current(&ctx) != 0) return 0;
  if (!ctx) {  // the runtime has not made its context current on this thread yet
    if (cudaSetDevice(dev) != cudaSuccess || get_current(&ctx) != 0 || !ctx) return 0;
  }
  unsigned long long id = 0;
  return get_id(ctx, &id) == 0 ? id : 0;
}

// The scratch array's device address and the grid of the current device.
// Host code cannot use the array's name as a device address: the address is
// looked up with cudaGetSymbolAddress once per device, with that device
// current, and again only if the device's context was replaced since (e.g.
// after cudaDeviceReset), so that a stale address is never passed on.
cudaError_t device_setup(DeviceSetup* out) {
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (dev < 0 || dev >= kNaMaxDevices) return cudaErrorInvalidDevice;
  const unsigned long long ctx = current_context_id(dev);
  if (ctx == 0) return cudaErrorInitializationError;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  DeviceSetup& st = g_setup[dev];
  if (st.ctx_id != ctx) {
    void* p = nullptr;
    err = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (err != cudaSuccess) return err;
    int sms = 0, per_sm = 0;
    err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute((const void*)k_na_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, kNaCap * 4);
    if (err == cudaSuccess)
      err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_na_topk, kNaThreads, kNaCap * 4);
    if (err != cudaSuccess) return err;
    if (sms < 1 || per_sm < 1) return cudaErrorLaunchOutOfResources;
    st.scratch = static_cast<NaScratch*>(p);
    st.blocks = sms < kNaMaxBlocks ? sms : kNaMaxBlocks;
    st.ctx_id = ctx;
  }
  *out = st;
  return cudaSuccess;
}

}  // namespace

void noalloc_leave_barrier(uint64_t wait_limit_ns) { g_leave_ns.store(wait_limit_ns); }

}  // namespace gmc

extern "C" int gmc_topk_noalloc(const float* x_dev, int64_t n, int64_t k, uint32_t* idx_dev,
                                float* val_dev, void* stream) {
  using namespace gmc;
  if (!x_dev || !idx_dev || !val_dev || n < 1 || k < 1 || k > n) return GMC_EINVAL;
  if (n > kNoallocMaxN) return GMC_ETOOBIG;
  DeviceSetup dv;
  if (device_setup(&dv) != cudaSuccess) return GMC_ECUDA;
  // a block per SM, fewer where a block would have less than kNaBlockMin values
  const int64_t want = (n + kNaBlockMin - 1) / kNaBlockMin;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(want < dv.blocks ? want : dv.blocks));
  cfg.blockDim = dim3(kNaThreads);
  cfg.dynamicSmemBytes = kNaCap * 4;
  cfg.stream = static_cast<cudaStream_t>(stream);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;  // its blocks meet at grid barriers
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const uint64_t leave_ns = g_leave_ns.exchange(0);
  // the launch's own error: earlier, unrelated work's is neither read nor cleared
  cudaError_t err = cudaMemsetAsync(dv.scratch, 0, offsetof(NaScratch, above), cfg.stream);
  if (err != cudaSuccess) return GMC_ECUDA;
  // fewer blocks where the context may use fewer SMs than the device has, as long
  // as kNaOwn chunks of at most 2^15 values (16-bit counts) a block cover x
  const unsigned least = (unsigned)((n + 3 + kNaOwn * 32768ll - 1) / (kNaOwn * 32768ll));
  for (;;) {
    err = refuse_cooperative()
              ? cudaErrorCooperativeLaunchTooLarge
              : cudaLaunchKernelEx(&cfg, k_na_topk, x_dev, n, (uint32_t)k, dv.scratch, idx_dev, val_dev,
                                   leave_ns ? leave_ns : kWaitLimitNs, leave_ns ? 1 : 0);
    if (!too_large_here(err) || cfg.gridDim.x <= least) break;
    cudaGetLastError();  // this launch's
    cfg.gridDim.x = cfg.gridDim.x / 2 > least ? cfg.gridDim.x / 2 : least;
  }
  return err == cudaSuccess ? GMC_OK : GMC_ECUDA;
}
