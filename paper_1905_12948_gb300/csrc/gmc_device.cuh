// Device-side definitions shared by the GMC kernels: per-worker selection
// state, step counters, the fp32 accumulator operation, magnitude keys, and
// warp / block scan primitives.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace gmc {

constexpr uint32_t kKeyMask = 0x7fffffffu;   // |v| through its bit pattern
constexpr uint32_t kNoCandidate = 0xffffffffu; // threshold above every key
constexpr int kThreads = 256;                // block size of the streaming kernels
constexpr int kWarps = kThreads / 32;
constexpr int kSampleThreads = 1024;
constexpr int kSampleRun = 16;               // consecutive coordinates per sampled run (power of two):
                                             // 64 bytes of a row, one DRAM burst
constexpr int kSampleAll = 32768;            // d at or below which every element is sampled
constexpr int kSampleSlots = 32768;          // sampled positions per worker (= kSampleAll)
constexpr int kSampleChunks = kSampleSlots / kSampleRun;  // sampled runs per worker
static_assert((kSampleRun & (kSampleRun - 1)) == 0 && kSampleRun <= 32, "kSampleRun: a power of two, at most a warp");
constexpr int kHistBins = 2048;              // first radix digit: key bits 30..20
constexpr int kThetaBins = kHistBins + 2048;  // the approximate top-s sample's three digits
constexpr int kRelBins = 2048;               // bins of the candidates' relative histogram
constexpr int kBucketCap = 12288;            // candidates of one bin ranked in shared memory

// Per-worker top-k selection state, rewritten every step.
struct WorkerSel {
  uint32_t theta;    // candidate threshold key from the sample (kNoCandidate = none)
  uint32_t count;    // candidates appended by the accumulate pass (may exceed cap)
  uint32_t prefix;   // approximate top-s: theta's digits found so far
  uint32_t rank;     // and its 1-based rank among the sampled keys with that prefix
  uint32_t T;        // the k-th largest key
  uint32_t n_tie;    // elements equal to T that are kept (lowest indices first)
  uint32_t ties;     // candidates equal to T
  uint32_t t_idx;    // a candidate equal to T is kept iff its index <= t_idx
  uint32_t dense;    // 1: this worker's selection is made by the dense path
  uint32_t done[4];  // finished-block counters: -, the select finish, the approximate
                     // top-s threshold's pass, and (worker 0's) the dense select's blocks
  uint32_t count_bucket;  // candidates collected from the k-th key's bin
  uint32_t nsel;     // approximate top-s: components sent (the count varies by step)
  uint32_t shift;    // log2 of the relative histogram's bin width, in keys (from the sample)
};

// Step counters (see GMC_STAT_* in gmc.h), unsigned 64-bit slots.
struct Counters {
  unsigned long long v[8];
};
enum CounterSlot { kSteps = 0, kPairs = 1, kNnz = 2, kUnion = 3, kChanged = 4,
                   kFallbacks = 5, kNonfinite = 6 };
// The end of a step (a whole warp, after every kernel of the step that counts):
// the pairs counted on the host, the step mark, and the step into the totals, a
// lane per counter. The step's counts may come from other blocks of the calling
// kernel: they are read from L2.
__device__ __forceinline__ void finalize_counters(Counters* step, Counters* total,
                                                  unsigned long long pairs_add) {
  const int i = (int)(threadIdx.x & 31);
  if (i >= 8) return;
  unsigned long long x = __ldcg(&step->v[i]);
  if (i == kPairs) x += pairs_add;
  if (i == kSteps) x = 1;
  if (i == kPairs || i == kSteps) step->v[i] = x;
  total->v[i] += x;
}

// Device status bits (gmc_check).
constexpr unsigned kStatusNonfinite = 1u;
constexpr unsigned kStatusInternal = 2u;
constexpr unsigned kStatusTimeout = 4u;     // a bounded wait gave up (see wait_bounded): tiles were skipped
constexpr int kChunksPerTile = 8;           // candidate sub-chunks per tile: one per warp
constexpr uint32_t kNone = 0xffffffffu;     // no coordinate

__device__ __forceinline__ uint32_t mag_key(float v) {
  return __float_as_uint(v) & kKeyMask;
}
__device__ __forceinline__ bool is_nonfinite(float v) {
  return (__float_as_uint(v) & 0x7f800000u) == 0x7f800000u;
}
// e_{t+1/2} = (e + g) - (c * dl): three operations, each rounded once (Alg. 1).
__device__ __forceinline__ float accumulate(float e, float g, float c, float dl) {
  return __fsub_rn(__fadd_rn(e, g), __fmul_rn(c, dl));
}
// The dense path decides this worker's C(v) when its sampled filter missed:
// fewer candidates than k, a candidate region overflowed, or too many ties.
__device__ __forceinline__ bool needs_dense(const WorkerSel& s, uint32_t ksel, uint32_t cap) {
  return s.count < ksel || s.count > cap || s.dense != 0;
}
// bfloat16 gradients: the upper 16 bits of an fp32 pattern, widened exactly.
__device__ __forceinline__ float bf16_f32(uint32_t b) { return __uint_as_float(b << 16); }
// Four consecutive bf16 values at p (2-byte aligned, shared or global memory).
__device__ __forceinline__ float4 bf16x4(const uint16_t* p) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  uint32_t lo, hi;
  if ((a & 7) == 0) {
    const uint2 x = *reinterpret_cast<const uint2*>(p);
    lo = x.x;
    hi = x.y;
  } else if ((a & 3) == 0) {
    lo = *reinterpret_cast<const uint32_t*>(p);
    hi = *reinterpret_cast<const uint32_t*>(p + 2);
  } else {
    lo = (uint32_t)p[0] | ((uint32_t)p[1] << 16);
    hi = (uint32_t)p[2] | ((uint32_t)p[3] << 16);
  }
  return make_float4(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u),
                     __uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
}
// Elements j .. j+3 of a bf16 row of d, zeros past d.
__device__ __forceinline__ float4 load_g4_bf16(const uint16_t* g, int64_t j, int64_t d) {
  if (j + 3 < d) return bf16x4(g + j);
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  if (j < d) r.x = bf16_f32(g[j]);
  if (j + 1 < d) r.y = bf16_f32(g[j + 1]);
  if (j + 2 < d) r.z = bf16_f32(g[j + 2]);
  return r;
}

// Elements j .. j+3 of an fp32 row of d, zeros past d; mode: g_mode of the row.
// (Not __restrict__: the kernel that writes the row may end only after this one began.)
__device__ __forceinline__ float4 load_g4(const float* g, int64_t j, int64_t d, int mode) {
  if (j + 3 < d) {
    if (mode == 4) return __ldcs(reinterpret_cast<const float4*>(g + j));
    if (mode == 2) {
      const float2 a = __ldcs(reinterpret_cast<const float2*>(g + j));
      const float2 b = __ldcs(reinterpret_cast<const float2*>(g + j + 2));
      return make_float4(a.x, a.y, b.x, b.y);
    }
    return make_float4(__ldcs(g + j), __ldcs(g + j + 1), __ldcs(g + j + 2), __ldcs(g + j + 3));
  }
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  if (j < d) r.x = g[j];
  if (j + 1 < d) r.y = g[j + 1];
  if (j + 2 < d) r.z = g[j + 2];
  return r;
}

__device__ __forceinline__ int g_mode(const float* p) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  return (a & 15) == 0 ? 4 : ((a & 7) == 0 ? 2 : 1);
}

// One group of 128 consecutive floats of a warp (lane l: elements 4l .. 4l+3)
// stored at p, any 4-byte alignment: 16-byte stores of the aligned quads, each
// made of its own and the next lane's values, and single floats at both ends.
// mis: floats from p to the next 16-byte boundary (uniform over the warp).
__device__ __forceinline__ void store_row128(float* p, float4 x, int mis, int lane) {
  if (mis == 0) {
    __stcs(reinterpret_cast<float4*>(p + lane * 4), x);
    return;
  }
  float4 n;  // the next lane's values
  n.x = __shfl_down_sync(0xffffffffu, x.x, 1);
  n.y = __shfl_down_sync(0xffffffffu, x.y, 1);
  n.z = __shfl_down_sync(0xffffffffu, x.z, 1);
  const float4 q = mis == 1 ? make_float4(x.y, x.z, x.w, n.x)
                            : (mis == 2 ? make_float4(x.z, x.w, n.x, n.y) : make_float4(x.w, n.x, n.y, n.z));
  if (lane < 31) __stcs(reinterpret_cast<float4*>(p + lane * 4 + mis), q);
  if (lane == 0) {
    p[0] = x.x;
    if (mis > 1) p[1] = x.y;
    if (mis > 2) p[2] = x.z;
  }
  if (lane == 31) {  // the elements past the last whole quad
    p[127] = x.w;
    if (mis < 3) p[126] = x.z;
    if (mis < 2) p[125] = x.y;
  }
}
__device__ __forceinline__ int row_mis(const float* p) {
  return (int)((4u - (uint32_t)(reinterpret_cast<uintptr_t>(p) >> 2)) & 3u);
}
// A lane's 4 elements at offset l of a sub-tile with lim valid elements, at row.
__device__ __forceinline__ void store_row(float* row, int l, int lim, float4 x, int lane) {
  // l - lane*4: the start of the warp's 128 elements
  const int g0 = l - lane * 4;
  if (g0 + 128 <= lim) {
    store_row128(row + g0, x, row_mis(row + g0), lane);
    return;
  }
  if (l < lim) row[l] = x.x;
  if (l + 1 < lim) row[l + 1] = x.y;
  if (l + 2 < lim) row[l + 2] = x.z;
  if (l + 3 < lim) row[l + 3] = x.w;
}

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014): output function, the key of
// step t's stream (stream 0 = shared by all workers, k+1 = worker k), the
// stream's i-th draw, and [0, n) from a draw's top 32 bits by multiply-shift.
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
__device__ __forceinline__ uint64_t sm64_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ uint64_t stream_key(uint64_t seed, int64_t t, uint64_t stream) {
  const uint64_t k1 = sm64_mix(seed + kGamma * (uint64_t)(t + 1));
  return sm64_mix(k1 + kGamma * (stream + 1));
}
__device__ __forceinline__ uint64_t draw(uint64_t key, uint64_t i) {
  return sm64_mix(key + kGamma * (i + 1));
}
__device__ __forceinline__ uint32_t below(uint64_t x, uint64_t n) {
  return (uint32_t)(((x >> 32) * n) >> 32);
}
__device__ __forceinline__ uint32_t warp_excl_scan(uint32_t x, uint32_t* total) {
  const int lane = threadIdx.x & 31;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  *total = __shfl_sync(0xffffffffu, incl, 31);
  return incl - x;
}
// Membership of a candidate in C(v): above the k-th key, or equal to it with
// an index no larger than the last tie kept (ties go to the lower index).
__device__ __forceinline__ bool selected(uint32_t key, uint32_t j, uint32_t T, uint32_t t_idx) {
  return key > T || (key == T && j <= t_idx);
}
// Shared-memory histogram increment, aggregated over the lanes of a warp that
// hit the same bucket (all lanes of the warp must call it; inactive: bin < 0).
__device__ __forceinline__ void warp_hist_add(uint32_t* hist, int bin) {
  const uint32_t peers = __match_any_sync(0xffffffffu, bin);
  const int leader = __ffs(peers) - 1;
  if (bin >= 0 && (int)(threadIdx.x & 31) == leader) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
}
// Sum over the 32 lanes of a warp (all lanes must call it).
template <typename V>
__device__ __forceinline__ V warp_sum(V x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Inclusive scan of one value per thread over the block (blockDim a multiple
// of 32, at most 1024). `ws` needs 32 words of shared memory. Returns the
// inclusive prefix; *total receives the block total.
template <typename V>
__device__ __forceinline__ V block_inclusive_scan(V x, V* ws, V* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    V y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  if (warp == 0) {
    V w = lane < nwarps ? ws[lane] : V(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      V y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    ws[lane] = w;  // inclusive warp-total prefix
  }
  __syncthreads();
  V add = warp > 0 ? ws[warp - 1] : V(0);
  V tot = ws[nwarps - 1];
  __syncthreads();  // ws may be reused by the caller
  *total = tot;
  return x + add;
}

// Given a histogram hist[nbins] (shared memory) of keys and a 1-based rank r
// counted from the largest key, find the bucket b that holds the r-th largest
// key and the rank of that key inside b. nbins must be a multiple of
// blockDim.x. All threads receive the result.
__device__ __forceinline__ void block_find_from_top(const uint32_t* hist, int nbins, uint32_t r,
                                                    uint32_t* ws, uint32_t* out_bin,
                                                    uint32_t* out_rank) {
  const int per = nbins / blockDim.x;
  // thread t owns buckets [nbins - (t+1)*per, nbins - t*per): thread 0 the top ones
  const int hi = nbins - threadIdx.x * per;
  uint32_t mine = 0;
  for (int i = 1; i <= per; ++i) mine += hist[hi - i];
  uint32_t total;
  uint32_t incl = block_inclusive_scan<uint32_t>(mine, ws, &total);
  uint32_t above = incl - mine;  // keys in buckets above mine
  if (above < r && r <= incl) {
    for (int i = 1; i <= per; ++i) {
      const uint32_t h = hist[hi - i];
      if (r <= above + h) {
        *out_bin = uint32_t(hi - i);
        *out_rank = r - above;
        break;
      }
      above += h;
    }
  }
  __syncthreads();
}

// The same for two ranks at once (one scan): out[0], out[1] = bin and rank of
// the r0-th, out[2], out[3] of the r1-th largest key (out: shared memory).
__device__ __forceinline__ void block_find2_from_top(const uint32_t* hist, int nbins, uint32_t r0, uint32_t r1,
                                                     uint32_t* ws, uint32_t* out) {
  const int per = nbins / blockDim.x;
  const int hi = nbins - threadIdx.x * per;
  uint32_t mine = 0;
  for (int i = 1; i <= per; ++i) mine += hist[hi - i];
  uint32_t total;
  const uint32_t incl = block_inclusive_scan<uint32_t>(mine, ws, &total);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const uint32_t r = q ? r1 : r0;
    uint32_t above = incl - mine;
    if (above < r && r <= incl) {
      for (int i = 1; i <= per; ++i) {
        const uint32_t h = hist[hi - i];
        if (r <= above + h) {
          out[2 * q] = uint32_t(hi - i);
          out[2 * q + 1] = r - above;
          break;
        }
        above += h;
      }
    }
  }
  __syncthreads();
}

// The same for any power-of-two nbins, also fewer bins than threads (a thread
// owns at most max(1, nbins / blockDim.x) of them; the others none).
__device__ __forceinline__ void block_find_from_top_any(const uint32_t* hist, int nbins, uint32_t r,
                                                        uint32_t* ws, uint32_t* out_bin,
                                                        uint32_t* out_rank) {
  const int per = nbins >= (int)blockDim.x ? nbins / (int)blockDim.x : 1;
  const int hi = nbins - (int)threadIdx.x * per;  // this thread's bins: [hi - per, hi), none when hi <= 0
  uint32_t mine = 0;
  for (int i = 1; i <= per && hi - i >= 0; ++i) mine += hist[hi - i];
  uint32_t total;
  const uint32_t incl = block_inclusive_scan<uint32_t>(mine, ws, &total);
  uint32_t above = incl - mine;
  if (above < r && r <= incl) {
    for (int i = 1; i <= per && hi - i >= 0; ++i) {
      const uint32_t h = hist[hi - i];
      if (r <= above + h) {
        *out_bin = uint32_t(hi - i);
        *out_rank = r - above;
        break;
      }
      above += h;
    }
  }
  __syncthreads();
}

// Radix select in shared memory over values below 2^bits (bits <= 31), taken
// relative to `base` (x[i] - base): digits of at most 11 bits from the top.
// Returns base + the r-th largest; rank_out = its rank among the values equal
// to it. With bits = 31 and base = 0 this is a select over whole keys.
__device__ __forceinline__ uint32_t smem_select_bits(const uint32_t* x, uint32_t n, uint32_t r, int bits,
                                                     uint32_t base, uint32_t* h, uint32_t* ws,
                                                     uint32_t* s_bin, uint32_t* s_rank, uint32_t* rank_out) {
  uint32_t prefix = 0;  // the digits fixed so far
  int done = 0;         // bits fixed so far (from the top)
  while (done < bits) {
    const int width = min(11, bits - done), shift = bits - done - width, nbins = 1 << width;
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) h[b] = 0;
    if (threadIdx.x == 0) {
      *s_bin = 0;
      *s_rank = 0;
    }
    __syncthreads();
    for (uint32_t i0 = 0; i0 < n; i0 += blockDim.x) {
      const uint32_t i = i0 + threadIdx.x;
      if (i < n) {
        const uint32_t v = x[i] - base;
        // the digits above this one must match the prefix (a shift by 32 is
        // avoided: no digit is fixed before the first pass)
        if (done == 0 || (v >> (shift + width)) == prefix) atomicAdd(&h[(v >> shift) & (uint32_t)(nbins - 1)], 1u);
      }
    }
    __syncthreads();
    block_find_from_top_any(h, nbins, r, ws, s_bin, s_rank);
    prefix = (prefix << width) | *s_bin;
    r = *s_rank;
    done += width;
    __syncthreads();
  }
  *rank_out = r;
  return base + prefix;
}

// Radix select in shared memory: the r-th largest of n values (digits 11/10/10).
__device__ __forceinline__ uint32_t smem_select(const uint32_t* x, uint32_t n, uint32_t r,
                                                uint32_t* h, uint32_t* ws, uint32_t* s_bin,
                                                uint32_t* s_rank, uint32_t* rank_out) {
  uint32_t prefix = 0;
  for (int pass = 0; pass < 3; ++pass) {
    const int nbins = pass == 0 ? 2048 : 1024;
    const int shift = pass == 0 ? 20 : (pass == 1 ? 10 : 0);
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) h[b] = 0;
    if (threadIdx.x == 0) {
      *s_bin = 0;
      *s_rank = 0;
    }
    __syncthreads();
    for (uint32_t i0 = 0; i0 < n; i0 += blockDim.x) {
      const uint32_t i = i0 + threadIdx.x;
      int bin = -1;
      if (i < n) {
        const uint32_t v = x[i];
        if (pass == 0 || (v >> (shift + 10)) == prefix) bin = (int)((v >> shift) & (uint32_t)(nbins - 1));
      }
      if (bin >= 0) atomicAdd(&h[bin], 1u);  // plain atomics measured faster than match_any here
    }
    __syncthreads();
    block_find_from_top(h, nbins, r, ws, s_bin, s_rank);
    prefix = pass == 0 ? *s_bin : ((prefix << 10) | *s_bin);
    r = *s_rank;
    __syncthreads();
  }
  *rank_out = r;
  return prefix;
}

// ---------------------------------------------------------------------------
// mbarrier and bulk-copy primitives (inline PTX, sm_90+ / sm_103a)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;"
               ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bound of every mbarrier wait of the bulk passes (a test may shorten it for
// one step), and of the wait for a CTA's own copies in flight before it exits.
constexpr uint64_t kWaitLimitNs = 2000000000ull;
// Wait for the phase with the given parity to complete, giving up after
// limit_ns (returns false): a wait never hangs the GPU.
__device__ __forceinline__ bool wait_bounded(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_ns() - t0 > limit_ns) return false;
  }
  return true;
}
// Programmatic dependent launch: a step's kernels are launched with
// programmatic stream serialization, so one may be scheduled while the one
// before it finishes; each waits here, before it touches memory, until its
// predecessor's writes are visible. Without that launch attribute it returns
// at once.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Barriers of a cooperative launch (every block resident): one word counts the
// blocks' arrivals and is never put back. The launch's b-th barrier ends when the
// count has grown by b * gridDim.x since the launch began, told by the sign of
// the difference, so that the word may wrap. An arrival needs no answer (a
// reduction with release), so a barrier costs the word's way to L2 and back once,
// for the blocks that poll it. A wait is bounded: wait() is false, for the whole
// block, when it gave up, and from then on (the block does not arrive again: it
// would stand for the one that is missing). The count then no longer matches what
// the next launch expects: it must be cleared first.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
struct GridBarrier {
  uint32_t* count;    // arrivals
  uint32_t reached;   // what the count has reached after the barriers passed so far (at launch: its value)
  uint64_t limit_ns;
  uint32_t* s_ok;     // a word of shared memory
  bool alive = true;  // no wait gave up yet
  __device__ __forceinline__ bool wait() {
    if (!alive) return false;
    reached += gridDim.x;
    __syncthreads();
    if (gridDim.x == 1) return true;
    if (threadIdx.x == 0) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
      uint64_t since = 0;
      bool here = false;
      for (uint32_t polls = 1; !(here = (int32_t)(ld_acquire(count) - reached) >= 0); ++polls) {
        if (polls & 1023u) continue;  // the clock now and then
        const uint64_t now = global_ns();
        if (since == 0) since = now;
        if (now - since > limit_ns) break;
      }
      *s_ok = here ? 1u : 0u;
    }
    __syncthreads();
    return alive = *s_ok != 0u;
  }
};
// Tiles of a persistent streaming pass. A CTA's first kFixed tiles are fixed,
// blockIdx.x + n * gridDim.x; every later one is claimed from a counter that
// the step's previous kernel zeroed, kFixed - 1 tiles before the CTA starts
// it, so that a CTA whose streams run faster takes more tiles and all of them
// finish together. The CTA's producer thread, when it starts its tile n,
// publishes the claim it made at tile n - 1 (for tile n - 1 + kFixed) in
// tq[(n - 1 + kFixed) % kQ], and then claims the next one; a thread reads
// tq[m % kQ] only after it has synchronised with the producer's start of tile
// m + 1 - kFixed. kQ must exceed the tiles between the oldest slot a thread
// may still read and the newest the producer may write.
// The number of fixed tiles may also be chosen at run time (uniform over the
// grid): tile_at_n / tile_claim_n.
template <int kQ>
__device__ __forceinline__ int64_t tile_at_n(const uint32_t* tq, uint32_t n, uint32_t fixed) {
  return n < fixed ? (int64_t)blockIdx.x + (int64_t)n * gridDim.x : (int64_t)tq[n % kQ];
}
// The order in which a pass visits its tiles, in blocks of G = gridDim.x
// consecutive tiles: the i-th tile claimed is order[i / G] * G + i mod G over
// the nb = n_tiles / G whole blocks (the partial block at the end stays last;
// order: a permutation of [0, nb), or NULL for index order; i >= n_tiles: past
// the last, unchanged). Within a block consecutive tiles still go to
// different CTAs at about the same time, so a layer's tiles spread over the
// CTAs' candidate parts as in index order.
__device__ __forceinline__ int64_t tile_order(int64_t i, int64_t n_tiles, const uint32_t* order) {
  if (i >= n_tiles || !order) return i;
  const uint32_t G = gridDim.x, nb = (uint32_t)(n_tiles / G);
  if ((uint64_t)i >= (uint64_t)nb * G) return i;
  const uint32_t b = (uint32_t)i / G, o = (uint32_t)i - b * G;
  // (constant for the kernel's life: k_sample_pending, two kernels or more ahead,
  // ended before the kernel between them did, and this one began after that)
  const uint32_t ob = __ldg(order + b);
  return (int64_t)(ob < nb ? ob : b) * G + o;
}
template <int kFixed, int kQ>
__device__ __forceinline__ int64_t tile_at(const uint32_t* tq, uint32_t n) {
  return tile_at_n<kQ>(tq, n, (uint32_t)kFixed);
}
// The producer's part at the start of its tile n: returns the tile.
template <int kQ>
__device__ __forceinline__ int64_t tile_claim_n(uint32_t* tq, uint32_t n, uint32_t fixed, uint32_t* ctr,
                                                uint32_t& claim, int64_t n_tiles) {
  if (n > 0) tq[(n - 1 + fixed) % kQ] = fixed * gridDim.x + claim;
  const int64_t tile = tile_at_n<kQ>(tq, n, fixed);
  if (tile < n_tiles) claim = atomicAdd(ctr, 1u);
  return tile;
}
template <int kFixed, int kQ>
__device__ __forceinline__ int64_t tile_claim(uint32_t* tq, uint32_t n, uint32_t* ctr, uint32_t& claim,
                                              int64_t n_tiles) {
  return tile_claim_n<kQ>(tq, n, (uint32_t)kFixed, ctr, claim, n_tiles);
}

// Order this thread's generic-proxy shared-memory accesses before later
// async-proxy (bulk copy) accesses to the same memory.
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Bulk copy global -> this CTA's shared memory, completing on `bar` (tx bytes).
// dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

}  // namespace gmc
