// RBGS path of one GMC / GMC+ step (Alg. 1 / Alg. 2 with the random-block
// compressor of Sec. 4 and Sec. 5.2), and the small kernels shared by both
// compressors (GMC+ detach, counters).
//
//   pick   per block-choice stream (one shared by all workers, or one per
//          worker): m distinct blocks out of nb by Floyd's sampling driven by a
//          SplitMix64 counter stream keyed by (seed, t[, k]); writes the sorted
//          block list, a block -> slot map and the union flags, and clears the
//          step's counters
//   step   ONE dense pass per tile for all K workers in ascending order:
//          v = (e + g) - c*(w_t - w_{t-1}); inside chosen blocks v is sent
//          (copied to the worker's slab), summed into the aggregate and its
//          residual set to +0, elsewhere v is the residual; then, on the union,
//          w -= (eta/K) * sum and w_{t+1} - w_t is stored for the next step.
//          With a detach output (Alg. 2) the same pass writes the rows
//          w_{t+1} - b*e_{t+1,k}: 4 bytes a value on top of the step's 12,
//          where a pass of its own read e back as well (d = 25.6 M, K = 32:
//          step and rows 3,249 -> 2,040 us). The last block ends the step
//          (end_step): two launches a step in all, where there were five; one
//          where a small step's blocks each make the choice (pick_here).
#include "gmc_internal.h"

namespace gmc {
namespace {

constexpr int kPickSmemWords = 12288;  // bitmap words kept in shared memory

__device__ __forceinline__ uint32_t block_of(int64_t j, const RbgsArgs& A) {
  return A.B_shift != 0xffffffffu ? (uint32_t)(j >> A.B_shift) : (uint32_t)(j / A.B);
}

// ---------------------------------------------------------------------------
// pick: one block per stream.
//
// Floyd's sampling takes, for i = 0 .. m-1 with top_i = nb-m+i, the draw r_i
// uniform on [0, top_i], or top_i when r_i was taken before. It need not run
// one draw after another: r_i was taken iff an earlier draw was the same block,
// or r_i is an earlier step's top (r_i = top_i', i' < i) and that step took its
// top, i.e. collided itself. The first is a table of each block's first draw
// (atomicMin), the second a walk to smaller i. So every draw is decided by a
// thread of its own: a chain of a few shared-memory reads, where the serial
// form cost about 50 ns a draw (m = 62: 9.9 us, m = 3,906: 200 us).
// ---------------------------------------------------------------------------
// Draw i's block: `first(b)` the first draw that gave block b, `drawn(i)` draw i. I: an index type.
template <typename I, typename First, typename Drawn>
__device__ __forceinline__ uint32_t floyd_pick(I i, I top0, First&& first, Drawn&& drawn) {
  const uint32_t r0 = drawn(i);
  I at = i, b = (I)r0;
  while (first(b) >= (int32_t)at) {      // no draw before `at` gave block b
    if (b < top0 || b - top0 >= at) return r0;  // nor is it an earlier step's top
    at = b - top0;                       // taken iff that step took its top (`at` decreases at every turn)
    b = (I)drawn(at);
  }
  return (uint32_t)(top0 + i);
}

constexpr int kPickThreads = 1024;
constexpr int kFirstWords = 16384;  // first-draw table kept in shared memory up to this many blocks

__global__ void __launch_bounds__(kPickThreads) k_rbgs_pick(RbgsArgs A) {
  griddep_wait();
  if (blockIdx.x == 0) {
    if (threadIdx.x < 8) A.acc_ctr->v[threadIdx.x] = 0ull;
    if (threadIdx.x < 2) A.tile_ctr[threadIdx.x] = 0u;  // tiles claimed by the fused pass, its warps done
  }
  extern __shared__ uint32_t pick_s[];
  __shared__ uint32_t ws[32];
  const int s = blockIdx.x;
  const int64_t nbw = (A.nb + 31) / 32;
  const bool in_smem = nbw <= kPickSmemWords;
  const bool first_smem = A.nb <= kFirstWords;
  int32_t* rank = A.rank + (int64_t)s * A.nb;
  int32_t* blk = A.blocks + (int64_t)s * A.m;
  uint32_t* bm = in_smem ? pick_s : A.bitmap + (int64_t)s * nbw;
  // a block's first draw (the slot map's memory holds it until the map is written)
  int32_t* first = first_smem ? reinterpret_cast<int32_t*>(pick_s + nbw) : rank;
  if (in_smem)
    for (int64_t i = threadIdx.x; i < nbw; i += blockDim.x) bm[i] = 0u;
  for (int64_t b = threadIdx.x; b < A.nb; b += blockDim.x) first[b] = 0x7fffffff;
  __syncthreads();
  const uint64_t key = stream_key(A.seed, A.t, A.per_worker ? (uint64_t)s + 1 : 0ull);
  const int64_t top0 = A.nb - A.m;
  auto drawn = [&](int64_t i) { return below(draw(key, (uint64_t)i), (uint64_t)(top0 + i) + 1); };
  for (int64_t i = threadIdx.x; i < A.m; i += blockDim.x) atomicMin(&first[drawn(i)], (int32_t)i);
  __syncthreads();
  for (int64_t i = threadIdx.x; i < A.m; i += blockDim.x) {
    const uint32_t pick =
        floyd_pick<int64_t>(i, top0, [&](int64_t b) { return first_smem ? first[b] : __ldcg(first + b); }, drawn);
    atomicOr(&bm[pick >> 5], 1u << (pick & 31));
  }
  __syncthreads();
  uint32_t carry = 0;
  for (int64_t w0 = 0; w0 < nbw; w0 += blockDim.x) {
    const int64_t wi = w0 + threadIdx.x;
    const uint32_t word = wi < nbw ? (in_smem ? bm[wi] : __ldcg(bm + wi)) : 0u;
    uint32_t tot;
    const uint32_t inc = block_inclusive_scan<uint32_t>((uint32_t)__popc(word), ws, &tot);
    const uint32_t q0 = carry + inc - (uint32_t)__popc(word);
    if (!in_smem && wi < nbw) bm[wi] = 0u;  // the global bitmap stays zero between steps
    // a warp's 32 words, one after another: lane l takes block 32 * word + l
    const int lane = threadIdx.x & 31;
#pragma unroll 4
    for (int i = 0; i < 32; ++i) {
      const uint32_t wd = __shfl_sync(0xffffffffu, word, i);
      const uint32_t qd = __shfl_sync(0xffffffffu, q0, i);
      const int64_t b = (wi - lane + i) * 32 + lane;
      if (b < A.nb) {
        const bool on = (wd >> lane) & 1u;
        const uint32_t q = qd + __popc(wd & lanemask_lt());
        rank[b] = on ? (int32_t)q : -1;
        if (on) {
          blk[q] = (int32_t)b;
          if (A.bulk) A.uflag_cur[b] = 1;
        }
      }
    }
    carry += tot;
  }
}

// ---------------------------------------------------------------------------
// The end of the fused step, by the `warps` consumer warps of every block (red:
// shared memory, 5 words a warp; they meet at named barrier 1): the block's
// counts into acc_ctr with one atomic each, and the last block out moves them to
// step_ctr, adds them to the totals, leaves acc_ctr zero for the next step, and
// clears the flags of the step before, which the next step's pick sets again.
// (With a set of atomics per warp the d = 272 k step's 2,129 warps queued at one
// line.)
// ---------------------------------------------------------------------------
constexpr int kEndWords = 5;
__device__ __forceinline__ void end_step(const RbgsArgs& A, unsigned long long* red, int warp, int warps, int lane,
                                         unsigned long long nonfinite, unsigned long long pairs,
                                         unsigned long long nnz, unsigned long long uni,
                                         unsigned long long changed) {
  const unsigned long long c[kEndWords] = {warp_sum(pairs), warp_sum(nnz), warp_sum(uni), warp_sum(changed),
                                           warp_sum(nonfinite)};
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < kEndWords; ++i) red[warp * kEndWords + i] = c[i];
  asm volatile("bar.sync 1, %0;" ::"r"(warps * 32) : "memory");
  if (warp != 0) return;
  if (lane < kEndWords) {
    constexpr int slot[kEndWords] = {kPairs, kNnz, kUnion, kChanged, kNonfinite};
    unsigned long long x = 0;
    for (int w = 0; w < warps; ++w) x += red[w * kEndWords + lane];
    int at = slot[0];
#pragma unroll
    for (int i = 1; i < kEndWords; ++i) at = lane == i ? slot[i] : at;
    if (x) {
      atomicAdd(&A.acc_ctr->v[at], x);
      if (lane == kEndWords - 1) atomicOr(A.status, kStatusNonfinite);
    }
    __threadfence();
  }
  __syncwarp();
  uint32_t last = 0;
  if (lane == 0) {
    __threadfence();
    last = atomicAdd(A.tile_ctr + 1, 1u) == gridDim.x - 1 ? 1u : 0u;
  }
  last = __shfl_sync(0xffffffffu, last, 0);
  if (last) {
    __threadfence();
    if (lane < 8) {
      A.step_ctr->v[lane] = __ldcg(&A.acc_ctr->v[lane]);
      A.acc_ctr->v[lane] = 0ull;
    }
    if (lane == 0) A.tile_ctr[1] = 0u;
    finalize_counters(A.step_ctr, A.total_ctr, 0ull);
  }
  if (last && A.bulk && A.clear_flags)
    for (int64_t b = lane * 4; b < A.nb; b += 128)  // allocated in whole words
      *reinterpret_cast<uint32_t*>(A.uflag_prev + b) = 0u;
}

// GMC+ detach (Alg. 2): w_{t+1} - b*e_{t+1,k} of 4 elements.
__device__ __forceinline__ float4 detached4(float4 w, float b, float4 e) {
  return make_float4(__fsub_rn(w.x, __fmul_rn(b, e.x)), __fsub_rn(w.y, __fmul_rn(b, e.y)),
                     __fsub_rn(w.z, __fmul_rn(b, e.z)), __fsub_rn(w.w, __fmul_rn(b, e.w)));
}
// ---------------------------------------------------------------------------
// fused step with plain loads and stores, for few tiles: a warp owns 128
// elements (a lane 4) and runs through the workers in ascending order, kWk of
// them loaded at a time. Bound by the latency of a few dependent loads, so it
// has none it can do without: the slots of a lane's blocks are looked up for
// every worker along with e and g (no union flags first), and w_t - w_{t-1} is
// read as it lies, zero outside the last union.
// ---------------------------------------------------------------------------
constexpr int kLsSub = 128;  // elements per warp
constexpr int kWk = 4;       // workers loaded together

// With kPick the step is one launch: every block makes the step's whole choice
// for itself in shared memory (pick_here), before it waits for the kernel ahead
// of it, and looks the slots up there. The choice costs each block what the
// launch of k_rbgs_pick and the wait for it cost the step, or less, while there
// are few streams and the block has little else to do (us a step, shared unless
// noted, k_rbgs_pick and step against one launch):
//   d = 65,536, K = 4             10.4 -> 7.0     d = 272,474, K = 8, per worker  14.9 -> 12.1
//   d = 600,000, K = 12, per w.   23.1 -> 22.6    d = 600,000, K = 16             27.5 -> 27.3
// and past the lines below:
//   d = 1,700, K = 16, per worker 17.7 -> 19.0    d = 600,000, K = 16, per worker 27.5 -> 28.2
//   d = 600,000, K = 32           52.4 -> 53.0    d = 2,310, K = 32, per worker   25.5 -> 29.0
constexpr int kPickHereStreams = 12;
constexpr int64_t kPickHereValues = 10 << 20;  // K * d
constexpr int kPickHereWords = 11264;  // shared words: a first-draw table, bitmap and its prefix per stream (44 KB)
constexpr int kPickHereDraws = 1024;   // draws of all streams: four a thread (K = 4, m = nb = 1,024: 14.4 -> 11.7)

// Words of shared memory that pick_here needs.
__host__ __device__ __forceinline__ int64_t pick_here_words(const RbgsArgs& A) {
  return (A.per_worker ? A.K : 1) * (A.nb + 2 * ((A.nb + 31) / 32));
}

struct Choice {
  const uint32_t* bm;   // streams x nbw: the chosen blocks
  const uint32_t* pre;  // streams x nbw: chosen blocks before the word's first
  int nbw;
  __device__ __forceinline__ int32_t slot(int s, uint32_t b) const {
    const int at = s * nbw + (int)(b >> 5);
    const uint32_t word = bm[at];
    return (word >> (b & 31)) & 1u ? (int32_t)(pre[at] + __popc(word & ((1u << (b & 31)) - 1u))) : -1;
  }
};

// The choice of k_rbgs_pick, of every stream, by one block of kThreads.
__device__ __forceinline__ Choice pick_here(const RbgsArgs& A, uint32_t* sm) {
  const int streams = A.per_worker ? A.K : 1;
  const int nb = (int)A.nb, m = (int)A.m, nbw = (nb + 31) / 32;
  int32_t* first = reinterpret_cast<int32_t*>(sm);
  uint32_t* bm = sm + streams * nb;
  uint32_t* pre = bm + streams * nbw;
  for (int i = threadIdx.x; i < streams * nb; i += kThreads) first[i] = 0x7fffffff;
  for (int i = threadIdx.x; i < streams * nbw; i += kThreads) bm[i] = 0u;
  __syncthreads();
  const int top0 = nb - m;
  auto drawn = [&](uint64_t key, int i) { return below(draw(key, (uint64_t)i), (uint64_t)(top0 + i) + 1); };
  auto key_of = [&](int s) { return stream_key(A.seed, A.t, A.per_worker ? (uint64_t)s + 1 : 0ull); };
  for (int x = threadIdx.x; x < streams * m; x += kThreads) {
    const int s = x / m, i = x - s * m;
    atomicMin(&first[s * nb + (int)drawn(key_of(s), i)], i);
  }
  __syncthreads();
  for (int x = threadIdx.x; x < streams * m; x += kThreads) {
    const int s = x / m, i = x - s * m;
    const uint64_t key = key_of(s);
    const uint32_t pick = floyd_pick<int>(i, top0, [&](int b) { return first[s * nb + b]; },
                                          [&](int q) { return drawn(key, q); });
    atomicOr(&bm[s * nbw + (int)(pick >> 5)], 1u << (pick & 31));
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int s = threadIdx.x >> 5; s < streams; s += kWarps) {
    uint32_t carry = 0;
    for (int w0 = 0; w0 < nbw; w0 += 32) {
      const uint32_t n = w0 + lane < nbw ? (uint32_t)__popc(bm[s * nbw + w0 + lane]) : 0u;
      uint32_t tot;
      const uint32_t exc = warp_excl_scan(n, &tot);
      if (w0 + lane < nbw) pre[s * nbw + w0 + lane] = carry + exc;
      carry += tot;
    }
  }
  __syncthreads();
  return Choice{bm, pre, nbw};
}

template <bool kBf16, bool kDetach, bool kPick>
__global__ void __launch_bounds__(kThreads) k_rbgs_step(RbgsArgs A) {
  extern __shared__ uint32_t pick_sm[];
  Choice choice = {};
  if (kPick) choice = pick_here(A, pick_sm);
  griddep_wait();
  if (kPick) {  // the lists of chosen blocks, a stream a block (gmc_selected reads them)
    for (int s = blockIdx.x; s < (A.per_worker ? A.K : 1); s += gridDim.x)
      for (int b = threadIdx.x; b < (int)A.nb; b += kThreads) {
        const int32_t q = choice.slot(s, (uint32_t)b);
        if (q >= 0) A.blocks[(int64_t)s * A.m + q] = b;
      }
  }
  __shared__ unsigned long long red[kWarps * kEndWords];
  const int lane = threadIdx.x & 31;
  uint32_t nonfinite = 0, pairs = 0, nnz = 0, uni = 0, changed = 0;
  const int64_t slab_ld = A.m * A.B;
  const int64_t nw = (int64_t)gridDim.x * kWarps;

  for (int64_t g0 = ((int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5)) * kLsSub; g0 < A.d; g0 += nw * kLsSub) {
    const int64_t j = g0 + lane * 4;
    const int lim = A.d - g0 < kLsSub ? (int)(A.d - g0) : kLsSub;
    const float4 d4 = *reinterpret_cast<const float4*>(A.dlt + j);
    const float4 w4 = *reinterpret_cast<const float4*>(A.w + j);
    uint32_t bid[4];
    float acc[4];
    uint32_t inU = 0;  // bit i: coordinate in this step's union
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc[i] = 0.f;
      bid[i] = lane * 4 + i < lim ? block_of(j + i, A) : 0u;
    }
    for (int k0 = 0; k0 < A.K; k0 += kWk) {
      float4 ev[kWk], gv[kWk];
      int32_t at[kWk][4];  // slot of the element's block among worker k's chosen ones, or -1
#pragma unroll
      for (int q = 0; q < kWk; ++q) {
        const int k = k0 + q;
        if (k < A.K) {
          ev[q] = __ldcs(reinterpret_cast<const float4*>(A.e + (int64_t)k * A.ld + j));
          const float* gk = A.grads + (int64_t)k * A.d;
          gv[q] = kBf16 ? load_g4_bf16(A.grads16 + (int64_t)k * A.d, j, A.d) : load_g4(gk, j, A.d, g_mode(gk));
          const int32_t* rk = A.rank + (A.per_worker ? (int64_t)k * A.nb : 0);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            at[q][i] = lane * 4 + i < lim ? (kPick ? choice.slot(A.per_worker ? k : 0, bid[i]) : rk[bid[i]]) : -1;
        }
      }
#pragma unroll
      for (int q = 0; q < kWk; ++q) {
        const int k = k0 + q;
        if (k < A.K) {
          float* sk = A.slab + (int64_t)k * slab_ld;
          const float v[4] = {accumulate(ev[q].x, gv[q].x, A.c, d4.x), accumulate(ev[q].y, gv[q].y, A.c, d4.y),
                              accumulate(ev[q].z, gv[q].z, A.c, d4.z), accumulate(ev[q].w, gv[q].w, A.c, d4.w)};
          float en[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            en[i] = v[i];
            if (lane * 4 + i < lim) nonfinite += is_nonfinite(v[i]) ? 1u : 0u;
            if (at[q][i] >= 0) {
              inU |= 1u << i;
              acc[i] = __fadd_rn(acc[i], v[i]);
              sk[(int64_t)at[q][i] * A.B + (j + i - (int64_t)bid[i] * A.B)] = v[i];
              en[i] = 0.f;  // e_{t+1,k} = +0 where sent
              ++pairs;
              nnz += (v[i] != 0.f);
            }
          }
          __stcs(reinterpret_cast<float4*>(A.e + (int64_t)k * A.ld + j), make_float4(en[0], en[1], en[2], en[3]));
        }
      }
    }
    float wo[4] = {w4.x, w4.y, w4.z, w4.w};
    float dd[4] = {0.f, 0.f, 0.f, 0.f};
    bool touch = (__float_as_uint(d4.x) | __float_as_uint(d4.y) | __float_as_uint(d4.z) | __float_as_uint(d4.w)) != 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (inU & (1u << i)) {
        const float wn = __fsub_rn(wo[i], __fmul_rn(A.a, acc[i]));
        A.w[j + i] = wn;
        dd[i] = __fsub_rn(wn, wo[i]);
        wo[i] = wn;
        changed += (dd[i] != 0.f);
        ++uni;
        touch = true;
      }
    }
    if (touch) *reinterpret_cast<float4*>(A.dlt + j) = make_float4(dd[0], dd[1], dd[2], dd[3]);
    if (kDetach) {  // the residuals as this lane stored them
      const float4 wn4 = make_float4(wo[0], wo[1], wo[2], wo[3]);
#pragma unroll 8
      for (int k = 0; k < A.K; ++k) {
        const float4 e4 = *reinterpret_cast<const float4*>(A.e + (int64_t)k * A.ld + j);
        store_row(A.det + (int64_t)k * A.det_ld + g0, lane * 4, lim, detached4(wn4, A.det_b, e4), lane);
      }
    }
  }
  end_step(A, red, threadIdx.x >> 5, kWarps, lane, nonfinite, pairs, nnz, uni, changed);
}

// (index, value) pairs of worker k's last C(.), in ascending index order.
__global__ void k_rbgs_expand(RbgsArgs A, int k, uint32_t* idx_out, float* val_out) {
  griddep_wait();
  const int64_t n = A.m * A.B;
  const int32_t* blk = A.blocks + (A.per_worker ? (int64_t)k * A.m : 0);
  const float* sk = A.slab + (int64_t)k * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q = i / A.B, off = i - q * A.B;
    const int64_t j = (int64_t)blk[q] * A.B + off;
    if (j < A.d) {
      idx_out[i] = (uint32_t)j;
      val_out[i] = sk[i];
    }
  }
}

// GMC+ detach: out[k][j] = w[j] - b * e[k][j] (Alg. 2), where the step's own
// pass does not write it (top-k steps, gmc_get_worker_params). Streaming, bound
// by memory: a warp loads its 128 floats of w once and runs through the
// workers of its slice (blockIdx.y).
__global__ void __launch_bounds__(kThreads) k_detach(DetachArgs A, int per) {
  griddep_wait();
  const int lane = threadIdx.x & 31;
  const int k_lo = A.k0 + blockIdx.y * per, k_hi = min(A.k1, k_lo + per);
  const int64_t nw = (int64_t)gridDim.x * kWarps;
  for (int64_t g0 = ((int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5)) * 128; g0 < A.d; g0 += nw * 128) {
    const int lim = A.d - g0 < 128 ? (int)(A.d - g0) : 128;
    // w and the rows of e are allocated in whole tiles: reads past d stay inside
    const float4 w4 = *reinterpret_cast<const float4*>(A.w + g0 + lane * 4);
#pragma unroll 4
    for (int k = k_lo; k < k_hi; ++k) {
      const float4 e4 = __ldcs(reinterpret_cast<const float4*>(A.e + (int64_t)k * A.ld + g0 + lane * 4));
      store_row(A.out + (int64_t)(k - A.k0) * A.out_ld + g0, lane * 4, lim, detached4(w4, A.b, e4), lane);
    }
  }
}

// dst[0..n) = src[0..n), src 16-byte aligned and readable to the next 128
// floats. As fast as cudaMemcpyAsync at every size (138.4 M floats: 169 against
// 170 us) and begins while the kernel before it ends (d = 272 k: 1.8 against
// 5.4 us on the device, 11.4 against 17 us a call on the host). src is not
// __restrict__: the kernel before, which writes it, may still run when this one
// begins, so its loads must not be taken for loads of constant memory.
__global__ void __launch_bounds__(kThreads) k_copy_row(const float* src, float* dst, int64_t n) {
  griddep_wait();
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * kWarps;
  for (int64_t g0 = ((int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5)) * 128; g0 < n; g0 += nw * 128) {
    const float4 x = *reinterpret_cast<const float4*>(src + g0 + lane * 4);
    store_row(dst + g0, lane * 4, n - g0 < 128 ? (int)(n - g0) : 128, x, lane);
  }
}

__global__ void k_finalize(Counters* step, Counters* total, unsigned long long pairs_add) {
  griddep_wait();
  finalize_counters(step, total, pairs_add);  // one warp
}


// ---------------------------------------------------------------------------
// The same step as k_rbgs_step, with e and g streamed through a shared-memory
// ring by bulk copies. One persistent CTA per SM: a producer thread issues
// each (tile, worker) item's cp.async.bulk copies of e and g into the ring;
// sixteen consumer warps each own 256 elements of every tile and run through
// the K workers in ascending order (the aggregate adds in that order).
// Producer and consumers meet only at mbarriers; every wait is bounded. A
// CTA's first two tiles are fixed and every later one is claimed from a
// counter (tile_at, tile_claim), so that CTAs whose streams run faster take
// more tiles and all of them finish together.
// ---------------------------------------------------------------------------
namespace rbulk {
constexpr int kT = kRbgsTile;
constexpr int kStages = 4;
constexpr int kConsumers = 16;
constexpr int kSub = kT / kConsumers;      // 256 elements per consumer warp
constexpr int kGLen = kT + 8;              // g stage: up to 3 leading floats of misalignment
constexpr int kThreadsAll = (kConsumers + 1) * 32;
constexpr int kG = kSub / 128;             // float4 groups per lane
struct Smem {
  float e[kStages][kT];
  float g[kStages][kGLen];
  uint64_t full[kStages];                  // e, g landed (1 arrival + tx bytes)
  uint64_t empty[kStages];                 // all consumer warps read the stage
  int32_t gmeta[kStages];                  // leading floats in the g stage, -1 = not copied
  uint32_t tq[8];                          // claimed tiles (tile_at)
  unsigned long long red[kConsumers * kEndWords];  // the warps' counts (end_step)
};
// Tiles: the first two of a CTA fixed, the rest claimed one tile ahead of the
// producer's start of the tile before it. A consumer reads a tile's slot at
// its start, after waiting on the previous tile's items (the producer's start
// of that tile is two tiles on from the claim's); the producer runs at most
// kStages items (tiles, for K = 1) ahead of the slowest consumer.
constexpr int kFixed = 2;
constexpr int kQ = 8;
static_assert(kQ > kStages + kFixed, "the producer may overwrite a claimed tile not yet read");
}  // namespace rbulk

template <bool kBf16, bool kDetach>
__global__ void __launch_bounds__(rbulk::kThreadsAll, 1) k_rbgs_bulk(RbgsArgs A) {
  griddep_wait();
  using namespace rbulk;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], kConsumers);
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp == kConsumers) {
    // ---- producer ----
    if (lane != 0) return;
    // gradient rows of es-byte elements (fp32, or bf16 from gmc_step_bf16)
    constexpr int es = kBf16 ? 2 : 4;
    const char* g_lo = kBf16 ? reinterpret_cast<const char*>(A.grads16) : reinterpret_cast<const char*>(A.grads);
    const char* g_hi = g_lo + (int64_t)A.K * A.d * es;
    uint32_t item = 0, claim = 0;
    uint32_t held = ~0u;  // test hook: the item not copied
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      const int64_t tile = tile_claim<kFixed, kQ>(sm.tq, n, A.tile_ctr, claim, A.n_tiles);
      if (tile >= A.n_tiles) break;
      const int64_t j0 = tile * kT;
      const int64_t nvalid = A.d - j0 < kT ? A.d - j0 : kT;
      for (int k = 0; k < A.K; ++k, ++item) {
        const uint32_t s = item % kStages, r = item / kStages;
        if (r > 0 && !wait_bounded(&sm.empty[s], (r - 1) & 1, A.wait_ns)) {
          ok = false;
          break;
        }
        if (tile == A.hold_tile && k == A.hold_k) {  // the stage's phase never completes
          held = item;
          continue;
        }
        const float* esrc = A.e + (int64_t)k * A.ld + j0;
        const uintptr_t ga = reinterpret_cast<uintptr_t>(g_lo + ((int64_t)k * A.d + j0) * es);
        const uint32_t off = (uint32_t)(ga & 15) / es;  // leading elements before the row's tile
        const char* gsrc = reinterpret_cast<const char*>(ga - off * es);
        const uint32_t gbytes = (uint32_t)(((nvalid + off) * es + 15) & ~int64_t(15));
        const bool gbulk = !A.g_direct && (ga % es) == 0 && gsrc >= g_lo && gsrc + gbytes <= g_hi;
        sm.gmeta[s] = gbulk ? (int32_t)off : -1;
        mbar_arrive_expect_tx(&sm.full[s], kT * 4 + (gbulk ? gbytes : 0));
        bulk_load(sm.e[s], esrc, kT * 4, &sm.full[s]);
        if (gbulk) bulk_load(sm.g[s], gsrc, gbytes, &sm.full[s]);
      }
    }
    if (!ok) atomicOr(A.status, kStatusTimeout);
    // Every copy issued lands before the CTA's shared memory goes away, even
    // when the consumers gave up on their waits: the last kStages items (the
    // earlier ones were read, as their stages' empty barriers showed) read
    // valid global memory and complete without any other warp's help; no
    // later phase is armed on their stages.
    const uint32_t first = item > (uint32_t)kStages ? item - kStages : 0u;
    for (uint32_t i = first; i < item; ++i)
      if (i != held && !wait_bounded(&sm.full[i % kStages], (i / kStages) & 1, kWaitLimitNs))
        atomicOr(A.status, kStatusTimeout | kStatusInternal);
    return;
  }

  // ---- consumers ----
  const int64_t slab_ld = A.m * A.B;
  uint32_t nonfinite = 0;
  unsigned long long pairs = 0, nnz = 0, uni = 0, changed = 0;
  uint32_t item = 0;
  bool ok = true;
  for (uint32_t n = 0; ok; ++n) {
    const int64_t tile = tile_at<kFixed, kQ>(sm.tq, n);
    if (tile >= A.n_tiles) break;
    const int64_t s0 = tile * kT + warp * kSub;
    const int64_t rem = A.d - s0;
    const int lim = rem < kSub ? (rem > 0 ? (int)rem : 0) : kSub;
    // does the sub-tile touch the last step's union (tp) or this step's (tc)?
    int tp = 0, tc = 0;
    if (lim > 0) {
      const int64_t b_lo = block_of(s0, A), b_hi = block_of(s0 + lim - 1, A);
      for (int64_t b = b_lo + lane; b <= b_hi; b += 32) {
        tp |= A.has_prev ? A.uflag_prev[b] : 0;
        tc |= A.uflag_cur[b];
      }
    }
    tp = __any_sync(0xffffffffu, tp);
    tc = __any_sync(0xffffffffu, tc);
    float dl[kG][4], acc[kG][4];
    float4 w4[kG];  // detach output: w_t, which is w_{t+1} outside the union
    uint32_t bid[kG][4];
    uint32_t inU = 0;  // bit (u*4+i): coordinate in this step's union
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      const int l = u * 128 + lane * 4;
      if (kDetach) w4[u] = *reinterpret_cast<const float4*>(A.w + s0 + l);
      float4 d4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (tp && l < lim) d4 = *reinterpret_cast<const float4*>(A.dlt + s0 + l);
      dl[u][0] = d4.x; dl[u][1] = d4.y; dl[u][2] = d4.z; dl[u][3] = d4.w;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[u][i] = 0.f;
        const bool in = l + i < lim;
        bid[u][i] = (in && tc) ? block_of(s0 + l + i, A) : 0u;
        if (in && tc && A.uflag_cur[bid[u][i]]) inU |= 1u << (u * 4 + i);
      }
    }
    for (int k = 0; k < A.K; ++k, ++item) {
      const uint32_t s = item % kStages, r = item / kStages;
      if (!__all_sync(0xffffffffu, wait_bounded(&sm.full[s], r & 1, A.wait_ns))) {  // warp-uniform
        ok = false;
        break;
      }
      const int32_t off = sm.gmeta[s];
      const float* se = sm.e[s] + warp * kSub;
      const float* sg = sm.g[s] + (off > 0 ? off : 0) + warp * kSub;
      float v[kG][4];
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        const int l = u * 128 + lane * 4;
        const float4 e4 = *reinterpret_cast<const float4*>(se + l);
        float4 g4;
        if constexpr (kBf16) {
          if (off >= 0)
            g4 = bf16x4(reinterpret_cast<const uint16_t*>(sm.g[s]) + off + warp * kSub + l);
          else
            g4 = load_g4_bf16(A.grads16 + (int64_t)k * A.d, s0 + l, A.d);
        } else if (off == 0) {
          g4 = *reinterpret_cast<const float4*>(sg + l);
        } else if (off == 2) {
          const float2 a = *reinterpret_cast<const float2*>(sg + l);
          const float2 b = *reinterpret_cast<const float2*>(sg + l + 2);
          g4 = make_float4(a.x, a.y, b.x, b.y);
        } else if (off > 0) {
          g4 = make_float4(sg[l], sg[l + 1], sg[l + 2], sg[l + 3]);
        } else {
          const float* gk = A.grads + (int64_t)k * A.d;
          g4 = load_g4(gk, s0 + l, A.d, g_mode(gk));
        }
        if (lim < kSub && off >= 0) {  // past d the stage holds bytes of no meaning
          if (l >= lim) g4.x = 0.f;
          if (l + 1 >= lim) g4.y = 0.f;
          if (l + 2 >= lim) g4.z = 0.f;
          if (l + 3 >= lim) g4.w = 0.f;
        }
        v[u][0] = accumulate(e4.x, g4.x, A.c, dl[u][0]);
        v[u][1] = accumulate(e4.y, g4.y, A.c, dl[u][1]);
        v[u][2] = accumulate(e4.z, g4.z, A.c, dl[u][2]);
        v[u][3] = accumulate(e4.w, g4.w, A.c, dl[u][3]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.empty[s]);  // this warp is done reading stage s
      float* ek = A.e + (int64_t)k * A.ld + s0;
      const int32_t* rk = A.rank + (A.per_worker ? (int64_t)k * A.nb : 0);
      float* sk = A.slab + (int64_t)k * slab_ld;
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        const int l = u * 128 + lane * 4;
        float en[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          en[i] = v[u][i];
          if (l + i < lim) {
            nonfinite += is_nonfinite(v[u][i]) ? 1u : 0u;
            if (tc) {
              const int32_t q = rk[bid[u][i]];
              if (q >= 0) {  // in one of worker k's chosen blocks: sent
                acc[u][i] = __fadd_rn(acc[u][i], v[u][i]);
                sk[(int64_t)q * A.B + (s0 + l + i - (int64_t)bid[u][i] * A.B)] = v[u][i];
                en[i] = 0.f;  // e_{t+1,k} = +0 where sent
                ++pairs;
                nnz += (v[u][i] != 0.f);
              }
            }
          }
        }
        const float4 e4 = make_float4(en[0], en[1], en[2], en[3]);
        __stcs(reinterpret_cast<float4*>(ek + l), e4);
        if (kDetach && !tc)
          store_row(A.det + (int64_t)k * A.det_ld + s0, l, lim, detached4(w4[u], A.det_b, e4), lane);
      }
    }
    if (ok && (tp || tc)) {  // the union: w_{t+1} = w_t - a * sum, and w_{t+1} - w_t for the next step
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        const int l = u * 128 + lane * 4;
        if (l >= lim) continue;
        float dd[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (inU & (1u << (u * 4 + i))) {
            const float wo = A.w[s0 + l + i];
            const float wn = __fsub_rn(wo, __fmul_rn(A.a, acc[u][i]));
            A.w[s0 + l + i] = wn;
            dd[i] = __fsub_rn(wn, wo);
            changed += (dd[i] != 0.f);
            ++uni;
          }
        }
        *reinterpret_cast<float4*>(A.dlt + s0 + l) = make_float4(dd[0], dd[1], dd[2], dd[3]);
      }
    }
    if (kDetach && ok && tc) {  // w_{t+1} is known now; w and the residuals as this lane stored them
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        const int l = u * 128 + lane * 4;
        const float4 wn4 = *reinterpret_cast<const float4*>(A.w + s0 + l);
        for (int k = 0; k < A.K; ++k) {
          const float4 e4 = *reinterpret_cast<const float4*>(A.e + (int64_t)k * A.ld + s0 + l);
          store_row(A.det + (int64_t)k * A.det_ld + s0, l, lim, detached4(wn4, A.det_b, e4), lane);
        }
      }
    }
  }
  if (!ok) atomicOr(A.status, kStatusTimeout);
  end_step(A, sm.red, warp, kConsumers, lane, nonfinite, pairs, nnz, uni, changed);
}

}  // namespace

cudaError_t configure_rbgs_kernels() {
  cudaError_t err = cudaFuncSetAttribute((const void*)k_rbgs_pick, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kPickSmemWords * 4 + kFirstWords * 4);
  for (const void* f : {(const void*)k_rbgs_bulk<false, false>, (const void*)k_rbgs_bulk<true, false>,
                        (const void*)k_rbgs_bulk<false, true>, (const void*)k_rbgs_bulk<true, true>}) {
    const cudaError_t e2 =
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(rbulk::Smem));
    if (err == cudaSuccess) err = e2;
  }
  return err;
}

int rbgs_blocks_per_sm() {
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_rbgs_step<false, true, false>, kThreads, 0);
  return n > 0 ? n : 1;
}

// Whether the load/store step makes its choice itself.
bool rbgs_picks_in_step(const RbgsArgs& A) {
  const int streams = A.per_worker ? A.K : 1;
  return !A.bulk && streams <= kPickHereStreams && A.K * A.d <= kPickHereValues &&
         pick_here_words(A) <= kPickHereWords && streams * A.m <= kPickHereDraws;
}

cudaError_t launch_rbgs_pick(const RbgsArgs& A, cudaStream_t s) {
  const int64_t nbw = (A.nb + 31) / 32;
  const int smem = (nbw <= kPickSmemWords ? (int)(nbw * 4) : 0) + (A.nb <= kFirstWords ? (int)(A.nb * 4) : 0);
  return launch_pdl(k_rbgs_pick, dim3(A.per_worker ? A.K : 1), dim3(kPickThreads), smem, s, A);
}

cudaError_t launch_rbgs_step(const RbgsArgs& A, int grid, cudaStream_t s) {
  if (A.bulk) {
    const dim3 g(grid), b(rbulk::kThreadsAll);
    const size_t sm = sizeof(rbulk::Smem);
    if (A.det) return launch_pdl(A.bf16 ? k_rbgs_bulk<true, true> : k_rbgs_bulk<false, true>, g, b, sm, s, A);
    return launch_pdl(A.bf16 ? k_rbgs_bulk<true, false> : k_rbgs_bulk<false, false>, g, b, sm, s, A);
  }
  const dim3 g(grid), b(kThreads);
  if (rbgs_picks_in_step(A)) {
    const size_t sm = (size_t)pick_here_words(A) * 4;
    if (A.det) return launch_pdl(A.bf16 ? k_rbgs_step<true, true, true> : k_rbgs_step<false, true, true>, g, b, sm, s, A);
    return launch_pdl(A.bf16 ? k_rbgs_step<true, false, true> : k_rbgs_step<false, false, true>, g, b, sm, s, A);
  }
  if (A.det) return launch_pdl(A.bf16 ? k_rbgs_step<true, true, false> : k_rbgs_step<false, true, false>, g, b, 0, s, A);
  return launch_pdl(A.bf16 ? k_rbgs_step<true, false, false> : k_rbgs_step<false, false, false>, g, b, 0, s, A);
}

cudaError_t launch_rbgs_expand(const RbgsArgs& A, int k, uint32_t* idx_out, float* val_out,
                               cudaStream_t s) {
  const int64_t n = A.m * A.B;
  const int grid = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  k_rbgs_expand<<<grid > 0 ? grid : 1, 256, 0, s>>>(A, k, idx_out, val_out);
  return cudaGetLastError();
}

cudaError_t launch_detach(const DetachArgs& A, cudaStream_t s) {
  // enough warps for small d: the workers are split over blockIdx.y until about 2,048 blocks run
  const int64_t blocks = (A.d + 128 * kWarps - 1) / (128 * kWarps);
  const int K = A.k1 - A.k0;
  const int split = (int)(blocks >= 2048 ? 1 : (2048 / blocks < K ? 2048 / blocks : K));
  const int per = (K + split - 1) / split;
  const dim3 grid((unsigned)(blocks < 65536 ? blocks : 65536), (unsigned)((K + per - 1) / per));
  return launch_pdl(k_detach, grid, dim3(kThreads), 0, s, A, per);
}

cudaError_t launch_copy_row(const float* src, float* dst, int64_t n, int device, cudaStream_t s) {
  // the kernel writes this device's memory; what else dst may be (host memory,
  // another device's, no memory at all) is cudaMemcpyAsync's to copy to or refuse
  cudaPointerAttributes at;
  const cudaError_t err = cudaPointerGetAttributes(&at, dst);
  if (err != cudaSuccess) cudaGetLastError();
  if (err != cudaSuccess || at.type != cudaMemoryTypeDevice || at.device != device ||
      (reinterpret_cast<uintptr_t>(dst) & 3u))
    return cudaMemcpyAsync(dst, src, (size_t)n * sizeof(float), cudaMemcpyDeviceToDevice, s);
  const int64_t blocks = (n + 128 * kWarps - 1) / (128 * kWarps);
  return launch_pdl(k_copy_row, dim3((unsigned)blocks), dim3(kThreads), 0, s, src, dst, n);
}

cudaError_t launch_finalize(Counters* step, Counters* total, unsigned long long pairs_add,
                            cudaStream_t s) {
  const cudaError_t err = launch_pdl(k_finalize, dim3(1), dim3(32), 0, s, step, total, pairs_add);
  if (err != cudaSuccess) return err;
  return cudaGetLastError();
}

}  // namespace gmc
