// Server-side kernels: reduce the gradient queue and apply it to the weights.
//
// All three server steps of the paper are elementwise over the parameter vector and stream the
// queue exactly once, so they are bound by HBM bandwidth: per queued gradient 4*P_PAD bytes are
// read, and per step the weights are read once and written once (plus once more for the
// chain-replication mirror).  Threads own float4 columns of the parameter vector, so every load
// and store is a coalesced 16-byte access; the K loop is unrolled to keep many independent loads
// in flight per thread.
#include <algorithm>

#include "kernels.h"
#include "tc5_common.cuh"
#include "device_common.cuh"

namespace psk {

namespace {

constexpr int TPB = 256;
constexpr int COL_BLOCKS = (P_VEC4 + TPB - 1) / TPB;   // 795

__device__ __forceinline__ float4 ld_stream(const float4* p) { return __ldcs(p); }

__device__ __forceinline__ void add4(float4& a, const float4& b) {
  a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
}

__device__ __forceinline__ void fma4(float c, const float4& v, float4& a) {
  a.x = fmaf(c, v.x, a.x); a.y = fmaf(c, v.y, a.y); a.z = fmaf(c, v.z, a.z); a.w = fmaf(c, v.w, a.w);
}

// Adds p to a running sum and what the addition rounds away to another, for two columns at once.  (Exact while |acc| >= |p|;
// otherwise off by a rounding of p, which is small then.)
__device__ __forceinline__ void add_compensated(u64 p, u64& acc, u64& err) {
  u64 t, d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(acc), "l"(p));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(t), "l"(acc));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(p), "l"(d));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(err) : "l"(err), "l"(d));
  acc = t;
}
// The two together; a sum that is not finite stays what it is (its second part is no number then).
__device__ __forceinline__ float2 compensated(u64 acc, u64 err) {
  float a0, a1, e0, e1;
  unpack2(acc, a0, a1);
  unpack2(err, e0, e1);
  return make_float2(isfinite(e0) ? a0 + e0 : a0, isfinite(e1) ? a1 + e1 : a1);
}

// Sum of slots [k0, k1) of one float4 column, in a fixed order: eight interleaved running sums
// (slot k goes to sum k mod 8 relative to k0), combined pairwise at the end.  With WEIGHTED every slot is
// multiplied by its own factor coef_k[k] (the stale-gradient treatments) as it is added.
template <bool WEIGHTED>
__device__ __forceinline__ float4 column_sum(const float4* __restrict__ q, int64_t k0, int64_t k1, const float* __restrict__ coef_k) {
  float4 acc[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
  int64_t k = k0;
  for (; k + 8 <= k1; k += 8) {
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = ld_stream(q + (k + u) * (int64_t)P_VEC4);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (WEIGHTED) fma4(coef_k[k + u], v[u], acc[u]);
      else add4(acc[u], v[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < 7; ++u)
    if (k + u < k1) {
      const float4 v = ld_stream(q + (k + u) * (int64_t)P_VEC4);
      if (WEIGHTED) fma4(coef_k[k + u], v, acc[u]);
      else add4(acc[u], v);
    }
  add4(acc[0], acc[1]); add4(acc[2], acc[3]); add4(acc[4], acc[5]); add4(acc[6], acc[7]);
  add4(acc[0], acc[2]); add4(acc[4], acc[6]);
  add4(acc[0], acc[4]);
  return acc[0];
}

// theta_out = theta_in - coef * sum_k g_k (or - sum_k coef_k[k] g_k), whole queue in one pass (small K).
template <bool WEIGHTED>
__global__ void __launch_bounds__(TPB) sum_apply_direct(const float4* __restrict__ queue, int64_t K,
                                                        const float4* theta_in, float4* theta_out,
                                                        float4* __restrict__ replica, float coef, const float* __restrict__ coef_k) {
  // theta_in and theta_out may be the same buffer (a ring of depth one): each thread reads its column before it
  // writes it, and the two pointers carry no no-alias promise
  int col = blockIdx.x * TPB + threadIdx.x;
  if (col >= P_VEC4) return;
  pdl_enter();
  float4 s = column_sum<WEIGHTED>(queue + col, 0, K, coef_k);
  float4 t = theta_in[col];
  t.x = fmaf(-coef, s.x, t.x); t.y = fmaf(-coef, s.y, t.y);
  t.z = fmaf(-coef, s.z, t.z); t.w = fmaf(-coef, s.w, t.w);
  theta_out[col] = t;
  if (replica) replica[col] = t;
}

// Stage 1 of the long-queue reduction: block (x, y) sums slot range y of column block x.
template <bool WEIGHTED>
__global__ void __launch_bounds__(TPB) sum_partial(const float4* __restrict__ queue, int64_t K,
                                                   int n_split, float4* __restrict__ partial, const float* __restrict__ coef_k) {
  int col = blockIdx.x * TPB + threadIdx.x;
  if (col >= P_VEC4) return;
  pdl_enter();
  int s = blockIdx.y;
  int64_t per = (K + n_split - 1) / n_split;
  int64_t k0 = s * per, k1 = k0 + per < K ? k0 + per : K;
  float4 acc = k0 < k1 ? column_sum<WEIGHTED>(queue + col, k0, k1, coef_k) : make_float4(0.f, 0.f, 0.f, 0.f);
  partial[(int64_t)s * P_VEC4 + col] = acc;
}

// Stage 2: sums the partials in slot order and applies the update.
__global__ void __launch_bounds__(TPB) sum_finish(const float4* __restrict__ partial, int n_split,
                                                  const float4* theta_in, float4* theta_out,   // may alias (see above)
                                                  float4* __restrict__ replica, float coef) {
  int col = blockIdx.x * TPB + threadIdx.x;
  if (col >= P_VEC4) return;
  pdl_enter();
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = 0; i < n_split; ++i) add4(s, partial[(int64_t)i * P_VEC4 + col]);
  float4 t = theta_in[col];
  t.x = fmaf(-coef, s.x, t.x); t.y = fmaf(-coef, s.y, t.y);
  t.z = fmaf(-coef, s.z, t.z); t.w = fmaf(-coef, s.w, t.w);
  theta_out[col] = t;
  if (replica) replica[col] = t;
}

// Ordered one-by-one application: each thread keeps its float4 of the weights in registers,
// subtracts the gradients in arrival order (the same sequence of roundings as K separate
// updates), and stores only the versions that stay readable: the last ring_depth ones.
__global__ void __launch_bounds__(TPB) async_apply(AsyncApplyArgs a, AsyncOrder ord) {
  int col = blockIdx.x * TPB + threadIdx.x;
  if (col >= P_VEC4) return;
  pdl_enter();
  const float4* q = reinterpret_cast<const float4*>(a.queue) + col;
  float4 t = reinterpret_cast<const float4*>(a.theta_in)[col];
  constexpr int U = 8;
  for (int k0 = 0; k0 < a.K; k0 += U) {
    float4 g[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u < a.K) g[u] = ld_stream(q + (int64_t)ord.slot[k0 + u] * P_VEC4);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      int k = k0 + u;
      if (k < a.K) {
        const float c = a.coef_k ? a.coef_k[ord.slot[k]] : a.coef;
        t.x = fmaf(-c, g[u].x, t.x); t.y = fmaf(-c, g[u].y, t.y);
        t.z = fmaf(-c, g[u].z, t.z); t.w = fmaf(-c, g[u].w, t.w);
        if (k >= a.first_stored) {
          int slot = (int)((a.v0 + (uint64_t)k + 1) % (uint64_t)a.ring_depth);
          reinterpret_cast<float4*>(a.ring[slot])[col] = t;
        }
        for (int m = 0; m < a.n_mirror; ++m)
          if (k == a.mirror_k[m]) reinterpret_cast<float4*>(a.replica[m])[col] = t;
      }
    }
  }
}

// Copies rows of P_PAD floats; used for the copying form of enqueue.
__global__ void __launch_bounds__(TPB) copy_rows(float4* __restrict__ dst, const float4* __restrict__ src,
                                                 int64_t n_vec) {
  int64_t i = (int64_t)blockIdx.x * TPB + threadIdx.x;
  int64_t stride = (int64_t)gridDim.x * TPB;
  for (; i < n_vec; i += stride) dst[i] = src[i];
}

// ---- clipping by global norm ------------------------------------------------------------------------------------
// Block (c, k) sums the squares of chunk c of gradient k: every thread over its float4 columns in four interleaved
// sums, then lanes and warps in a fixed order.
constexpr int NORM_VEC = P_VEC4 / NORM_CHUNKS;      // 25,416 float4 columns per chunk
static_assert(NORM_VEC * NORM_CHUNKS == P_VEC4, "chunks tile the vector");
__global__ void __launch_bounds__(TPB) sq_norm_partial(const float4* __restrict__ queue, float* __restrict__ norm_part) {
  __shared__ float warp_sum[TPB / 32];
  const int64_t k = blockIdx.y;
  const float4* g = queue + k * (int64_t)P_VEC4 + (int64_t)blockIdx.x * NORM_VEC;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  int i = threadIdx.x;
  for (; i + 3 * TPB < NORM_VEC; i += 4 * TPB) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = g[i + u * TPB];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = fmaf(v[u].x, v[u].x, fmaf(v[u].y, v[u].y, fmaf(v[u].z, v[u].z, fmaf(v[u].w, v[u].w, acc[u]))));
  }
  for (; i < NORM_VEC; i += TPB) {
    const float4 v = g[i];
    acc[0] = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, acc[0]))));
  }
  float t = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < TPB / 32; ++w) s += warp_sum[w];
    norm_part[k * NORM_CHUNKS + blockIdx.x] = s;
  }
}

__global__ void __launch_bounds__(TPB) clip_coef_finish(const float* __restrict__ norm_part, int64_t K, float clip, float* __restrict__ coef_k) {
  const int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (k >= K) return;
  float n2 = 0.f;
#pragma unroll
  for (int c = 0; c < NORM_CHUNKS; ++c) n2 += norm_part[k * NORM_CHUNKS + c];
  coef_k[k] *= fminf(1.0f, clip / sqrtf(n2));      // a zero gradient keeps its factor (clip / 0 = inf)
}

// ---- clipping by global norm, summed and applied in one pass over a long queue ------------------------------------
// A gradient's factor needs its whole norm, so summing clipped gradients takes two reads of the queue, unless a gradient
// stays on the chip in between.  It does here: one CTA per SM owns a fixed range of float4 columns, every gradient's share
// of it (22 KB) arrives by a bulk copy in a ring of ten shared-memory slots, is squared, and stays in its slot until the
// CTAs have exchanged their partial sums of squares through global memory; then it is added with its factor.  HBM sees
// every gradient once: the kernel's bound is one read of the queue.
// Warps: one group squares, one adds (each thread keeps the sums of its four columns in registers): a warp's step per
// gradient is a chain of latencies, which two groups halve.  One warp issues the copies, one publishes the CTA's partial
// sums, CS_GATHER gather the other CTAs' in turn.  A word of the exchange carries its gradient's number beside the sum, so
// it needs no flag, and the words of CS_RING gradients are used in turn; every CTA writes its word CS_COPIES times and a
// CTA polls one of the copies only: the polls of all CTAs on one copy slow the stores down.
// Precision: a thread adds `fold` gradients in single precision, and that to a sum kept in two parts, whose error does not
// grow with its terms.  Relative error (2-norm) of the sum of gradients N(0.02, 0.01^2) with one running sum / so / in two
// passes (eight running sums, from 160 gradients on in up to sixteen ranges): K = 16: 6.6e-8 / 3.1e-8 / 4.1e-8, 300: 2.6e-7 /
// 2.8e-8 / 5.5e-8, 12,800: 1.5e-6 / 1.9e-8 / 5.6e-8.  It costs 1 % at K = 1600 (872 -> 880 us for the whole call); a sum in
// two parts at every gradient, every second and every fourth cost 4.2, 4.1 and 2.3 %.
// Measured (B200), us for clipping by norm, summing and applying K gradients, two passes over the queue (norms, factors,
// weighted sum) -> this kernel: K = 1: 27 -> 12, 16: 39 -> 19, 128: 159 -> 86, 1600: 1466 -> 793 (6.6 TB/s), 6400: 5700 -> 3131.
// At 1600 also: three gathering warps 902, four 1028 (more polls); 16 copies 812; squaring and adding by the same warps,
// four gradients held in registers behind the ring, 887; a copy polled word by word by everybody 1124.
// The CTAs wait for one another, so the launch is cooperative; every wait is bounded, and a warp gives up as a whole.
constexpr int CS_ADD = 11, CS_ADD_PER = 4, CS_SQ = 8, CS_SQ_PER = 6, CS_GATHER = 2;      // warps, columns per thread
constexpr int CS_THREADS = 32 * (CS_ADD + CS_SQ + 2 + CS_GATHER);
constexpr int CS_MAX_COLS = 32 * CS_ADD * CS_ADD_PER;
static_assert(CS_MAX_COLS <= 32 * CS_SQ * CS_SQ_PER, "both groups cover the columns");
constexpr int CS_DEPTH = 16;                       // gradients whose sums / factors are kept in shared memory (>= slots)
constexpr int CS_MAX_SLOTS = 16, CS_MISC = 2048, CS_SMEM = 227 * 1024;
struct ClipShared {
  uint64_t full[CS_MAX_SLOTS], empty[CS_MAX_SLOTS], norm_ready[CS_DEPTH], coef_ready[CS_DEPTH];
  float warp_sum[CS_DEPTH][CS_SQ];
  float coef[CS_DEPTH];
  volatile uint32_t abort_flag;
};
static_assert(sizeof(ClipShared) <= CS_MISC, "shared memory");

// Sixteen or more runs, so that what their own roundings add stays below the last one's; longer ones than 32 save no time.
inline int clip_fold(int64_t K) { return (int)(K / 16 < 1 ? 1 : (K / 16 > 32 ? 32 : K / 16)); }

__global__ void __launch_bounds__(CS_THREADS, 1) clip_sum_apply(const float4* __restrict__ queue, int K, int cols, int slots, int fold, float clip,
                                                                const float* __restrict__ coef_k, u64* words, const float4* theta_in,
                                                                float4* theta_out, float4* __restrict__ replica, uint32_t* status) {
  extern __shared__ __align__(128) uint8_t sm[];
  ClipShared* sh = reinterpret_cast<ClipShared*>(sm);
  float4* ring = reinterpret_cast<float4*>(sm + CS_MISC);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_cta = gridDim.x;
  const int col0 = blockIdx.x * cols, n = min(cols, P_VEC4 - col0);      // n > 0 for every block
  if (tid == 0) {
    for (int i = 0; i < slots; ++i) { mbar_init(&sh->full[i], 1); mbar_init(&sh->empty[i], CS_ADD); }
    for (int i = 0; i < CS_DEPTH; ++i) { mbar_init(&sh->norm_ready[i], CS_SQ); mbar_init(&sh->coef_ready[i], 1); }
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // true for the whole warp or for none of it
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (__all_sync(0xffffffffu, mbar_try(smem_u32(bar), parity))) return true;
    const bool done = mbar_wait(bar, parity) && !sh->abort_flag;
    if (__all_sync(0xffffffffu, done)) return true;
    sh->abort_flag = 1;
    return false;
  };
  bool ok = true;
  if (warp < CS_ADD) {
    // ---------------- sums
    u64 part[2 * CS_ADD_PER], acc[2 * CS_ADD_PER], err[2 * CS_ADD_PER];
#pragma unroll
    for (int j = 0; j < 2 * CS_ADD_PER; ++j) part[j] = acc[j] = err[j] = 0ull;
    int slot = 0, run = 0;
    for (int k = 0; k < K; ++k) {
      if (!(ok = wait(&sh->coef_ready[k % CS_DEPTH], (k / CS_DEPTH) & 1))) break;
      const float ck = sh->coef[k % CS_DEPTH];
      const u64 c = pack2(ck, ck);
      const float4* g = ring + slot * cols;
      float4 v[CS_ADD_PER];
#pragma unroll
      for (int j = 0; j < CS_ADD_PER; ++j) {
        const int i = tid + 32 * CS_ADD * j;
        v[j] = i < n ? g[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->empty[slot]);
#pragma unroll
      for (int j = 0; j < CS_ADD_PER; ++j) {
        part[2 * j] = ffma2(c, pack2(v[j].x, v[j].y), part[2 * j]);
        part[2 * j + 1] = ffma2(c, pack2(v[j].z, v[j].w), part[2 * j + 1]);
      }
      if (++run == fold || k == K - 1) {
        run = 0;
#pragma unroll
        for (int j = 0; j < 2 * CS_ADD_PER; ++j) {
          add_compensated(part[j], acc[j], err[j]);
          part[j] = 0ull;
        }
      }
      if (++slot == slots) slot = 0;
    }
    if (ok) {
#pragma unroll
      for (int j = 0; j < CS_ADD_PER; ++j) {
        const int i = tid + 32 * CS_ADD * j;
        if (i < n) {
          float4 t = theta_in[col0 + i];
          const float2 lo = compensated(acc[2 * j], err[2 * j]), hi = compensated(acc[2 * j + 1], err[2 * j + 1]);
          t.x -= lo.x; t.y -= lo.y; t.z -= hi.x; t.w -= hi.y;
          theta_out[col0 + i] = t;
          if (replica) replica[col0 + i] = t;
        }
      }
    }
  } else if (warp < CS_ADD + CS_SQ) {
    // ---------------- sums of squares
    const int id = tid - 32 * CS_ADD;
    int slot = 0;
    uint32_t phase = 0;
    for (int k = 0; k < K; ++k) {
      if (!(ok = wait(&sh->full[slot], phase))) break;
      const float4* g = ring + slot * cols;
      float s[CS_SQ_PER];
#pragma unroll
      for (int j = 0; j < CS_SQ_PER; ++j) {
        const int i = id + 32 * CS_SQ * j;
        const float4 v = i < n ? g[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        s[j] = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, v.w * v.w)));
      }
      float t = ((s[0] + s[1]) + (s[2] + s[3])) + (s[4] + s[5]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) { sh->warp_sum[k % CS_DEPTH][warp - CS_ADD] = t; mbar_arrive(&sh->norm_ready[k % CS_DEPTH]); }
      if (++slot == slots) { slot = 0; phase ^= 1; }
    }
  } else if (warp == CS_ADD + CS_SQ) {
    // ---------------- copies
    int slot = 0;
    uint32_t phase = 1;                              // flips to 0 when the first slot is used again
    for (int k = 0; k < K; ++k) {
      if (k >= slots && !(ok = wait(&sh->empty[slot], phase))) break;
      if (lane == 0) {
        mbar_expect_tx(&sh->full[slot], n * 16);
        bulk_load(ring + slot * cols, queue + k * (int64_t)P_VEC4 + col0, n * 16, &sh->full[slot]);
      }
      if (++slot == slots) { slot = 0; phase ^= 1; }
    }
  } else if (warp == CS_ADD + CS_SQ + 1) {
    // ---------------- this CTA's partial sums out
    for (int k = 0; k < K; ++k) {
      if (!(ok = wait(&sh->norm_ready[k % CS_DEPTH], (k / CS_DEPTH) & 1))) break;
      if (lane < CS_COPIES) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < CS_SQ; ++w) t += sh->warp_sum[k % CS_DEPTH][w];
        const u64 word = ((u64)(uint32_t)(k + 1) << 32) | __float_as_uint(t);
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(words + ((k % CS_RING) * CS_COPIES + lane) * NORM_WORDS + blockIdx.x), "l"(word) : "memory");
      }
    }
  } else {
    // ---------------- all CTAs' partial sums in, and the factor
    for (int k = warp - (CS_ADD + CS_SQ + 2); k < K; k += CS_GATHER) {
      const u64* w = words + ((k % CS_RING) * CS_COPIES + blockIdx.x % CS_COPIES) * NORM_WORDS;
      // a lane's words are asked for together, the missing ones again and again until all have arrived
      constexpr int PER_LANE = (NORM_WORDS + 31) / 32;
      u64 v[PER_LANE];
#pragma unroll
      for (int i = 0; i < PER_LANE; ++i) v[i] = lane + 32 * i < n_cta ? 0ull : (u64)(uint32_t)(k + 1) << 32;
      const long long t0 = clock64();
      for (;;) {
        bool all = true;
#pragma unroll
        for (int i = 0; i < PER_LANE; ++i)
          if ((uint32_t)(v[i] >> 32) != (uint32_t)(k + 1)) asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v[i]) : "l"(w + lane + 32 * i) : "memory");
#pragma unroll
        for (int i = 0; i < PER_LANE; ++i) all = all && (uint32_t)(v[i] >> 32) == (uint32_t)(k + 1);
        if (__all_sync(0xffffffffu, all)) break;
        if (__any_sync(0xffffffffu, clock64() - t0 > WAIT_LIMIT_CYCLES || sh->abort_flag)) { ok = false; break; }
        __nanosleep(20);
      }
      float t = 0.f;
#pragma unroll
      for (int i = 0; i < PER_LANE; ++i) t += __uint_as_float((uint32_t)v[i]);
      if (!__all_sync(0xffffffffu, ok)) { sh->abort_flag = 1; break; }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) {
        sh->coef[k % CS_DEPTH] = coef_k[k] * fminf(1.0f, clip / sqrtf(t));      // a zero gradient keeps its factor (clip / 0 = inf)
        mbar_arrive(&sh->coef_ready[k % CS_DEPTH]);
      }
    }
  }
  __syncthreads();
  if (tid == 0 && sh->abort_flag) {
    atomicOr(status, STATUS_WAIT_TIMEOUT);
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);      // let copies already issued land before the CTA ends
  }
}

}  // namespace

#define TIMED(id, launch) do { if (prof) prof->begin(id, st); launch; if (prof) prof->end(st); } while (0)

const char* kernel_name(int id) {
  static const char* names[K_COUNT] = {
      "conv1_fwd", "conv2_fwd", "fc1_fwd", "fc2_fwd_bwd", "fc1_dw", "fc1_dx", "conv2_bwd", "conv1_bwd",
      "conv_grad_reduce", "sum_apply_direct", "sum_partial", "sum_finish", "async_apply", "copy_rows",
      "dropout_mask", "conv2_dw", "prep_w1", "sq_norm_partial", "clip_coef_finish", "eval_finish", "clip_sum_apply"};
  return id >= 0 && id < K_COUNT ? names[id] : "?";
}

int launch_sum_apply(const SumApplyArgs& a, cudaStream_t st, Profiler* prof) {
  const float4* q = reinterpret_cast<const float4*>(a.queue);
  const float4* tin = reinterpret_cast<const float4*>(a.theta_in);
  float4* tout = reinterpret_cast<float4*>(a.theta_out);
  float4* rep = reinterpret_cast<float4*>(a.replica);
  int n_split = 1;
  if (a.K > 160 && a.max_split > 1) {
    int64_t want = (a.K + 31) / 32;
    n_split = (int)(want < a.max_split ? want : a.max_split);
  }
  int launches = 0;
  const float* ck = a.coef_k;
  const float coef = ck ? 1.0f : a.coef;      // the per-gradient factors already carry the learning rate
  if (n_split <= 1) {
    if (ck) TIMED(K_SUM_APPLY_DIRECT, (sum_apply_direct<true><<<COL_BLOCKS, TPB, 0, st>>>(q, a.K, tin, tout, rep, coef, ck)));
    else TIMED(K_SUM_APPLY_DIRECT, launch_pdl(sum_apply_direct<false>, dim3(COL_BLOCKS), TPB, 0, st, q, a.K, tin, tout, rep, coef, nullptr));
    launches = 1;
  } else {
    float4* part = reinterpret_cast<float4*>(a.partial);
    if (ck) TIMED(K_SUM_PARTIAL, (sum_partial<true><<<dim3(COL_BLOCKS, n_split), TPB, 0, st>>>(q, a.K, n_split, part, ck)));
    else TIMED(K_SUM_PARTIAL, launch_pdl(sum_partial<false>, dim3(COL_BLOCKS, n_split), TPB, 0, st, q, a.K, n_split, part, nullptr));
    TIMED(K_SUM_FINISH, launch_pdl(sum_finish, dim3(COL_BLOCKS), TPB, 0, st, part, n_split, tin, tout, rep, coef));
    launches = 2;
  }
  return cudaGetLastError() == cudaSuccess ? launches : -1;
}

int launch_clip_factors(const float* queue, int64_t K, float clip, float* coef_k, float* norm_part, cudaStream_t st, Profiler* prof) {
  TIMED(K_SQ_NORM, (sq_norm_partial<<<dim3(NORM_CHUNKS, (unsigned)K), TPB, 0, st>>>(reinterpret_cast<const float4*>(queue), norm_part)));
  TIMED(K_COEF_FINISH, (clip_coef_finish<<<(unsigned)((K + TPB - 1) / TPB), TPB, 0, st>>>(norm_part, K, clip, coef_k)));
  return cudaGetLastError() == cudaSuccess ? 2 : -1;
}

int configure_apply_kernels() {
  return allow_smem((const void*)clip_sum_apply, CS_SMEM) == cudaSuccess ? 0 : -1;
}

// The one-pass kernel's shape on a device of `sms` SMs: a CTA per SM, its columns, its ring of gradients.  A CTA's threads cover
// CS_MAX_COLS columns, so it takes 145 SMs or more.
struct ClipShape { int grid, cols, slots; };
static ClipShape clip_shape(int sms) {
  ClipShape c;
  c.grid = std::min(std::max(sms, 1), NORM_WORDS);
  c.cols = (P_VEC4 + c.grid - 1) / c.grid;
  c.slots = std::min(CS_MAX_SLOTS, (CS_SMEM - CS_MISC) / (c.cols * 16));
  return c;
}
bool clip_sum_fits(int sms) {
  const ClipShape c = clip_shape(sms);
  return c.cols <= CS_MAX_COLS && c.slots >= 3 && (int64_t)(c.grid - 1) * c.cols < P_VEC4;
}

int launch_clip_sum_apply(const SumApplyArgs& a, float clip, uint64_t* words, uint32_t* status, cudaStream_t st, Profiler* prof) {
  if (!clip_sum_fits(g_sm_count)) return 0;
  const ClipShape c = clip_shape(g_sm_count);
  if (cudaMemsetAsync(words, 0, CLIP_EXCHANGE_BYTES, st) != cudaSuccess) return -1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c.grid);
  cfg.blockDim = dim3(CS_THREADS);
  cfg.dynamicSmemBytes = (size_t)(CS_MISC + c.slots * c.cols * 16);
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaError_t e = cudaSuccess;
  TIMED(K_CLIP_SUM, e = cudaLaunchKernelEx(&cfg, clip_sum_apply, reinterpret_cast<const float4*>(a.queue), (int)a.K, c.cols, c.slots, clip_fold(a.K),
                                           clip, a.coef_k, reinterpret_cast<u64*>(words), reinterpret_cast<const float4*>(a.theta_in),
                                           reinterpret_cast<float4*>(a.theta_out), reinterpret_cast<float4*>(a.replica), status));
  if (e == cudaErrorCooperativeLaunchTooLarge) {      // a stream that may use part of the device only
    cudaGetLastError();
    return 0;
  }
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_async_apply(const AsyncApplyArgs& a, const AsyncOrder& ord, cudaStream_t st, Profiler* prof) {
  TIMED(K_ASYNC_APPLY, launch_pdl(async_apply, dim3(COL_BLOCKS), TPB, 0, st, a, ord));
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_copy_rows(float* dst, const float* src, int64_t rows, cudaStream_t st, Profiler* prof) {
  int64_t n_vec = rows * P_VEC4;
  int64_t blocks = (n_vec + TPB - 1) / TPB;
  if (blocks > 148 * 16) blocks = 148 * 16;
  TIMED(K_COPY_ROWS, (copy_rows<<<(int)blocks, TPB, 0, st>>>(reinterpret_cast<float4*>(dst),
                                                            reinterpret_cast<const float4*>(src), n_vec)));
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace psk
