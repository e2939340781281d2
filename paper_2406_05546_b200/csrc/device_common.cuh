// Device helpers shared by the grad-step kernel files.
#pragma once
#include <utility>
#include "kernels.h"

namespace psk {

// Programmatic dependent launch.  A kernel launched with launch_pdl may start while the kernel before it in the stream still
// runs; up to pdl_enter() it may only set itself up and read what kernels before that one have written (every kernel of the
// chain enters before it lets the next one start, so those have finished).  The launch and the set-up of a kernel then
// overlap the one before: us per pass without -> with, tensor-core path: 5 x 37 102 -> 83, 8 x 64 107 -> 94, 128 x 128 691 -> 681,
// evaluation 80 x 125 179 -> 168.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---- Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplications; the high
// halves are xored with the neighbouring counter words and the key; the key advances by two Weyl
// constants per round.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
  constexpr uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
    uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += W0; k.y += W1;
  }
  return c;
}

// Pairs of fp32 values in one 64-bit register, for the packed multiply-add.
typedef unsigned long long u64;
__device__ __forceinline__ u64 pack2(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(u64 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// Two independent single-rounded fp32 multiply-adds in one instruction.
__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// Asynchronous copies global -> shared, in groups.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
// 16 bytes; zeros if !valid
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The largest of three (a NaN counts as less than anything).
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Rounds to TF32 (10-bit mantissa, nearest, ties away from zero); the result is still an fp32 value.
__device__ __forceinline__ float round_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// fp32 -> BF16, round to nearest even.
__device__ __forceinline__ uint16_t bf16_bits(float x) {
  uint16_t r;
  asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {   // lo in the low half
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// prmt.b32 in its default mode: selector nibble n picks byte (n & 7) of {b, a}; with bit 3 of the nibble set, the
// picked byte's top bit is replicated over the whole output byte instead.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t selector) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(selector));
  return r;
}
// x << n for a 64-bit x, with n >= 64 giving 0 (PTX clamps the shift amount; C++ leaves it undefined).
__device__ __forceinline__ unsigned long long shl64_clamped(unsigned long long x, uint32_t n) {
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
}

// Where element (channel oc, pooled position p) of a sample's pooled gradient dp2 and of its pooling decisions
// sits on the tensor-core path: [channel quad][position][4 channels], so that a thread of the backward
// kernels takes four channels of a position with one vector load.  `canonical` = oc * 49 + p.
__host__ __device__ __forceinline__ int dp2_column(int canonical) {
  const int oc = canonical / 49, p = canonical - oc * 49;
  return (oc >> 2) * 196 + p * 4 + (oc & 3);
}

__device__ __forceinline__ const float* group_theta(const WorkerTable& wt, const GroupTable& gt, int s) {
  return gt.theta[wt.group[s]];
}

// bias + ReLU + dropout of four consecutive units n..n+3 of row m.  (tc5_gemm's epilogue has its own: a lane stays on one row
// there and keeps what depends on it; calling this made an evaluation of 10,000 samples 2 us longer.)
__device__ __forceinline__ float4 fc1_activation(float4 v, int m, int n, const float* theta, const GradStepArgs& a, const WorkerTable& wt) {
  const float4 bias = *reinterpret_cast<const float4*>(theta + OFF_F1B + n);
  const float scale = 1.0f / (1.0f - a.drop_p);
  const int s = m / a.b, i = m - s * a.b;
  const uint4 rnd = philox4x32_10(make_uint4((uint32_t)((i * HID + n) >> 2), (uint32_t)wt.wid[s], (uint32_t)a.step, (uint32_t)(a.step >> 32)),
                                  make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32)));
  return make_float4(rnd.x >= a.drop_thresh ? fmaxf(v.x + bias.x, 0.f) * scale : 0.f, rnd.y >= a.drop_thresh ? fmaxf(v.y + bias.y, 0.f) * scale : 0.f,
                     rnd.z >= a.drop_thresh ? fmaxf(v.z + bias.z, 0.f) * scale : 0.f, rnd.w >= a.drop_thresh ? fmaxf(v.w + bias.w, 0.f) * scale : 0.f);
}

// Maps a tile index to (group, first row of the tile, end row of the group) for TM-row tiles laid
// out group after group.
template <int TM>
__device__ __forceinline__ bool locate_group_tile(const GroupTable& gt, int b, int tile, int& g, int& m0, int& m_end) {
  for (g = 0; g < gt.n_groups; ++g) {
    int rows = (gt.first[g + 1] - gt.first[g]) * b;
    int tiles = (rows + TM - 1) / TM;
    if (tile < tiles) {
      m0 = gt.first[g] * b + tile * TM;
      m_end = gt.first[g + 1] * b;
      return true;
    }
    tile -= tiles;
  }
  return false;
}

// Same with a run-time range length: range `index` covers rows [r0, r1) of weight group g (ranges never cross
// from one weight group into the next).  False past the last range.
__device__ __forceinline__ bool locate_row_range(const GroupTable& gt, int b, int len, int index, int& g, int& r0, int& r1) {
  for (g = 0; g < gt.n_groups; ++g) {
    const int first = gt.first[g] * b, end = gt.first[g + 1] * b;
    const int n = (end - first + len - 1) / len;
    if (index < n) {
      r0 = first + index * len;
      r1 = min(r0 + len, end);
      return true;
    }
    index -= n;
  }
  return false;
}

// Host: a range length (a multiple of `unit` rows) that gives about `slots` ranges over all rows, and the number
// of ranges it makes when no range crosses a weight-group boundary.
inline int plan_row_ranges(const GroupTable& gt, int b, int slots, int unit, int* len_out) {
  const int total = gt.first[gt.n_groups] * b;
  int len = (total + slots - 1) / slots;
  len = (len + unit - 1) / unit * unit;
  if (len < unit) len = unit;
  int n = 0;
  for (int g = 0; g < gt.n_groups; ++g) n += ((gt.first[g + 1] - gt.first[g]) * b + len - 1) / len;
  *len_out = len;
  return n;
}

inline int group_tiles(const GroupTable& gt, int b, int tm) {
  int t = 0;
  for (int g = 0; g < gt.n_groups; ++g) t += ((gt.first[g + 1] - gt.first[g]) * b + tm - 1) / tm;
  return t;
}

// Host: launches a kernel that may start before the one before it in the stream has ended (see pdl_enter).  The attribute lifts
// the dependence on that kernel only: a wait for another stream's event holds back all work behind it, this launch included.
// Where the launch code has put such a wait just before the kernel there is nothing to overlap, and `overlap` false makes it a
// plain launch; where the caller has, out of this code's sight, the kernel starts when the wait is over and finds the kernel
// before it ended or waits for it.
template <typename... P, typename... A>
inline void launch_pdl_if(bool overlap, void (*fn)(P...), dim3 grid, int threads, int smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, fn, static_cast<P>(std::forward<A>(args))...);
}
template <typename... P, typename... A>
inline void launch_pdl(void (*fn)(P...), dim3 grid, int threads, int smem, cudaStream_t st, A&&... args) {
  launch_pdl_if(true, fn, grid, threads, smem, st, std::forward<A>(args)...);
}

// Host: the same in clusters of cluster_z blocks along z.
template <typename F, typename... Args>
inline void launch_cluster(F* fn, dim3 grid, int threads, int smem, int cluster_z, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = (unsigned)cluster_z;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  cudaLaunchKernelEx(&cfg, fn, args...);
}

}  // namespace psk
