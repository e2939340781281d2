// The three products of the 512-unit dense layer on the FP32 path:
//   forward          C[m][n] = sum_k p2[m][k] * W1[n][k]      (rows of one weight group; bias, ReLU, dropout)
//   input gradient   C[m][n] = sum_k dA1[m][k] * W1[k][n]     (rows of one weight group)
//   weight gradient  C[m][n] = sum_k dA1[k][m] * p2[k][n]     (k = the samples of one worker)
// 802,816 multiply-adds per sample each; at large sizes the FP32 pipes bound them, at small ones latency does.
//
// sgemm_tile: 256 threads, a (16 TM) x (16 TN) tile in registers (TM x TN sums per thread, packed multiply-adds over
// pairs of columns), 16 values of k per step in a three-stage shared-memory ring.  A operand with k contiguous stays as
// it lies ([row][16 k], a thread takes four k with one 16-byte load); the B operand must have its columns contiguous for
// the packed multiply-adds, so W1 of the forward product is transposed on its way through registers.
// Few rows have forms of their own: the forward product keeps every sum's order of k (sgemm_fwd_seq, sgemm_fwd_rows), the
// input gradient splits k over a cluster (sgemm_dx_skinny, sgemm_tile with SPLIT), whose partial tiles are added through
// distributed shared memory in a fixed order.
//
// Measured (B200; 26.3 GFLOP per product at 128 workers x 128 samples, 0.36 ms at the FP32 pipes' rate): forward 0.78 -> 0.56,
// input gradient 0.74 -> 0.54, weight gradient 0.72 -> 0.52 ms; at 2 x 8: 89 -> 18, 33 -> 11, 9 -> 9 us (event overhead
// of ~6 us included).  The former kernels took 64 x 64 x 16 tiles with 4 x 4 sums per thread and nothing in flight.
#include <cooperative_groups.h>

#include "device_common.cuh"
#include "kernels.h"

namespace psk {

namespace {

namespace cg = cooperative_groups;

enum { G_FWD = 0, G_DX = 1, G_DW = 2 };
template <int OP> struct GemmShape {
  static constexpr int N = OP == G_FWD ? HID : FLAT;
  static constexpr bool A_K = OP != G_DW, B_K = OP == G_FWD;      // is k the contiguous index of the operand?
  static constexpr int LDA = OP == G_FWD ? FLAT : HID, LDB = FLAT, LDC = N;
};

// Operands and destination of the block's tile: rows m0 .. m_end - 1 (all of them < m_end are valid)
struct TileIo { const float *A, *B, *theta; float* C; int m0, m_end, K; };
template <int OP, int BM>
__device__ __forceinline__ bool locate_tile(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, TileIo& io) {
  if (OP == G_DW) {
    const int s = blockIdx.z;
    io.A = ws.da1 + (int64_t)s * a.b * HID;
    io.B = ws.p2 + (int64_t)s * a.b * FLAT;
    io.theta = nullptr;
    io.C = wt.grad[s] + OFF_F1W;
    io.m0 = blockIdx.y * BM;
    io.m_end = HID;
    io.K = a.b;
    return true;
  }
  int g;
  if (!locate_group_tile<BM>(gt, a.b, blockIdx.y, g, io.m0, io.m_end)) return false;
  io.theta = gt.theta[g];
  io.A = OP == G_FWD ? ws.p2 : ws.da1;
  io.B = io.theta + OFF_F1W;
  io.C = OP == G_FWD ? ws.d : ws.dp2;
  io.K = OP == G_FWD ? FLAT : HID;
  return true;
}

constexpr int GK = 16, G_STAGES = 3, GA_PITCH = GK + 4;      // 20-word rows: 16-byte loads of consecutive rows meet no bank twice
template <int OP, int TM, int TN> struct Tile {
  static constexpr int BM = 16 * TM, BN = 16 * TN, B_PITCH = GemmShape<OP>::B_K ? BN + 4 : BN;
  static constexpr int A_WORDS = GemmShape<OP>::A_K ? BM * GA_PITCH : GK * BM, B_WORDS = GK * B_PITCH;
  static constexpr int STAGE = A_WORDS + B_WORDS, SMEM = 4 * G_STAGES * STAGE;
  static_assert(A_WORDS % 4 == 0 && STAGE % 4 == 0, "16-byte pieces");
  static_assert(SMEM >= 4 * BM * BN || TM > 4, "a partial tile fits the ring (split products)");
};

// grid: (column tiles, row tiles, split of k (cluster) or workers)
template <int OP, int TM, int TN, bool SPLIT>
__global__ void __launch_bounds__(256, 2) sgemm_tile(GradStepArgs a, WorkerTable wt, GroupTable gt, Workspace ws) {
  using S = GemmShape<OP>;
  using T = Tile<OP, TM, TN>;
  constexpr int BM = T::BM, BN = T::BN;
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ty = (warp >> 1) * 4 + (lane >> 3), tx = (warp & 1) * 8 + (lane & 7);     // a warp covers 4 x 8 threads of the 16 x 16
  TileIo io;
  if (!locate_tile<OP, BM>(a, wt, gt, ws, io)) return;
  pdl_enter();
  const int n0 = blockIdx.x * BN;
  int kt0 = 0, kt1 = (io.K + GK - 1) / GK;
  if (SPLIT) {
    const int per = (kt1 + gridDim.z - 1) / gridDim.z;
    kt0 = min(kt1, (int)blockIdx.z * per);
    kt1 = min(kt1, kt0 + per);
  }
  constexpr int PER_A = (TM + 3) / 4, PER_B = TN / 4;       // 16-byte pieces per thread and step
  float4 breg[S::B_K ? PER_B : 1];
  auto issue = [&](int kt, int buf) {                       // copies of step kt (and, for a transposed B, the loads into registers)
    float* As = sm + buf * T::STAGE;
    float* Bs = As + T::A_WORDS;
#pragma unroll
    for (int p = 0; p < PER_A; ++p) {
      const int e = tid + 256 * p;
      if (TM % 4 != 0 && e >= 4 * BM) break;
      if (S::A_K) {
        const int m = e >> 2, kq = (e & 3) * 4, k = kt * GK + kq;
        cp_async16(As + m * GA_PITCH + kq, io.A + (int64_t)min(io.m0 + m, io.m_end - 1) * S::LDA + k, true);
      } else {
        const int kk = e / (BM / 4), mq = (e % (BM / 4)) * 4, k = kt * GK + kk;
        cp_async16(As + kk * BM + mq, io.A + (int64_t)min(k, io.K - 1) * S::LDA + io.m0 + mq, k < io.K);
      }
    }
#pragma unroll
    for (int p = 0; p < PER_B; ++p) {
      const int e = tid + 256 * p;
      if (S::B_K) {
        const int n = e >> 2, k = kt * GK + (e & 3) * 4;
        breg[p] = *reinterpret_cast<const float4*>(io.B + (int64_t)(n0 + n) * S::LDB + k);
      } else {
        const int kk = e / (BN / 4), nq = (e % (BN / 4)) * 4, k = kt * GK + kk;
        const bool in = k < io.K && n0 + nq < S::N;
        cp_async16(Bs + kk * T::B_PITCH + nq, in ? io.B + (int64_t)k * S::LDB + n0 + nq : io.B, in);
      }
    }
    cp_async_commit();
  };
  auto place = [&](int buf) {                               // the transposed B operand of the step just issued
    if (!S::B_K) return;
    float* Bs = sm + buf * T::STAGE + T::A_WORDS;
#pragma unroll
    for (int p = 0; p < PER_B; ++p) {
      const int e = tid + 256 * p, n = e >> 2, kq = (e & 3) * 4;
      Bs[kq * T::B_PITCH + n] = breg[p].x;
      Bs[(kq + 1) * T::B_PITCH + n] = breg[p].y;
      Bs[(kq + 2) * T::B_PITCH + n] = breg[p].z;
      Bs[(kq + 3) * T::B_PITCH + n] = breg[p].w;
    }
  };
  u64 acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
#pragma unroll
  for (int s = 0; s < G_STAGES - 1; ++s) {
    if (kt0 + s < kt1) { issue(kt0 + s, s); place(s); }
    else cp_async_commit();
  }
  int buf = 0;
  for (int kt = kt0; kt < kt1; ++kt) {
    cp_async_wait<G_STAGES - 2>();
    __syncthreads();                                        // step kt is complete; the buffer of step kt - 1 is free
    const int nbuf = buf == 0 ? G_STAGES - 1 : buf - 1;
    const bool more = kt + G_STAGES - 1 < kt1;
    if (more) issue(kt + G_STAGES - 1, nbuf);
    else cp_async_commit();
    const float* As = sm + buf * T::STAGE;
    const float* Bs = As + T::A_WORDS;
#pragma unroll
    for (int kq = 0; kq < GK; kq += 4) {
      float av[TM][4];                                      // [row][k]
      if (S::A_K) {
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const float4 v = *reinterpret_cast<const float4*>(As + (ty + 16 * i) * GA_PITCH + kq);
          av[i][0] = v.x; av[i][1] = v.y; av[i][2] = v.z; av[i][3] = v.w;
        }
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        u64 bv[TN / 2];
#pragma unroll
        for (int q = 0; q < TN / 4; ++q) {
          const float4 v = *reinterpret_cast<const float4*>(Bs + (kq + kk) * T::B_PITCH + tx * 4 + 64 * q);
          bv[2 * q] = pack2(v.x, v.y); bv[2 * q + 1] = pack2(v.z, v.w);
        }
        if (!S::A_K) {
#pragma unroll
          for (int q = 0; q < TM / 4; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(As + (kq + kk) * BM + ty * 4 + 64 * q);
            av[4 * q][kk] = v.x; av[4 * q + 1][kk] = v.y; av[4 * q + 2][kk] = v.z; av[4 * q + 3][kk] = v.w;
          }
        }
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const u64 ad = pack2(av[i][kk], av[i][kk]);
#pragma unroll
          for (int j = 0; j < TN / 2; ++j) acc[i][j] = ffma2(bv[j], ad, acc[i][j]);
        }
      }
    }
    if (more) place(nbuf);
    buf = buf == G_STAGES - 1 ? 0 : buf + 1;
  }
  cp_async_wait<0>();
  auto row_of = [&](int i) { return S::A_K ? ty + 16 * i : ty * 4 + 64 * (i >> 2) + (i & 3); };
  auto store = [&](int m, int n, float4 v) {
    if (OP == G_FWD) v = fc1_activation(v, m, n, io.theta, a, wt);
    *reinterpret_cast<float4*>(io.C + (int64_t)m * S::LDC + n) = v;
  };
  if constexpr (SPLIT) {
    // partial tiles through distributed shared memory: rank r adds its share of the tile over all ranks in order
    cg::cluster_group cl = cg::this_cluster();
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int q = 0; q < TN / 4; ++q) {
        float4 v;
        unpack2(acc[i][2 * q], v.x, v.y);
        unpack2(acc[i][2 * q + 1], v.z, v.w);
        *reinterpret_cast<float4*>(sm + row_of(i) * BN + tx * 4 + 64 * q) = v;
      }
    cl.sync();
    const int ranks = gridDim.z, rank = blockIdx.z;
    for (int e = rank * 256 + tid; e < BM * BN / 4; e += ranks * 256) {
      const int m = io.m0 + e / (BN / 4), n = n0 + (e % (BN / 4)) * 4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int r = 0; r < ranks; ++r) {
        const float4 u = reinterpret_cast<const float4*>(cl.map_shared_rank(sm, r))[e];
        v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
      }
      if (m < io.m_end && n < S::N) store(m, n, v);
    }
    cl.sync();                                              // a CTA's shared memory outlives its readers
  } else {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int m = io.m0 + row_of(i);
      if (m >= io.m_end) continue;
#pragma unroll
      for (int q = 0; q < TN / 4; ++q) {
        const int n = n0 + tx * 4 + 64 * q;
        if (n >= S::N) continue;
        float4 v;
        unpack2(acc[i][2 * q], v.x, v.y);
        unpack2(acc[i][2 * q + 1], v.z, v.w);
        store(m, n, v);
      }
    }
  }
}

// Forward product, few rows: tiles of TM x TN with RM x RN sums per thread of 128, every sum taken over k in order (a split
// of k would change its last bits, and with them the sign of a unit whose sum lies within rounding distance of zero).  Both
// operands stay as they lie, k contiguous; a thread takes four k of each with 16-byte loads, and steps of 32 k arrive in a
// three-stage ring of asynchronous copies.
constexpr int SQ_K = 32, SQ_PITCH = SQ_K + 4, SQ_STAGES = 3;
template <int TM, int TN, int RM, int RN>
__global__ void __launch_bounds__(128) sgemm_fwd_seq(GradStepArgs a, WorkerTable wt, GroupTable gt, Workspace ws) {
  constexpr int TX = TN / RN, TY = TM / RM, STAGE = (TM + TN) * SQ_PITCH, STEPS = FLAT / SQ_K;
  static_assert(TX * TY == 128 && FLAT % SQ_K == 0 && SQ_STAGES * STAGE * 4 <= 48 * 1024, "tile shape");
  __shared__ __align__(16) float sm[SQ_STAGES * STAGE];
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX, n0 = blockIdx.x * TN;
  TileIo io;
  if (!locate_tile<G_FWD, TM>(a, wt, gt, ws, io)) return;
  pdl_enter();
  auto issue = [&](int step, int buf) {
    if (step < STEPS) {
      float* dst = sm + buf * STAGE;
#pragma unroll
      for (int e0 = 0; e0 < (TM + TN) * 8; e0 += 128) {
        const int e = e0 + tid, r = e >> 3, kq = (e & 7) * 4, k = step * SQ_K + kq;
        const float* src = r < TM ? io.A + (int64_t)min(io.m0 + r, io.m_end - 1) * FLAT + k : io.B + (int64_t)(n0 + r - TM) * FLAT + k;
        cp_async16(dst + r * SQ_PITCH + kq, src, true);
      }
    }
    cp_async_commit();
  };
  float acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = 0.f;
#pragma unroll
  for (int s = 0; s < SQ_STAGES - 1; ++s) issue(s, s);
  for (int step = 0; step < STEPS; ++step) {
    cp_async_wait<SQ_STAGES - 2>();
    __syncthreads();                                        // this step is complete; the buffer of the one before is free
    issue(step + SQ_STAGES - 1, (step + SQ_STAGES - 1) % SQ_STAGES);
    const float* As = sm + (step % SQ_STAGES) * STAGE;
    const float* Bs = As + TM * SQ_PITCH;
#pragma unroll
    for (int kq = 0; kq < SQ_K; kq += 4) {
      float4 av[RM], bv[RN];
#pragma unroll
      for (int i = 0; i < RM; ++i) av[i] = *reinterpret_cast<const float4*>(As + (ty + TY * i) * SQ_PITCH + kq);
#pragma unroll
      for (int j = 0; j < RN; ++j) bv[j] = *reinterpret_cast<const float4*>(Bs + (tx + TX * j) * SQ_PITCH + kq);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(av[i].x, bv[j].x, acc[i][j]);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(av[i].y, bv[j].y, acc[i][j]);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(av[i].z, bv[j].z, acc[i][j]);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(av[i].w, bv[j].w, acc[i][j]);
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  // four consecutive units share a draw of the dropout generator: through shared memory into that order
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) sm[(ty + TY * i) * (TN + 4) + tx + TX * j] = acc[i][j];
  __syncthreads();
  for (int e = tid; e < TM * TN / 4; e += 128) {
    const int r = e / (TN / 4), m = io.m0 + r, q = e % (TN / 4), n = n0 + 4 * q;
    if (m < io.m_end)
      *reinterpret_cast<float4*>(io.C + (int64_t)m * HID + n) = fc1_activation(*reinterpret_cast<const float4*>(sm + r * (TN + 4) + 4 * q), m, n, io.theta, a, wt);
  }
}

// A load the compiler leaves where it stands: it would otherwise sink every operand to its use, and the chain of
// multiply-adds would wait for shared memory at every step.
__device__ __forceinline__ float4 lds4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// The same for very few rows: a tile of 16 x 16 whose operands (16 rows of each, all of k) fit into shared memory at once.
// They arrive by asynchronous copies in seven chunks of k, all asked for at the start, so that little but the chain of a
// sum's 1,568 multiply-adds takes time once the first chunk has landed.
constexpr int RW_CHUNKS = 7, RW_K = FLAT / RW_CHUNKS, RW_PITCH = FLAT + 4;     // 1,572 words: rows four banks apart
constexpr int RW_SMEM = 32 * RW_PITCH * 4;
static_assert(RW_CHUNKS == 7 && 32 * RW_K / 4 % 128 == 0, "the waits below; whole rounds of copies");
__global__ void __launch_bounds__(128) sgemm_fwd_rows(GradStepArgs a, WorkerTable wt, GroupTable gt, Workspace ws) {
  extern __shared__ __align__(16) float sm[];
  __shared__ __align__(16) float out[16 * 20];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, n0 = blockIdx.x * 16;
  TileIo io;
  if (!locate_tile<G_FWD, 16>(a, wt, gt, ws, io)) return;
  pdl_enter();
  for (int c = 0; c < RW_CHUNKS; ++c) {
#pragma unroll
    for (int i = 0; i < 32 * RW_K / 4 / 128; ++i) {
      const int e = tid + 128 * i, r = e / (RW_K / 4), k = c * RW_K + 4 * (e % (RW_K / 4));
      cp_async16(sm + r * RW_PITCH + k, r < 16 ? io.A + (int64_t)min(io.m0 + r, io.m_end - 1) * FLAT + k : io.B + (int64_t)(n0 + r - 16) * FLAT + k, true);
    }
    cp_async_commit();
  }
  float acc0 = 0.f, acc1 = 0.f;
  const float* ar = sm + ty * RW_PITCH;
  const float *b0 = sm + (16 + tx) * RW_PITCH, *b1 = b0 + 8 * RW_PITCH;
#pragma unroll
  for (int c = 0; c < RW_CHUNKS; ++c) {
    if (c == 0) cp_async_wait<6>();
    else if (c == 1) cp_async_wait<5>();
    else if (c == 2) cp_async_wait<4>();
    else if (c == 3) cp_async_wait<3>();
    else if (c == 4) cp_async_wait<2>();
    else if (c == 5) cp_async_wait<1>();
    else cp_async_wait<0>();
    __syncthreads();
    // groups of 16 k, the next group's operands on their way while this one's products are added
    const uint32_t ak = (uint32_t)__cvta_generic_to_shared(ar + c * RW_K), b0k = (uint32_t)__cvta_generic_to_shared(b0 + c * RW_K), b1k = (uint32_t)__cvta_generic_to_shared(b1 + c * RW_K);
    float4 av[2][4], v0[2][4], v1[2][4];
    auto load = [&](int g, int buf) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        av[buf][u] = lds4(ak + 16 * (4 * g + u));
        v0[buf][u] = lds4(b0k + 16 * (4 * g + u));
        v1[buf][u] = lds4(b1k + 16 * (4 * g + u));
      }
    };
    load(0, 0);
#pragma unroll
    for (int g = 0; g < RW_K / 16; ++g) {
      if (g + 1 < RW_K / 16) load(g + 1, (g + 1) & 1);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 x = av[g & 1][u], y = v0[g & 1][u], z = v1[g & 1][u];
        acc0 = fmaf(x.x, y.x, acc0); acc1 = fmaf(x.x, z.x, acc1);
        acc0 = fmaf(x.y, y.y, acc0); acc1 = fmaf(x.y, z.y, acc1);
        acc0 = fmaf(x.z, y.z, acc0); acc1 = fmaf(x.z, z.z, acc1);
        acc0 = fmaf(x.w, y.w, acc0); acc1 = fmaf(x.w, z.w, acc1);
      }
    }
  }
  out[ty * 20 + tx] = acc0;
  out[ty * 20 + tx + 8] = acc1;
  __syncthreads();
  if (tid < 64) {
    const int r = tid >> 2, m = io.m0 + r, n = n0 + 4 * (tid & 3);
    if (m < io.m_end)
      *reinterpret_cast<float4*>(io.C + (int64_t)m * HID + n) = fc1_activation(*reinterpret_cast<const float4*>(out + r * 20 + 4 * (tid & 3)), m, n, io.theta, a, wt);
  }
}

// Input gradient, few rows: tile of 16 rows x 32 columns, k split over a cluster of four CTAs and, inside a CTA, over two
// halves of its threads.  A CTA fetches its whole slice of k at once: one exposed latency.
constexpr int DXS_KS = 4, DXS_SLICE = HID / DXS_KS, DXS_PITCH = DXS_SLICE + 4;      // rows meet no bank twice
constexpr int DXS_SMEM = 4 * (16 * DXS_PITCH + DXS_SLICE * 32 + 2 * 16 * 32);
__global__ void __launch_bounds__(256) sgemm_dx_skinny(GradStepArgs a, WorkerTable wt, GroupTable gt, Workspace ws) {
  extern __shared__ __align__(16) float sm[];
  float *As = sm, *Bs = sm + 16 * DXS_PITCH, *part = Bs + DXS_SLICE * 32;
  const int tid = threadIdx.x, n0 = blockIdx.x * 32, rank = blockIdx.z, k0 = rank * DXS_SLICE;
  TileIo io;
  if (!locate_tile<G_DX, 16>(a, wt, gt, ws, io)) return;    // the same for all CTAs of a cluster
  pdl_enter();
  for (int e = tid; e < 16 * (DXS_SLICE / 4); e += 256) {
    const int m = e / (DXS_SLICE / 4), kq = (e % (DXS_SLICE / 4)) * 4;
    cp_async16(As + m * DXS_PITCH + kq, io.A + (int64_t)min(io.m0 + m, io.m_end - 1) * HID + k0 + kq, true);
  }
  for (int e = tid; e < 8 * DXS_SLICE; e += 256) {
    const int k = e >> 3, nq = (e & 7) * 4;
    cp_async16(Bs + k * 32 + nq, io.B + (int64_t)(k0 + k) * FLAT + n0 + nq, true);
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  const int half = tid >> 7, r = (tid & 127) >> 3, c = tid & 7;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};                      // columns 4 c + j
#pragma unroll 4
  for (int k = half * (DXS_SLICE / 2); k < (half + 1) * (DXS_SLICE / 2); k += 4) {
    const float4 av = *reinterpret_cast<const float4*>(As + r * DXS_PITCH + k);
    const float ak[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const float4 bv = *reinterpret_cast<const float4*>(Bs + (k + kk) * 32 + 4 * c);
      acc[0] = fmaf(ak[kk], bv.x, acc[0]); acc[1] = fmaf(ak[kk], bv.y, acc[1]);
      acc[2] = fmaf(ak[kk], bv.z, acc[2]); acc[3] = fmaf(ak[kk], bv.w, acc[3]);
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) part[half * 512 + r * 32 + 4 * c + j] = acc[j];
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  for (int e = rank + DXS_KS * tid; e < 128; e += DXS_KS * 256) {      // 128 quads of the tile, dealt out over the ranks
    const int m = io.m0 + (e >> 3), n = n0 + (e & 7) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < DXS_KS; ++q) {
      const float4* p = reinterpret_cast<const float4*>(cl.map_shared_rank(part, q));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 u = p[h * 128 + e];
        v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
      }
    }
    if (m < io.m_end) *reinterpret_cast<float4*>(io.C + (int64_t)m * FLAT + n) = v;
  }
  cl.sync();
}

// Which form a grouped product takes, by its number of rows.  us, with ~6 us of event overhead:
//   rows                     16   64   128   256   384   512   768   1024   1280   2048   4096   16384
//   forward       16 x 16    18   19    29    52
//                 32 x 16    22   21    22    30    40    52    74     85    105
//                 64 x 16              29    29    48    48    56     72     89    119
//                 128 x 64                                                   99     99    179     590
//                 112 x 128                                                        162    163     562
//                 (64 x 64 with k split over a cluster, other bits: 17 at 64 rows, 25 at 256, 37 at 512, 64 at 1024)
//   input grad.   skinny     11   17    27    43
//                 64 x 64    17   13    17    23          35           58           103
//                 128 x 64                                                   61     87    162     567
//                 112 x 128                                                         92    173     540
// (64 x 64: k split over a cluster of up to four CTAs, about 400 in all, at least eight steps of k each.)
// Beyond that the time is the number of tiles per SM times a tile's time, which for tiles taken two at a time is
// 0.86 of a single one's: 112 x 128 tiles cost 1 alone and 1.73 as a pair, 128 x 64 tiles 0.605 and 1.1.
template <int OP>
void run_grouped(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st) {
  constexpr int N = GemmShape<OP>::N;
  const int rows = a.W * a.b;
  if constexpr (OP == G_FWD) {
    if (rows <= 1280) {
      if (rows <= 64) launch_pdl(sgemm_fwd_rows, dim3(HID / 16, group_tiles(gt, a.b, 16)), 128, RW_SMEM, st, a, wt, gt, ws);
      else if (rows <= 448) launch_pdl(sgemm_fwd_seq<32, 16, 2, 2>, dim3(HID / 16, group_tiles(gt, a.b, 32)), 128, 0, st, a, wt, gt, ws);
      else launch_pdl(sgemm_fwd_seq<64, 16, 4, 2>, dim3(HID / 16, group_tiles(gt, a.b, 64)), 128, 0, st, a, wt, gt, ws);
      return;
    }
  } else {
    if (rows <= 32) {
      launch_cluster(sgemm_dx_skinny, dim3(N / 32, group_tiles(gt, a.b, 16), DXS_KS), 256, DXS_SMEM, DXS_KS, st, a, wt, gt, ws);
      return;
    }
    if (rows <= 1024) {
      const dim3 grid((N + 63) / 64, group_tiles(gt, a.b, 64));
      unsigned split = 1;
      while (split < 4 && grid.x * grid.y * split * 2 <= 400u) split *= 2;
      launch_cluster(sgemm_tile<OP, 4, 4, true>, dim3(grid.x, grid.y, split), 256, Tile<OP, 4, 4>::SMEM, (int)split, st, a, wt, gt, ws);
      return;
    }
  }
  const dim3 wide((N + 127) / 128, group_tiles(gt, a.b, 112)), narrow((N + 63) / 64, group_tiles(gt, a.b, 128));
  auto cost = [](const dim3& grid, float one, float two) {
    const int n = (int)((grid.x * grid.y + g_sm_count - 1) / g_sm_count);
    return (n / 2) * two + (n & 1) * one;
  };
  if (cost(wide, 1.f, 1.73f) < cost(narrow, 0.605f, 1.1f)) launch_pdl(sgemm_tile<OP, 7, 8, false>, wide, 256, Tile<OP, 7, 8>::SMEM, st, a, wt, gt, ws);
  else launch_pdl(sgemm_tile<OP, 8, 4, false>, narrow, 256, Tile<OP, 8, 4>::SMEM, st, a, wt, gt, ws);
}

}  // namespace

#define TIMED(id, launch) do { if (prof) prof->begin(id, st); launch; if (prof) prof->end(st); } while (0)

int configure_fp32_gemm_kernels() {
  const bool ok = allow_smem((const void*)sgemm_tile<G_FWD, 7, 8, false>, Tile<G_FWD, 7, 8>::SMEM) == cudaSuccess && allow_smem((const void*)sgemm_fwd_rows, RW_SMEM) == cudaSuccess && allow_smem((const void*)sgemm_tile<G_DX, 7, 8, false>, Tile<G_DX, 7, 8>::SMEM) == cudaSuccess &&
                  allow_smem((const void*)sgemm_tile<G_FWD, 8, 4, false>, Tile<G_FWD, 8, 4>::SMEM) == cudaSuccess && allow_smem((const void*)sgemm_tile<G_DX, 8, 4, false>, Tile<G_DX, 8, 4>::SMEM) == cudaSuccess &&
                  allow_smem((const void*)sgemm_tile<G_DX, 4, 4, true>, Tile<G_DX, 4, 4>::SMEM) == cudaSuccess &&
                  allow_smem((const void*)sgemm_tile<G_DW, 8, 8, false>, Tile<G_DW, 8, 8>::SMEM) == cudaSuccess &&
                  allow_smem((const void*)sgemm_dx_skinny, DXS_SMEM) == cudaSuccess;
  return ok ? 0 : -1;
}

void launch_fc1_fwd_fp32(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  TIMED(K_FC1_FWD, (run_grouped<G_FWD>(a, wt, gt, ws, st)));
}
void launch_fc1_dx_fp32(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  TIMED(K_FC1_DX, (run_grouped<G_DX>(a, wt, gt, ws, st)));
}
void launch_fc1_dw_fp32(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  // 128 x 128 tiles at every number of workers: 9 / 11 / 25 / 43 / 519 us at 2 x 8, 4 x 8, 8 x 64, 16 x 64, 128 x 128;
  // 64 x 64 tiles 9 / 11 / 29 / 52 / 680
  TIMED(K_FC1_DW, (sgemm_tile<G_DW, 8, 8, false><<<dim3((FLAT + 127) / 128, HID / 128, a.W), 256, Tile<G_DW, 8, 8>::SMEM, st>>>(a, wt, gt, ws)));
}

}  // namespace psk
