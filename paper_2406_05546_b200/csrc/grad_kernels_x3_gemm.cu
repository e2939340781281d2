// The three products of the 512-unit dense layer on the FP32 path, on the fifth-generation tensor cores: FP32 operands as
// three BF16 pieces each (bf16x3.cuh), six of their nine products, FP32 accumulation.
//   forward          C[m][n] = sum_k p2[m][k] * W1[n][k]      (rows of one weight group; bias, ReLU, dropout)
//   input gradient   C[m][n] = sum_k dA1[m][k] * W1[k][n]     (rows of one weight group)
//   weight gradient  C[m][n] = sum_k dA1[k][m] * p2[k][n]     (k = the samples of one worker)
// The pieces are made by the kernels that produce the operands ([piece][row][column] BF16); W1's by prep_w1_x3.  Each
// operand is read as it lies: k contiguous (64-byte swizzle, blocks of 32 k) or its row index contiguous (128-byte
// swizzle, blocks of 64 rows), so that nothing is transposed.
//
// A CTA per SM walks over output tiles.  Per block of 32 k it issues ten instructions for the small products, then two for
// the leading ones; after four blocks the leading sums are handed to the epilogue warps, which add them to sums in
// registers while the small products of the next block run (forward: after two, for the sake of precision; 119.6 -> 121.2 us at 128 x 128).  With few tiles the blocks of k are dealt out over a cluster
// of CTAs (SPLIT) and the partial tiles are added through distributed shared memory in a fixed order.
//
// Every wait on an mbarrier is bounded, as in the other tensor-core kernels.
//
// Measured (B200; 26.3 GFLOP per product at 128 workers x 128 samples, six times that on the tensor cores: 95 us at the measured BF16
// rate; ~6 us of event overhead included; before: packed FP32 multiply-adds): forward 560 -> 121, input gradient 539 -> 144, weight
// gradient 515 -> 163 us (its 411 MiB of writes take 66 us at the copy rate); at 16 x 64: 72 -> 22, 58 -> 23, 42 -> 21; at 2 x 8: 17 -> 15,
// 11 -> 13, 9 -> 11.  Ticks, with the second convolution's products there as well: 8 x 8 75 -> 67 us, 8 x 16 125 -> 82, 8 x 64 246 -> 115, 32 x 64 649
// -> 250: multiply-adds are better at no size.
#include <cooperative_groups.h>
#include <cuda.h>

#include "bf16x3.cuh"
#include "device_common.cuh"
#include "kernels.h"
#include "tc5_common.cuh"

namespace psk {

namespace {

namespace cg = cooperative_groups;

enum { X_FWD = 0, X_DX = 1, X_DW = 2 };
constexpr int BM = 128, BK = 32;      // tile rows; k per stage
constexpr int EPI_WARPS = 8, THREADS = 64 + 32 * EPI_WARPS;
constexpr int OUT_PITCH = 36, OUT_WARP_BYTES = 32 * OUT_PITCH * 4;      // a 32 x 32 block on its way to whole rows

// BUFS: accumulators of either kind that are used in turn.
template <int OP_, int BN_, int BUFS_, int STAGES_, bool SPLIT_> struct Shape {
  static constexpr int OP = OP_, BN = BN_, BUFS = BUFS_, STAGES = STAGES_;
  static constexpr bool SPLIT = SPLIT_, A_MN = OP == X_DW, B_MN = OP != X_FWD;      // is the operand's row index contiguous?
  static constexpr int ACC = BN <= 128 ? 128 : 256;                               // tensor-memory columns of an accumulator
  static constexpr int B_COLS = B_MN ? (BN + 63) / 64 * 64 : BN;
  static constexpr int A_BYTES = PIECES * BM * BK * 2, B_BYTES = PIECES * B_COLS * BK * 2, STAGE = A_BYTES + B_BYTES;
  static constexpr int A_PIECE = A_MN ? 64 * BK * 2 : BM * BK * 2, B_PIECE = B_MN ? 64 * BK * 2 : BN * BK * 2;
  static constexpr int SMEM = 1024 /* alignment slack */ + STAGES * STAGE + 256 /* barriers */ + (OP == X_DW ? EPI_WARPS * OUT_WARP_BYTES : 0);
  static constexpr int COLS = BN / 2, PART_PITCH = BN + 4;      // columns of an epilogue thread; partial tile in shared memory
  static constexpr int CHUNK = OP == X_FWD ? 2 : 4;             // stages whose leading products share an accumulator
  static constexpr int TRIP = COLS > 112 ? 32 : 64;             // columns of a read of the accumulator (three warps share 16,384 registers)
  static_assert(2 * BUFS * ACC <= 512 && STAGE % 1024 == 0 && SMEM <= 227 * 1024 && COLS % 16 == 0, "tile shape");
  static_assert(!SPLIT || BM * PART_PITCH * 4 <= STAGES * STAGE, "the partial tile takes the operands' place");
};
using Fwd = Shape<X_FWD, 256, 1, 3, false>;
using FwdSplit = Shape<X_FWD, 128, 2, 4, true>;
using Dx = Shape<X_DX, 224, 1, 3, false>;
using DxSplit = Shape<X_DX, 128, 2, 4, true>;
using Dw = Shape<X_DW, 128, 2, 3, false>;

// Shared-memory descriptors, high half: stride byte offset, version, layout type.  k contiguous: rows 64 bytes apart, groups of
// eight rows 512 apart, 64-byte swizzle (type 4).  Row index contiguous: one k = 128 bytes (64 rows), groups of eight k 1,024
// bytes apart, 128-byte swizzle (type 2), the next 64 rows a block further (leading byte offset).
template <bool MN> __host__ __device__ constexpr uint32_t desc_hi() { return MN ? (1024 >> 4) | (1u << 14) | (2u << 29) : (512 >> 4) | (1u << 14) | (4u << 29); }
template <bool MN> __device__ __forceinline__ uint32_t desc_lo(uint32_t addr) {
  constexpr uint32_t BLOCK = PIECES * 64 * BK * 2;
  return ((addr & 0x3FFFF) >> 4) | ((MN ? BLOCK >> 4 : 1u) << 16);
}
template <bool MN> __host__ __device__ constexpr uint32_t k_step() { return MN ? 16 * 128 / 16 : 32 / 16; }      // sixteen k further, in 16-byte units
// fp32 accumulate, BF16 x BF16; bits 15 / 16: the operand's row index is contiguous
template <class S> __host__ __device__ constexpr uint32_t instr_desc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | (S::A_MN ? 1u << 15 : 0u) | (S::B_MN ? 1u << 16 : 0u) | ((uint32_t)(S::BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

struct Maps { CUtensorMap a, b; };
struct GemmArgs { int K, n_tiles_n, n_tiles; };
struct Tile { int grp, m0, m_end, n0, z; };

template <class S>
__device__ __forceinline__ bool decode(const GemmArgs& ga, const GroupTable& gt, int b, int t, Tile& c) {
  const int rest = t / ga.n_tiles_n;
  c.n0 = (t - rest * ga.n_tiles_n) * S::BN;
  c.grp = c.z = 0;
  if (S::OP == X_DW) {
    c.z = rest / (HID / BM);
    c.m0 = (rest % (HID / BM)) * BM;
    c.m_end = HID;
    return true;
  }
  return locate_group_tile<BM>(gt, b, rest, c.grp, c.m0, c.m_end);
}

template <class S>
__global__ void __launch_bounds__(THREADS, 1) gemm_x3(const __grid_constant__ Maps maps, GemmArgs ga, GradStepArgs a, WorkerTable wt, GroupTable gt, Workspace ws) {
  constexpr int STAGES = S::STAGES, BUFS = S::BUFS, COLS = S::COLS, CHUNK = S::CHUNK;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* tiles = smem_raw + (base - smem_u32(smem_raw));
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + STAGES * S::STAGE);      // [STAGES] copies -> MMA
  uint64_t* empty = full + STAGES;           // [STAGES] MMA -> copies
  uint64_t* lead_full = empty + STAGES;      // [BUFS] MMA -> epilogue; a tile's last one covers its small products as well
  uint64_t* lead_empty = lead_full + BUFS;   // [BUFS] epilogue -> MMA
  uint64_t* small_empty = lead_empty + BUFS; // [BUFS] epilogue -> MMA
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(small_empty + BUFS);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
  const int n_k = (ga.K + BK - 1) / BK;
  int kb0 = 0, kb1 = n_k;                    // this CTA's blocks of k
  if (S::SPLIT) {
    kb0 = n_k * (int)blockIdx.z / (int)gridDim.z;
    kb1 = n_k * ((int)blockIdx.z + 1) / (int)gridDim.z;
  }
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int i = 0; i < BUFS; ++i) { mbar_init(&lead_full[i], 1); mbar_init(&lead_empty[i], EPI_WARPS); mbar_init(&small_empty[i], EPI_WARPS); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(*tmem_slot);
  pdl_enter();

  if (warp == 0) {
    if (lane == 0) {
      int s = 0;
      uint32_t use = 0;                      // how often the stages have been gone round
      bool ok = true;
      for (int t = blockIdx.x; t < ga.n_tiles && ok; t += gridDim.x) {
        Tile c;
        if (!decode<S>(ga, gt, a.b, t, c)) continue;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (use > 0 && !mbar_wait(&empty[s], (use - 1) & 1)) { *abort_flag = 1; ok = false; break; }
          if (*abort_flag) { ok = false; break; }
          uint8_t* A = tiles + s * S::STAGE;
          uint8_t* B = A + S::A_BYTES;
          mbar_expect_tx(&full[s], S::STAGE);
          if (S::A_MN) {
            for (int i = 0; i < BM / 64; ++i) tma_load_4d(A + i * PIECES * S::A_PIECE, &maps.a, &full[s], c.m0 + 64 * i, kb * BK, c.z, 0);
          } else {
            tma_load_3d(A, &maps.a, &full[s], kb * BK, c.m0, 0);
          }
          if (S::OP == X_FWD) {
            tma_load_3d(B, &maps.b, &full[s], kb * BK, c.n0, PIECES * c.grp);
          } else {
            for (int i = 0; i < S::B_COLS / 64; ++i) {
              if (S::OP == X_DX) tma_load_3d(B + i * PIECES * S::B_PIECE, &maps.b, &full[s], c.n0 + 64 * i, kb * BK, PIECES * c.grp);
              else tma_load_4d(B + i * PIECES * S::B_PIECE, &maps.b, &full[s], c.n0 + 64 * i, kb * BK, c.z, 0);
            }
          }
          if (++s == STAGES) { s = 0; ++use; }
        }
      }
    }
  } else if (warp == 1) {
    constexpr uint32_t idesc = instr_desc<S>(), ha = desc_hi<S::A_MN>(), hb = desc_hi<S::B_MN>();
    constexpr uint32_t pa = S::A_PIECE / 16, pb = S::B_PIECE / 16, ka = k_step<S::A_MN>(), kbs = k_step<S::B_MN>();
    int s = 0, lead = 0, tile_i = 0;       // stage; chunks of leading products, and tiles, so far
    uint32_t parity = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ga.n_tiles && ok; t += gridDim.x) {
      Tile c;
      if (!decode<S>(ga, gt, a.b, t, c)) continue;
      const uint32_t d_small = tmem + (BUFS + tile_i % BUFS) * S::ACC;
      if (tile_i >= BUFS && !warp_wait(&small_empty[tile_i % BUFS], ((tile_i / BUFS) - 1) & 1, abort_flag)) { *abort_flag = 1; break; }
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!warp_wait(&full[s], parity, abort_flag)) { *abort_flag = 1; ok = false; break; }
        tc_fence_after();
        const uint32_t a_lo = desc_lo<S::A_MN>(base + s * S::STAGE), b_lo = desc_lo<S::B_MN>(base + s * S::STAGE + S::A_BYTES);
        const bool first = (kb - kb0) % CHUNK == 0, last = (kb - kb0) % CHUNK == CHUNK - 1 || kb + 1 == kb1;
#pragma unroll
        for (int k = 0; k < BK / 16; ++k)
#pragma unroll
          for (int i = 0; i < 5; ++i) {    // l h, m m, h l, m h, h m
            const int i_a = i == 0 ? 2 : (i == 1 || i == 3 ? 1 : 0), i_b = i == 2 ? 2 : (i == 1 || i == 4 ? 1 : 0);
            umma_f16(d_small, a_lo + i_a * pa + k * ka, ha, b_lo + i_b * pb + k * kbs, hb, idesc, (k | i) ? 1u : (kb > kb0 ? 1u : 0u));
          }
        if (first && lead >= BUFS) {
          if (!warp_wait(&lead_empty[lead % BUFS], ((lead / BUFS) - 1) & 1, abort_flag)) { *abort_flag = 1; ok = false; break; }
          tc_fence_after();
        }
        const uint32_t d_lead = tmem + (lead % BUFS) * S::ACC;
#pragma unroll
        for (int k = 0; k < BK / 16; ++k) umma_f16(d_lead, a_lo + k * ka, ha, b_lo + k * kbs, hb, idesc, k ? 1u : (first ? 0u : 1u));
        umma_commit(&empty[s]);
        if (last) { umma_commit(&lead_full[lead % BUFS]); ++lead; }
        if (++s == STAGES) { s = 0; parity ^= 1; }
      }
      ++tile_i;
    }
  } else {
    const int quarter = warp & 3, half = (warp - 2) >> 2, col0 = half * COLS;
    const uint32_t t_lane = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col0;
    int lead = 0, tile_i = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ga.n_tiles && ok; t += gridDim.x) {
      Tile c;
      if (!decode<S>(ga, gt, a.b, t, c)) continue;
      float sum[COLS];
#pragma unroll
      for (int j = 0; j < COLS; ++j) sum[j] = 0.f;
      for (int kb = kb0; kb < kb1; kb += CHUNK) {
        const int lb = lead % BUFS, sb = tile_i % BUFS;
        if (!warp_wait(&lead_full[lb], (lead / BUFS) & 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        // as many columns per round trip to tensor memory as there are registers for: input gradient 145.9 -> 143.8 us at 128 x 128, the others
        // as with sixteen
        auto drain = [&](uint32_t at, auto add) {
#pragma unroll
          for (int j0 = 0; j0 < COLS; j0 += S::TRIP) {
            uint32_t r[S::TRIP / 16][16];
#pragma unroll
            for (int i = 0; i < S::TRIP / 16; ++i)
              if (j0 + 16 * i < COLS) tmem_ld16(at + j0 + 16 * i, r[i]);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < S::TRIP / 16; ++i)
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (j0 + 16 * i < COLS) sum[j0 + 16 * i + j] = add(sum[j0 + 16 * i + j], __uint_as_float(r[i][j]));
          }
        };
        drain(t_lane + lb * S::ACC, [](float a, float v) { return a + v; });
        const bool last = kb + CHUNK >= kb1;
        if (last) drain(t_lane + (BUFS + sb) * S::ACC, [](float a, float v) { return join3(a, v); });
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&lead_empty[lb]);
          if (last) mbar_arrive(&small_empty[sb]);
        }
        ++lead;
      }
      ++tile_i;
      if (!ok) {
        if (lane == 0) *abort_flag = 1;
        break;
      }
      const int m = c.m0 + quarter * 32 + lane;
      if (S::SPLIT) {                        // all copies have landed and been read: the partial tile takes their place
        float4* d = reinterpret_cast<float4*>(reinterpret_cast<float*>(tiles) + (quarter * 32 + lane) * S::PART_PITCH + col0);
#pragma unroll
        for (int j = 0; j < COLS / 4; ++j) d[j] = make_float4(sum[4 * j], sum[4 * j + 1], sum[4 * j + 2], sum[4 * j + 3]);
      } else if (S::OP == X_DW) {
        // through a padded block of shared memory, so that a store writes four whole 128-byte row segments
        float* stage = reinterpret_cast<float*>(tiles + STAGES * S::STAGE + 256) + (warp - 2) * (OUT_WARP_BYTES / 4);
        float* C = wt.grad[c.z] + OFF_F1W;
#pragma unroll
        for (int j0 = 0; j0 < COLS; j0 += 32) {
          const int n = c.n0 + col0 + j0;
          if (n < FLAT) {                    // 1,568 = 49 x 32
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 8; ++q)
              *reinterpret_cast<float4*>(stage + lane * OUT_PITCH + 4 * q) = make_float4(sum[j0 + 4 * q], sum[j0 + 4 * q + 1], sum[j0 + 4 * q + 2], sum[j0 + 4 * q + 3]);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int rr = i * 4 + (lane >> 3), cc = (lane & 7) * 4;
              *reinterpret_cast<float4*>(C + (int64_t)(c.m0 + quarter * 32 + rr) * FLAT + n + cc) = *reinterpret_cast<const float4*>(stage + rr * OUT_PITCH + cc);
            }
          }
        }
      } else if (m < c.m_end) {
        // a lane's row straight from its registers: a tile's products take ten times as long as these stores
#pragma unroll
        for (int j = 0; j < COLS / 4; ++j) {
          const float4 v = make_float4(sum[4 * j], sum[4 * j + 1], sum[4 * j + 2], sum[4 * j + 3]);
          const int n = c.n0 + col0 + 4 * j;
          if (S::OP == X_FWD) *reinterpret_cast<float4*>(ws.d + (int64_t)m * HID + n) = fc1_activation(v, m, n, gt.theta[c.grp], a, wt);
          else *reinterpret_cast<float4*>(ws.dp2 + (int64_t)m * FLAT + n) = v;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  if constexpr (S::SPLIT) {
    Tile c;
    if (decode<S>(ga, gt, a.b, blockIdx.x, c)) {             // the same for all CTAs of a cluster
      cg::cluster_group cl = cg::this_cluster();
      cl.sync();
      const int ranks = gridDim.z, rank = blockIdx.z, rows = min(BM, c.m_end - c.m0), cols = min(S::BN, (S::OP == X_FWD ? HID : FLAT) - c.n0);
      float* part = reinterpret_cast<float*>(tiles);
      for (int e = rank * THREADS + tid; e < rows * (S::BN / 4); e += ranks * THREADS) {
        const int r = e / (S::BN / 4), q = e - r * (S::BN / 4), m = c.m0 + r, n = c.n0 + 4 * q;
        if (4 * q >= cols) continue;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = 0; k < ranks; ++k) {
          const float4 u = *reinterpret_cast<const float4*>(cl.map_shared_rank(part, k) + r * S::PART_PITCH + 4 * q);
          v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
        }
        if (S::OP == X_FWD) *reinterpret_cast<float4*>(ws.d + (int64_t)m * HID + n) = fc1_activation(v, m, n, gt.theta[c.grp], a, wt);
        else *reinterpret_cast<float4*>(ws.dp2 + (int64_t)m * FLAT + n) = v;
      }
      cl.sync();                             // a CTA's shared memory outlives its readers
    }
  }
  if (tid == 0 && *abort_flag) {
    atomicOr(ws.status, STATUS_WAIT_TIMEOUT);
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);      // let copies already issued land before the CTA ends
  }
}

// The pieces of every weight group's W1.
__global__ void __launch_bounds__(256) prep_w1_x3(GroupTable gt, uint16_t* __restrict__ w1x) {
  const int i = (blockIdx.x * 256 + threadIdx.x) * 8;
  if (i < W1_ELEMS) split_w1(gt.theta[blockIdx.y], w1x, blockIdx.y, i);
}

// BF16 tensor of `rank` dimensions (dims[0] contiguous; pitch[i] elements between neighbours of dimension i + 1).
bool make_map(CUtensorMap* m, const uint16_t* base, int rank, const uint64_t* dims, const uint64_t* pitch, const uint32_t* box, bool wide) {
  uint64_t bytes[4];
  for (int i = 0; i + 1 < rank; ++i) bytes[i] = 2 * pitch[i];
  return encode_tensor_map_bf16(m, base, rank, dims, bytes, box, wide ? 128 : 64);
}
// [pieces][rows][cols], k = columns
bool map_k(CUtensorMap* m, const uint16_t* base, uint64_t cols, uint64_t rows, uint64_t planes, uint32_t box_rows) {
  const uint64_t dims[3] = {cols, rows, planes}, pitch[2] = {cols, cols * rows};
  const uint32_t box[3] = {BK, box_rows, PIECES};
  return make_map(m, base, 3, dims, pitch, box, false);
}
// [pieces][rows][cols], k = rows
bool map_mn(CUtensorMap* m, const uint16_t* base, uint64_t cols, uint64_t rows, uint64_t planes) {
  const uint64_t dims[3] = {cols, rows, planes}, pitch[2] = {cols, cols * rows};
  const uint32_t box[3] = {64, BK, PIECES};
  return make_map(m, base, 3, dims, pitch, box, true);
}
// [pieces][W][b][cols], k = the samples of a worker (those beyond b arrive as zeros)
bool map_worker(CUtensorMap* m, const uint16_t* base, uint64_t cols, uint64_t b, uint64_t W) {
  const uint64_t dims[4] = {cols, b, W, PIECES}, pitch[3] = {cols, cols * b, cols * b * W};
  const uint32_t box[4] = {64, BK, 1, PIECES};
  return make_map(m, base, 4, dims, pitch, box, true);
}

template <class S>
void run(const Maps& maps, const GemmArgs& ga, int split, bool overlap, const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st) {
  if constexpr (S::SPLIT) {
    launch_cluster(gemm_x3<S>, dim3(ga.n_tiles, 1, split), THREADS, S::SMEM, split, st, maps, ga, a, wt, gt, ws);
  } else {
    launch_pdl_if(overlap, gemm_x3<S>, dim3(ga.n_tiles < g_sm_count ? ga.n_tiles : g_sm_count), THREADS, S::SMEM, st, maps, ga, a, wt, gt, ws);
  }
}

// CTAs of a cluster that share a tile's blocks of k: as many as the chip has room for.  Tiles 128 columns wide while one round
// of them fits on the chip (their two accumulators of either kind hide a tile's read-out); beyond that wide ones, which read a
// third less from L2 per product.
int split_of(int tiles, int most) {
  int split = 1;
  while (split < most && tiles * split * 2 <= g_sm_count) split *= 2;
  return split;
}

}  // namespace

#define TIMED(id, launch) do { if (prof) prof->begin(id, st); launch; if (prof) prof->end(st); } while (0)

int configure_x3_gemm_kernels() {
  const bool ok = allow_smem((const void*)gemm_x3<Fwd>, Fwd::SMEM) == cudaSuccess && allow_smem((const void*)gemm_x3<FwdSplit>, FwdSplit::SMEM) == cudaSuccess &&
                  allow_smem((const void*)gemm_x3<Dx>, Dx::SMEM) == cudaSuccess && allow_smem((const void*)gemm_x3<DxSplit>, DxSplit::SMEM) == cudaSuccess &&
                  allow_smem((const void*)gemm_x3<Dw>, Dw::SMEM) == cudaSuccess;
  return ok ? 0 : -1;
}

void launch_prep_w1_x3(const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  TIMED(K_PREP_W1, (prep_w1_x3<<<dim3((W1_ELEMS / 8 + 255) / 256, gt.n_groups), 256, 0, st>>>(gt, ws.w1x)));
}

int launch_fc1_fwd_x3(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof, bool after_join) {
  Maps maps;
  const uint64_t rows = (uint64_t)a.W * a.b;
  const int mt = group_tiles(gt, a.b, BM), tiles = mt * (HID / FwdSplit::BN);
  const bool few = tiles <= g_sm_count;
  if (!map_k(&maps.a, ws.p2x, FLAT, rows, PIECES, BM) || !map_k(&maps.b, ws.w1x, FLAT, HID, (uint64_t)PIECES * gt.n_groups, few ? FwdSplit::BN : Fwd::BN)) return -1;
  if (few) TIMED(K_FC1_FWD, (run<FwdSplit>(maps, GemmArgs{FLAT, HID / FwdSplit::BN, tiles}, split_of(tiles, 8), true, a, wt, gt, ws, st)));
  else TIMED(K_FC1_FWD, (run<Fwd>(maps, GemmArgs{FLAT, HID / Fwd::BN, mt * (HID / Fwd::BN)}, 1, !after_join, a, wt, gt, ws, st)));
  return 1;
}

int launch_fc1_dx_x3(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  Maps maps;
  const uint64_t rows = (uint64_t)a.W * a.b;
  constexpr int NARROW = (FLAT + DxSplit::BN - 1) / DxSplit::BN;
  const int mt = group_tiles(gt, a.b, BM), tiles = mt * NARROW;
  if (!map_k(&maps.a, ws.da1x, HID, rows, PIECES, BM) || !map_mn(&maps.b, ws.w1x, FLAT, HID, (uint64_t)PIECES * gt.n_groups)) return -1;
  if (tiles <= g_sm_count) TIMED(K_FC1_DX, (run<DxSplit>(maps, GemmArgs{HID, NARROW, tiles}, split_of(tiles, 4), true, a, wt, gt, ws, st)));
  else TIMED(K_FC1_DX, (run<Dx>(maps, GemmArgs{HID, FLAT / Dx::BN, mt * (FLAT / Dx::BN)}, 1, true, a, wt, gt, ws, st)));
  return 1;
}

int launch_fc1_dw_x3(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  Maps maps;
  constexpr int NT = (FLAT + Dw::BN - 1) / Dw::BN;
  if (!map_worker(&maps.a, ws.da1x, HID, a.b, a.W) || !map_worker(&maps.b, ws.p2x, FLAT, a.b, a.W)) return -1;
  TIMED(K_FC1_DW, (run<Dw>(maps, GemmArgs{a.b, NT, NT * (HID / BM) * a.W}, 1, false, a, wt, gt, ws, st)));
  return 1;
}

}  // namespace psk
