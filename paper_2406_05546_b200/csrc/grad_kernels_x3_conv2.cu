// Second convolution (16 -> 32 channels, 3x3, pad 1, 14x14 maps) of the FP32 path on the fifth-generation tensor cores: forward
// with ReLU and 2x2 max pooling, the gradient with respect to its input, and its filter / bias gradient.  Operands are
// three BF16 pieces of every FP32 value (bf16x3.cuh), of whose nine products at least the six largest are taken, FP32
// accumulation in tensor memory, the leading products in accumulators of their own.
//
// No operand is laid out twice.  The first convolution writes its pooled output as
//   p1x[image row Y of the 16x16 bordered map][piece][octet of channels][slot][8 channels],  slot(X) = (X & 1) * 8 + X / 2,
// 16 bytes a slot, 256 a run, 1,536 an image row, 24,576 a sample, and all three shapes in which the products need it are
// strides of that:
//   - forward (k = channel): rows are pooled positions, eight consecutive slots (a stride of two columns) by every second image
//     row; the sixteen shifts of the 4x4 patch under a pooling window are start addresses.  A second sample follows the first
//     at the pitch of its rows, so that two make the 128 rows of a tile.
//   - filter gradient (k = position): the operand's row index is contiguous (eight channels of a slot), so positions need no
//     transposing; (filter row, piece, octet) are eighteen groups of eight columns 256 bytes apart, one stride.
// Sixteen k of a filter-gradient step are one column parity of two image rows: eight consecutive slots for every filter column.
//
// Products that share an operand piece share an instruction where their columns can be neighbours (input and filter gradient).
//
// Zero padding and window losers are multiplied like other values: where an infinite activation meets a zero gradient, the taps
// concerned are NaN, as in any FP32 sum over the map.  What is no position of the map is no part of a sum: the filter gradient's columns of
// padding never meet an infinity (see there).
//
// Measured (B200; 29.6 GFLOP per product at 128 workers x 128 samples, six times that on the tensor cores: 112 us at the measured
// BF16 rate; ~6 us of event overhead included; before: packed FP32 multiply-adds at two thirds of their pipe's rate): forward 696 ->
// 210, input gradient 636 -> 176, filter gradient 651 -> 271 us; at 16 x 64: 56 -> 25, 57 -> 21, 56 -> 31; at 2 x 8: 12 -> 13, 15 -> 11,
// 15 -> 14.  Forward and input gradient are bound by the instructions' own time; the filter gradient takes 1.5 times as many products as
// it needs, rounded up to 128 rows.  Relative error against float64, median over workers, 128 x 128: conv2.w 1.7e-7 -> 0.8e-7, conv1.w
// 1.7e-7 -> 1.0e-7; 2 x 8: 2.9e-7 -> 1.2e-7, 3.3e-7 -> 1.5e-7.
//
// Each kernel's stages (copies, staging, MMA issue, read-out) run in different warps and overlap through mbarriers; every wait
// is bounded.
#include "bf16x3.cuh"
#include "device_common.cuh"
#include "kernels.h"
#include "tc5_common.cuh"

namespace psk {

namespace {

constexpr int TMEM_ALL = 512;

// fp32 accumulate, BF16 x BF16, M = 128; mn: both operands' row index is contiguous
__host__ __device__ constexpr uint32_t idesc_x3(int n, bool mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? 3u << 15 : 0u) | ((uint32_t)(n >> 3) << 17) | (8u << 24);
}

__device__ __forceinline__ void tmem_alloc_all(uint32_t* slot) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(TMEM_ALL) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free_all(uint32_t tmem) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_ALL) : "memory");
}
__device__ __forceinline__ void report_abort(uint32_t* status) {
  atomicOr(status, STATUS_WAIT_TIMEOUT);
  for (int k = 0; k < 1000; ++k) __nanosleep(1000);   // let copies already issued land before the CTA ends
}

// ------------------------------------------------------------------------------------------------
// Forward.  Tile = two samples = 128 rows: row 8 g + i is pooled position (py = g mod 8, px = i) of sample g / 8 (py = 7 and
// px = 7 are padding rows whose results are dropped).  The four window elements c = 2 jy + jx go to four ranges of 32
// accumulator columns, so that a thread holds whole windows.  One MMA per input SHIFT: window element (jy, jx) and tap (ky, kx)
// read the input shifted by (jy + ky, jx + kx); the filters of the pairs that add up to a shift are stacked in column order.
// The ranges are ordered (0,0) (0,1) (1,1) (1,0): a shift's window elements are neighbours but for two shifts, which take
// two MMAs: 18 per product, 108 a tile.  The leading products of shifts with an even and with an odd sum of coordinates have an accumulator each
// (a sum of nine taps in one loses more to truncation than one of five and one of four; 200 -> 210 us at 128 x 128), so that a tile takes three of the four that there is room
// for, in turn: its small products, five sixths of its time, run while the tile before is read out.
// Warps: 0 = MMA issue and tensor memory, 1 = copies, 2..9 = epilogue.
// ------------------------------------------------------------------------------------------------
constexpr int F_THREADS = 320, F_STAGES = 2, F_OPS = 18;
constexpr int F_STAGE_BYTES = 2 * P1X_BYTES + 2 * P1X_ROW + 256;       // the padding rows' overrun
constexpr int F_W_PIECE = 2 * BANK3_FWD_ROWS * 16;                      // [octet][row][8 channels]
constexpr int F_BARS = 2 * F_STAGES + 1 + 1 + 1;
constexpr int F_SMEM = F_STAGES * F_STAGE_BYTES + BANK3_FWD_BYTES + 32 * 4 + F_BARS * 8 + 16;
static_assert(F_SMEM <= 227 * 1024 && F_STAGE_BYTES % 128 == 0, "shared memory");

struct FoldTable {
  int32_t a_off[F_OPS], d_col[F_OPS], b_row[F_OPS];      // shifted start (16-byte units), first column, first row of the stacked filters
  uint32_t idesc[F_OPS];
};
struct FoldTables {
  FoldTable fold;
  Bank3Taps taps;
  FoldTables() {
    constexpr int RANGE_OF[4] = {0, 1, 3, 2};            // window element -> column range
    int n_ops = 0, row = 0;
    auto add = [&](int sy, int sx, int first, int n) {
      fold.a_off[n_ops] = sy * (P1X_ROW / 16) + (sx & 1) * 8 + (sx >> 1);
      fold.d_col[n_ops] = 32 * first;
      fold.b_row[n_ops] = row;
      fold.idesc[n_ops] = idesc_x3(32 * n, false);
      for (int r = first; r < first + n; ++r, row += 32) {
        const int c = RANGE_OF[r];                       // its own inverse
        taps.tap[row / 32] = (uint8_t)((sy - (c >> 1)) * 3 + (sx - (c & 1)));
      }
      ++n_ops;
    };
    for (int pass = 0; pass < 4; ++pass)                 // either half begins with an op that covers all columns: it starts the sums
      for (int sy = 0; sy < 4; ++sy)
        for (int sx = 0; sx < 4; ++sx) {
          const bool starts = sy == 1 && (sx == 1 || sx == 2);
          if (((sy + sx) & 1) != pass >> 1 || starts != ((pass & 1) == 0)) continue;
          bool used[4] = {false, false, false, false};
          for (int jy = 0; jy < 2; ++jy)
            for (int jx = 0; jx < 2; ++jx)
              if (sy >= jy && sy - jy < 3 && sx >= jx && sx - jx < 3) used[RANGE_OF[2 * jy + jx]] = true;
          for (int r = 0; r < 4;) {
            int n = 0;
            while (r + n < 4 && used[r + n]) ++n;
            if (n) add(sy, sx, r, n);
            r += n ? n : 1;
          }
        }
    // n_ops == F_OPS and row == BANK3_FWD_ROWS by construction
  }
};
const FoldTables& fold_tables() {
  static const FoldTables t;
  return t;
}

__global__ void __launch_bounds__(F_THREADS, 1) conv2_fwd_x3(GradStepArgs a, GroupTable gt, Workspace ws, int range_len, const __grid_constant__ FoldTable fold) {
  extern __shared__ __align__(128) uint8_t smem[];
  uint8_t* Wk = smem + F_STAGES * F_STAGE_BYTES;
  float* bias = reinterpret_cast<float*>(Wk + BANK3_FWD_BYTES);
  uint64_t* a_full = reinterpret_cast<uint64_t*>(bias + 32);      // [F_STAGES] copies -> MMA
  uint64_t* a_empty = a_full + F_STAGES;                          // [F_STAGES] MMA -> copies
  uint64_t* acc_full = a_empty + F_STAGES;                        // MMA -> epilogue
  uint64_t* acc_empty = acc_full + 1;                             // epilogue -> MMA
  uint64_t* w_full = acc_empty + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w_full + 1);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
  // a CTA walks over a contiguous range of rows (worker-major samples) that share one weight snapshot
  int grp, r_begin, r_end;
  if (!locate_row_range(gt, a.b, range_len, blockIdx.x, grp, r_begin, r_end)) return;
  const int n_tiles = (r_end - r_begin + 1) / 2;

  // bytes never written by a copy (the overrun of the padding rows, a missing second sample) only feed rows that are dropped
  if (tid == 0) {
    for (int i = 0; i < F_STAGES; ++i) { mbar_init(&a_full[i], 1); mbar_init(&a_empty[i], 1); }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 8);
    mbar_init(w_full, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc_all(tmem_slot);
  pdl_enter();
  if (tid < 32) bias[tid] = gt.theta[grp][OFF_C2B + tid];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(*tmem_slot);

  if (warp == 0) {
    const uint32_t w_lo = plain_desc_lo(smem_u32(Wk), BANK3_FWD_ROWS * 16);
    const uint32_t a_lo0 = plain_desc_lo(smem_u32(smem), 256);
    bool ok = warp_wait(w_full, 0, abort_flag);
    if (!ok) *abort_flag = 1;
    for (int t = 0; ok && t < n_tiles; ++t) {
      const int buf = t & 1;
      if (!warp_wait(&a_full[buf], (t >> 1) & 1, abort_flag)) { *abort_flag = 1; break; }
      tc_fence_after();
      const uint32_t a_lo = a_lo0 + buf * (F_STAGE_BYTES / 16);
      // l h, m m, h l, m h, h m into accumulator 3 t, which the tile before the last has left, then h h into 3 t + 1 and 3 t + 2, once the last
      // tile has been read out
#pragma unroll 1
      for (int i = 0; i < 6; ++i) {
        if (i == 5 && t > 0) {
          ok = warp_wait(acc_empty, (t - 1) & 1, abort_flag);
          if (!ok) { *abort_flag = 1; break; }
          tc_fence_after();
        }
        const int i_a = (0x001012 >> (4 * i)) & 15, i_b = (0x010210 >> (4 * i)) & 15;
        const uint32_t ai = a_lo + i_a * (512 / 16), bi = w_lo + i_b * (F_W_PIECE / 16);
        const uint32_t d0 = tmem + ((3 * t + (i < 5 ? 0 : 1)) & 3) * 128, d1 = tmem + ((3 * t + (i < 5 ? 0 : 2)) & 3) * 128;
        const uint32_t start0 = i == 0 || i == 5 ? 0u : 1u, start1 = i == 5 ? 0u : 1u;
#pragma unroll
        for (int op = 0; op < F_OPS; ++op)
          umma_f16((op < F_OPS / 2 ? d0 : d1) + fold.d_col[op], ai + fold.a_off[op], plain_desc_hi(2 * P1X_ROW), bi + fold.b_row[op], plain_desc_hi(128),
                   fold.idesc[op], op == 0 ? start0 : (op == F_OPS / 2 ? start1 : 1u));
      }
      if (!ok) break;
      umma_commit(&a_empty[buf]);
      umma_commit(acc_full);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      mbar_expect_tx(w_full, BANK3_FWD_BYTES);
      bulk_load(Wk, ws.bank2 + (int64_t)grp * BANK3_BYTES, BANK3_FWD_BYTES, w_full);
      for (int t = 0; t < n_tiles; ++t) {
        const int buf = t & 1;
        if ((t >= F_STAGES && !mbar_wait(&a_empty[buf], ((t >> 1) - 1) & 1)) || *abort_flag) { *abort_flag = 1; break; }
        const uint32_t bytes = (uint32_t)min(2, r_end - (r_begin + 2 * t)) * P1X_BYTES;
        mbar_expect_tx(&a_full[buf], bytes);
        bulk_load(smem + buf * F_STAGE_BYTES, ws.p1x + (int64_t)(r_begin + 2 * t) * P1X_BYTES, bytes, &a_full[buf]);
      }
    }
  } else {
    const int quarter = warp & 3, ch = (warp - 2) >> 2;
    const int r = quarter * 32 + lane, g = r >> 3, px = r & 7, sp = g >> 3, py = g & 7, pp = py * 7 + px;
    const int64_t rows = (int64_t)a.W * a.b;
    for (int t = 0; t < n_tiles; ++t) {
      if (!warp_wait(acc_full, t & 1, abort_flag)) { *abort_flag = 1; break; }
      tc_fence_after();
      const int64_t row = r_begin + 2 * t + sp;
      float v[4][16];                        // [column range][channel]
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t small[16], even[16], odd[16];
        const uint32_t at = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(j * 32 + ch * 16);
        tmem_ld16(at + (3 * t & 3) * 128, small);
        tmem_ld16(at + ((3 * t + 1) & 3) * 128, even);
        tmem_ld16(at + ((3 * t + 2) & 3) * 128, odd);
        tmem_ld_wait();
#pragma unroll
        for (int o = 0; o < 16; ++o) v[j][o] = join3(__uint_as_float(even[o]) + __uint_as_float(odd[o]), __uint_as_float(small[o]));
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
      if (py < 7 && px < 7 && row < r_end) {
        uint32_t codes[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int o = 0; o < 16; o += 2) {
          float best[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {      // ReLU, then the first window element that reaches the maximum
            const float bv = bias[ch * 16 + o + h];
            const float e[4] = {v[0][o + h] + bv, v[1][o + h] + bv, v[3][o + h] + bv, v[2][o + h] + bv};
            best[h] = fmaxf(e[0], 0.f);
            uint32_t bi = 0;
#pragma unroll
            for (int j = 1; j < 4; ++j) {
              const float x = fmaxf(e[j], 0.f);
              if (x > best[h]) { best[h] = x; bi = j; }
            }
            codes[o >> 2] |= (best[h] > 0.f ? bi : 4u) << (8 * ((o + h) & 3));
          }
          const Bf16x3 s = split3(best[0], best[1]);      // its readers are the dense layer's products
          uint16_t* d = ws.p2x + row * FLAT + (ch * 16 + o) * 49 + pp;
#pragma unroll
          for (int p = 0; p < PIECES; ++p) {
            d[p * rows * FLAT] = (uint16_t)s.p[p];
            d[p * rows * FLAT + 49] = (uint16_t)(s.p[p] >> 16);
          }
        }
        // decisions as [channel quad][position][4 channels] bytes
        uint32_t* c2 = reinterpret_cast<uint32_t*>(ws.code2 + row * FLAT);
#pragma unroll
        for (int q = 0; q < 4; ++q) c2[(ch * 4 + q) * 49 + pp] = codes[q];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) { tc_fence_after(); tmem_free_all(tmem); }
  if (tid == 0 && *abort_flag) report_abort(ws.status);
}

// Staging of g2, the gradient at the convolution's output: the eight pooled gradients of (octet of channels, pooled position) in
// pieces, and for each element of its pooling window the pieces masked by "this element won" (store(j, piece, 16 bytes)).
// raw: a sample's pooled gradients [channel][49] FP32, then its decisions [channel quad][49][4] bytes.
constexpr int RAW_BYTES = FLAT * 4 + FLAT;
template <typename Store>
__device__ __forceinline__ void place_g2(const uint8_t* raw, int o8, int p, Store store) {
  const float* g = reinterpret_cast<const float*>(raw) + o8 * 8 * 49 + p;
  const uint32_t* code = reinterpret_cast<const uint32_t*>(raw + FLAT * 4) + 2 * o8 * 49 + p;
  const uint32_t ca = code[0], cb = code[49];
  Bf16x3 s[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) s[i] = split3(g[2 * i * 49], g[(2 * i + 1) * 49]);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    // a decision byte is 0..4, so (byte xor j) + 0x7F has its top bit set exactly when the byte differs from j; byte
    // permutes that replicate the top bit turn the flags into pairs of half-word masks
    const uint32_t ea = ~((ca ^ (0x01010101u * j)) + 0x7F7F7F7Fu) & 0x80808080u, eb = ~((cb ^ (0x01010101u * j)) + 0x7F7F7F7Fu) & 0x80808080u;
    const uint32_t m0 = prmt(ea, 0u, 0x9988u), m1 = prmt(ea, 0u, 0xBBAAu), m2 = prmt(eb, 0u, 0x9988u), m3 = prmt(eb, 0u, 0xBBAAu);
#pragma unroll
    for (int q = 0; q < PIECES; ++q) store(j, q, make_uint4(s[0].p[q] & m0, s[1].p[q] & m1, s[2].p[q] & m2, s[3].p[q] & m3));
  }
}

// ------------------------------------------------------------------------------------------------
// Gradient with respect to the convolution's input.  Tile = one sample = two 128-row blocks of the 16-wide position grid
// (row = y*16 + x; y, x >= 14 are padding rows).  g2 lies in zero-bordered planes of eight channels, [piece][octet], one position a
// 16-byte row; filter row ky reads them shifted by (2 - ky) rows of positions.  The three taps of a filter row sit side by side in
// 48 accumulator columns, and the pieces of the filters next to one another: g's h takes the filters' h, m, l (N = 144), its m h
// and m (N = 96, one range to the right), its l h (N = 48, two to the right): the first range holds the leading products, the
// other two the small ones.  36 MMAs a sample instead of 72; an MMA of M = 128, K = 16 takes 40 clk or N / 2, whichever is more.
// The epilogue adds a filter row's columns with lane shifts; with one group of four warps for both blocks it takes 178 instead of 176 us at
// 128 x 128.
// Warps: 0 = MMA, 1..8 = staging (two groups on alternate samples), 9..16 = epilogue (a group of four for either block of rows), 17 = copies.
// ------------------------------------------------------------------------------------------------
constexpr int X_THREADS = 576, X_RAW_SLOTS = 8, X_ACC = 3;
constexpr int X_PLANE_BYTES = (256 + 51) * 16;             // 34 rows of tap overrun; a pitch of 3 rows mod 8 spreads the staging stores over the banks
constexpr int X_PIECE_BYTES = 4 * X_PLANE_BYTES, X_BUF_BYTES = PIECES * X_PIECE_BYTES;
constexpr int X_BARS = 2 * 2 + 2 * X_ACC + 2 * X_RAW_SLOTS + 1;
constexpr int X_SMEM = 2 * X_BUF_BYTES + BANK3_DX_BYTES + X_RAW_SLOTS * RAW_BYTES + X_BARS * 8 + 16;
static_assert(X_SMEM <= 227 * 1024 && (2 * X_BUF_BYTES) % 16 == 0 && RAW_BYTES % 16 == 0, "shared memory");

__global__ void __launch_bounds__(X_THREADS, 1) conv2_dx_x3(GradStepArgs a, GroupTable gt, Workspace ws, int range_len) {
  extern __shared__ __align__(128) uint8_t smem[];
  uint8_t* Wk = smem + 2 * X_BUF_BYTES;
  uint8_t* raw = Wk + BANK3_DX_BYTES;
  uint64_t* a_full = reinterpret_cast<uint64_t*>(raw + X_RAW_SLOTS * RAW_BYTES);
  uint64_t* a_empty = a_full + 2;
  uint64_t* acc_full = a_empty + 2;
  uint64_t* acc_empty = acc_full + X_ACC;
  uint64_t* raw_full = acc_empty + X_ACC;
  uint64_t* raw_empty = raw_full + X_RAW_SLOTS;
  uint64_t* w_full = raw_empty + X_RAW_SLOTS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w_full + 1);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
  int grp, r_begin, r_end;
  if (!locate_row_range(gt, a.b, range_len, blockIdx.x, grp, r_begin, r_end)) return;
  const int n_tiles = r_end - r_begin;

  for (int i = tid; i < min(2, n_tiles) * X_BUF_BYTES / 16; i += X_THREADS) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) { mbar_init(&a_full[i], 4); mbar_init(&a_empty[i], 1); }
    for (int i = 0; i < X_ACC; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 4); }
    for (int i = 0; i < X_RAW_SLOTS; ++i) { mbar_init(&raw_full[i], 1); mbar_init(&raw_empty[i], 4); }
    mbar_init(w_full, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc_all(tmem_slot);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(*tmem_slot);
  pdl_enter();

  if (warp == 0) {
    constexpr uint32_t OCT = PIECES * 48 * 16;             // filters: [filter row][octet][piece][column = kx, input channel][8]
    const uint32_t w_lo = plain_desc_lo(smem_u32(Wk), OCT), a_lo0 = plain_desc_lo(smem_u32(smem), X_PLANE_BYTES);
    bool ok = warp_wait(w_full, 0, abort_flag);
    if (!ok) *abort_flag = 1;
    int ab = 0;
    uint32_t ab_parity = 1;                                // of the wait for the accumulator's last reader; the first round's pass at once
    for (int t = 0; ok && t < n_tiles; ++t) {
      const int buf = t & 1;
      if (!warp_wait(&a_full[buf], (t >> 1) & 1, abort_flag)) { *abort_flag = 1; break; }
      tc_fence_after();
#pragma unroll 1
      for (int m = 0; m < 2; ++m) {
        if (!warp_wait(&acc_empty[ab], ab_parity, abort_flag)) { *abort_flag = 1; ok = false; break; }
        tc_fence_after();
        const uint32_t a_lo = a_lo0 + buf * (X_BUF_BYTES / 16) + m * 128 + 1, d = tmem + ab * 144;
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
          for (int q = 0; q < 2; ++q)                      // sixteen output channels
#pragma unroll
            for (int p = 0; p < PIECES; ++p)
              umma_f16(d + p * 48, a_lo + p * (X_PIECE_BYTES / 16) + 2 * q * (X_PLANE_BYTES / 16) + (2 - ky) * 16, plain_desc_hi(128),
                            w_lo + (ky * 4 + 2 * q) * (OCT / 16), plain_desc_hi(128), idesc_x3(48 * (PIECES - p), false), (ky | q | p) ? 1u : 0u);
        umma_commit(&acc_full[ab]);
        if (++ab == X_ACC) { ab = 0; ab_parity ^= 1; }
      }
      if (ok) umma_commit(&a_empty[buf]);
    }
  } else if (warp <= 8) {
    const int grp_w = (warp - 1) >> 2, lt = (tid - 32) & 127;
    for (int t = grp_w; t < n_tiles; t += 2) {
      const int buf = t & 1, slot = t & (X_RAW_SLOTS - 1);
      bool ok = mbar_wait(&raw_full[slot], (t / X_RAW_SLOTS) & 1);
      if (ok && t >= 2) ok = mbar_wait(&a_empty[buf], ((t >> 1) - 1) & 1);
      if (!__all_sync(0xffffffffu, ok && !*abort_flag)) { *abort_flag = 1; break; }
      const uint8_t* rp = raw + slot * RAW_BYTES;
#pragma unroll 1
      for (int e = lt; e < 4 * 49; e += 128) {
        const int o8 = e / 49, p = e - o8 * 49, py = p / 7, px = p - py * 7;
        uint8_t* d = smem + buf * X_BUF_BYTES + o8 * X_PLANE_BYTES + ((2 * py + 1) * 16 + 2 * px + 1) * 16;
        place_g2(rp, o8, p, [&](int j, int q, uint4 v) { *reinterpret_cast<uint4*>(d + q * X_PIECE_BYTES + ((j >> 1) * 16 + (j & 1)) * 16) = v; });
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) { mbar_arrive(&a_full[buf]); mbar_arrive(&raw_empty[slot]); }
    }
  } else if (warp == 17) {
    if (lane == 0) {
      mbar_expect_tx(w_full, BANK3_DX_BYTES);
      bulk_load(Wk, ws.bank2 + (int64_t)grp * BANK3_BYTES + BANK3_FWD_BYTES, BANK3_DX_BYTES, w_full);
      for (int t = 0; t < n_tiles; ++t) {
        const int slot = t & (X_RAW_SLOTS - 1);
        if ((t >= X_RAW_SLOTS && !mbar_wait(&raw_empty[slot], (t / X_RAW_SLOTS - 1) & 1)) || *abort_flag) { *abort_flag = 1; break; }
        const int64_t row = r_begin + t;
        mbar_expect_tx(&raw_full[slot], RAW_BYTES);
        bulk_load(raw + slot * RAW_BYTES, ws.dp2 + row * FLAT, FLAT * 4, &raw_full[slot]);
        bulk_load(raw + slot * RAW_BYTES + FLAT * 4, ws.code2 + row * FLAT, FLAT, &raw_full[slot]);
      }
    }
  } else {
    const int quarter = warp & 3, m = (warp - 9) >> 2;
    int ab = m;
    uint32_t ab_parity = 0;
    for (int t = 0; t < n_tiles; ++t) {
      if (!warp_wait(&acc_full[ab], ab_parity, abort_flag)) { *abort_flag = 1; break; }
      tc_fence_after();
      // the thread's position holds, per filter column kx, what the gradient AT this position sends through the taps of that
      // column; the input gradient here collects kx = 0 from the position to the right, kx = 1 from itself and kx = 2 from
      // the position to the left (zero borders make the rows' ends right)
      float e[3][16];
#pragma unroll
      for (int kx = 0; kx < 3; ++kx) {
        uint32_t lead[16], s1[16], s2[16];
        const uint32_t at = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(ab * 144 + kx * 16);
        tmem_ld16(at, lead);
        tmem_ld16(at + 48, s1);
        tmem_ld16(at + 96, s2);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) e[kx][i] = join3(__uint_as_float(lead[i]), __uint_as_float(s1[i]) + __uint_as_float(s2[i]));
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[ab]);
      ab += 2;                             // every second use of the accumulators is this group's
      if (ab >= X_ACC) { ab -= X_ACC; ab_parity ^= 1; }
      const int r = m * 128 + quarter * 32 + lane, y = r >> 4, x = r & 15;
#pragma unroll
      for (int ic = 0; ic < 16; ++ic) {
        const float right = __shfl_down_sync(0xffffffffu, e[0][ic], 1), left = __shfl_up_sync(0xffffffffu, e[2][ic], 1);
        e[1][ic] = (e[1][ic] + right) + (x == 0 ? 0.f : left);
      }
      if (y < 14 && x < 14) {              // [channel quad][position][4 channels]
        float4* out = reinterpret_cast<float4*>(ws.dp1 + (int64_t)(r_begin + t) * P1_ELEMS) + y * 14 + x;
#pragma unroll
        for (int q = 0; q < 4; ++q) out[q * 196] = make_float4(e[1][4 * q], e[1][4 * q + 1], e[1][4 * q + 2], e[1][4 * q + 3]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) { tc_fence_after(); tmem_free_all(tmem); }
  if (tid == 0 && *abort_flag) report_abort(ws.status);
}

// ------------------------------------------------------------------------------------------------
// Filter and bias gradient: dW[oc][ic][ky][kx] = sum over samples and positions of g2[oc][y][x] * p1pad[ic][y + ky][x + kx].
// Rows of the product: (piece of g2, output channel), 96 of 128 (the other 32 read what lies behind and are dropped); columns:
// (ky, piece of p1, input channel), 144; k: column parity of two image rows.  One MMA then takes all nine products of the pieces
// for a filter row's three taps, 42 a sample (14 per filter column kx, which has an accumulator of its own), with nothing to
// stage but g2: p1x is used as it arrives.  A sample's sums (14 instructions' worth) are added up in registers, the leading ones with
// the products of h and the others' pieces; the warps of the three pieces of g2 meet only when a sum is written out.
// Warps: 0 = MMA, 1 = copies of p1x, 2 = copies of dp2 and decisions, 3, 7, 11, 15 = staging (3 also sums the bias gradient), the others =
// read-out (tensor-memory quarter = piece, group of four warps = filter column).  A read-out takes a round trip of 425 clk to tensor memory
// per load, so it has as many registers as sixteen warps leave: three trips instead of six.  A CTA walks over a contiguous range of
// rows and writes a partial sum every seg_len rows and where the range leaves a worker.
//
// The zeros in g2's columns 14 and 15 meet column 13 of the map (slot 7) in the products of filter column 0 with even columns, and column 0 (slot
// 8) in those of filter column 1 with odd and of filter column 2 with even columns, which take nothing else from there.  In a sample with an
// infinity in one of the two slots (p1x is never NaN) the products are therefore taken in another order, and either slot is cleared once
// only they are left of those that read it.  (The staging warp that has least to stage looks for one.  A sum of such a sample with plain multiply-adds by the
// read-out warps costs the others 5 us at 128 x 128, by their registers.)
// ------------------------------------------------------------------------------------------------
constexpr int D_THREADS = 512, D_READERS = 288, D_P1_SLOTS = 3, D_RAW_SLOTS = 4;
constexpr int D_G_ROW = PIECES * 4 * 256;                    // image row of g2: [piece][octet][slot (x & 1) * 8 + x / 2][8 channels]
constexpr int D_G_BYTES = 14 * D_G_ROW + 1024;               // the dropped rows of the last image row read a kilobyte behind it
constexpr int D_GAP = 128;
constexpr int D_XCHG_BYTES = 3 * 2 * 48 * 32 * 4;            // read-out: [kx][piece m, l][column][lane]
constexpr int D_OUT_PITCH = 145;                             // write-out: an output channel's 144 filter taps, one word of padding
static_assert(32 * D_OUT_PITCH * 4 <= D_XCHG_BYTES, "the taps take the exchange area's place");
constexpr int D_BARS = 2 * D_P1_SLOTS + 2 * D_RAW_SLOTS + 2 * 2 + 2 * 3 + 1;
constexpr int D_SMEM = 2 * D_G_BYTES + D_P1_SLOTS * P1X_BYTES + D_GAP + D_XCHG_BYTES + D_RAW_SLOTS * RAW_BYTES + D_BARS * 8 + 16;
static_assert(D_SMEM <= 227 * 1024 && D_G_BYTES % 16 == 0, "shared memory");

__global__ void __launch_bounds__(D_THREADS, 1) conv2_dw_x3(GradStepArgs a, Workspace ws, int segs, int seg_len, int slots) {
  extern __shared__ __align__(128) uint8_t smem[];
  uint8_t* p1s = smem + 2 * D_G_BYTES;
  float* xchg = reinterpret_cast<float*>(p1s + D_P1_SLOTS * P1X_BYTES + D_GAP);
  uint8_t* raw = reinterpret_cast<uint8_t*>(xchg) + D_XCHG_BYTES;
  uint64_t* p1_full = reinterpret_cast<uint64_t*>(raw + D_RAW_SLOTS * RAW_BYTES);
  uint64_t* p1_empty = p1_full + D_P1_SLOTS;
  uint64_t* raw_full = p1_empty + D_P1_SLOTS;
  uint64_t* raw_empty = raw_full + D_RAW_SLOTS;
  uint64_t* g_full = raw_empty + D_RAW_SLOTS;
  uint64_t* g_empty = g_full + 2;
  uint64_t* acc_full = g_empty + 2;
  uint64_t* acc_empty = acc_full + 3;
  uint64_t* read = acc_empty + 3;                // the products so far have read their operands
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(read + 1);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  volatile uint32_t* infinite = tmem_slot + 2;   // [2] has the staged sample an infinity in columns 0 or 13?
  const int tid = threadIdx.x, lane = tid & 31, warp = warp_uniform(tid >> 5);
  const int total = a.W * a.b, r0 = blockIdx.x * segs * seg_len, r1 = min(r0 + segs * seg_len, total), n_samples = r1 - r0;

  // g2's columns 14 and 15 are never staged: zeros; what they meet has to be finite, also the sixteen bytes that a shifted read
  // goes beyond a sample's slot (border zeros of the next slot's sample, which may not have arrived yet or never will)
  for (int i = tid; i < 2 * 14 * PIECES * 4 * 2; i += D_THREADS) {
    const int run = i >> 1;
    *reinterpret_cast<uint4*>(smem + (run / (14 * PIECES * 4)) * D_G_BYTES + (run % (14 * PIECES * 4)) * 256 + 112 + (i & 1) * 128) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (tid <= D_P1_SLOTS) *reinterpret_cast<uint4*>(p1s + tid * P1X_BYTES) = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    for (int i = 0; i < D_P1_SLOTS; ++i) { mbar_init(&p1_full[i], 1); mbar_init(&p1_empty[i], 1); }
    for (int i = 0; i < D_RAW_SLOTS; ++i) { mbar_init(&raw_full[i], 1); mbar_init(&raw_empty[i], 4); }
    for (int i = 0; i < 2; ++i) { mbar_init(&g_full[i], 4); mbar_init(&g_empty[i], 1); }
    for (int i = 0; i < 3; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 3); }
    mbar_init(read, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc_all(tmem_slot);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(*tmem_slot);

  if (warp == 0) {
    constexpr uint32_t idesc = idesc_x3(144, true);
    // row index contiguous, no swizzle: the stride byte offset leads to the next eight rows (columns), the leading byte offset
    // to the next eight k, here the next image row
    const uint32_t g_lo0 = plain_desc_lo(smem_u32(smem), D_G_ROW), p_lo0 = plain_desc_lo(smem_u32(p1s), P1X_ROW);
    int slot = 0;
    uint32_t slot_parity = 0, read_parity = 0;
    bool ok = true;
    for (int n = 0; ok && n < n_samples; ++n) {
      const int st = n & 1;
      if (!warp_wait(&p1_full[slot], slot_parity, abort_flag) || !warp_wait(&g_full[st], (n >> 1) & 1, abort_flag)) { *abort_flag = 1; break; }
      tc_fence_after();
      const uint32_t g_lo = g_lo0 + st * (D_G_BYTES / 16), p_lo = p_lo0 + slot * (P1X_BYTES / 16);
      auto issue = [&](int kx, int k, uint32_t add) {                    // image rows 2 (k / 2) and + 1, columns of parity k & 1
        const int xp = (k & 1) + kx;                       // the first column read, 0 .. 3
        umma_f16(tmem + kx * 144, g_lo + (k >> 1) * (2 * D_G_ROW / 16) + (k & 1) * 8, plain_desc_hi(256),
                 p_lo + (k >> 1) * (2 * P1X_ROW / 16) + (xp & 1) * 8 + (xp >> 1), plain_desc_hi(256), idesc, add);
      };
      if (warp_uniform(infinite[st])) {
        for (int kx = 0; ok && kx < 3 && n > 0; ++kx) ok = warp_wait(&acc_empty[kx], (n - 1) & 1, abort_flag);
        tc_fence_after();
        auto clear = [&](int x_slot) {                     // of all rows and octets, in the leading piece
          umma_commit(read);
          if (!warp_wait(read, read_parity, abort_flag)) { ok = false; return; }
          read_parity ^= 1;
          *reinterpret_cast<uint4*>(p1s + slot * P1X_BYTES + (lane >> 1) * P1X_ROW + (lane & 1) * 256 + x_slot * 16) = make_uint4(0u, 0u, 0u, 0u);
          fence_proxy_async_smem();
          __syncwarp();
          tc_fence_after();
        };
        if (ok) {
#pragma unroll 1
          for (int k = 1; k < 14; k += 2) issue(0, k, k > 1);
#pragma unroll 1
          for (int k = 0; k < 14; k += 2) issue(1, k, k > 0);
          clear(8);
        }
        if (ok) {
#pragma unroll 1
          for (int k = 1; k < 14; k += 2) issue(1, k, 1);
#pragma unroll 1
          for (int k = 0; k < 14; ++k) issue(2, k, k > 0);
          clear(7);
        }
        if (ok) {
#pragma unroll 1
          for (int k = 0; k < 14; k += 2) issue(0, k, 1);
          for (int kx = 0; kx < 3; ++kx) umma_commit(&acc_full[kx]);
        } else {
          *abort_flag = 1;
        }
      } else {
#pragma unroll 1
        for (int kx = 0; kx < 3; ++kx) {
          if (n > 0 && !warp_wait(&acc_empty[kx], (n - 1) & 1, abort_flag)) { *abort_flag = 1; ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < 14; ++k) issue(kx, k, k > 0);
          umma_commit(&acc_full[kx]);
        }
      }
      if (!ok) break;
      umma_commit(&p1_empty[slot]);
      umma_commit(&g_empty[st]);
      if (++slot == D_P1_SLOTS) { slot = 0; slot_parity ^= 1; }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int slot = 0, use = 0;
      for (int n = 0; n < n_samples; ++n) {
        if ((use > 0 && !mbar_wait(&p1_empty[slot], (use - 1) & 1)) || *abort_flag) { *abort_flag = 1; break; }
        mbar_expect_tx(&p1_full[slot], P1X_BYTES);
        bulk_load(p1s + slot * P1X_BYTES, ws.p1x + (int64_t)(r0 + n) * P1X_BYTES, P1X_BYTES, &p1_full[slot]);
        if (++slot == D_P1_SLOTS) { slot = 0; ++use; }
      }
    }
  } else if (warp == 2) {
    if (lane == 0) {
      for (int n = 0; n < n_samples; ++n) {
        const int slot = n % D_RAW_SLOTS;
        if ((n >= D_RAW_SLOTS && !mbar_wait(&raw_empty[slot], (n / D_RAW_SLOTS - 1) & 1)) || *abort_flag) { *abort_flag = 1; break; }
        const int64_t row = r0 + n;
        mbar_expect_tx(&raw_full[slot], RAW_BYTES);
        bulk_load(raw + slot * RAW_BYTES, ws.dp2 + row * FLAT, FLAT * 4, &raw_full[slot]);
        bulk_load(raw + slot * RAW_BYTES + FLAT * 4, ws.code2 + row * FLAT, FLAT, &raw_full[slot]);
      }
    }
  } else if ((warp & 3) == 3) {
    const int lt = (warp >> 2) * 32 + lane;
    int s = r0 / a.b, wend = (s + 1) * a.b, seg = blockIdx.x * segs, send = r0 + seg_len;
    float gb = 0.f;                          // bias gradient; lane = output channel
    for (int n = 0; n < n_samples; ++n) {
      const int st = n & 1, slot = n % D_RAW_SLOTS, row = r0 + n;
      bool ok = mbar_wait(&raw_full[slot], (n / D_RAW_SLOTS) & 1);
      if (ok && n >= 2) ok = mbar_wait(&g_empty[st], ((n >> 1) - 1) & 1);
      if (!__all_sync(0xffffffffu, ok && !*abort_flag)) { *abort_flag = 1; break; }
      const uint8_t* rp = raw + slot * RAW_BYTES;
      if (warp == 15) {                      // (it stages one item a thread, the others two)
        const int p1_slot = n % D_P1_SLOTS;
        ok = mbar_wait(&p1_full[p1_slot], (n / D_P1_SLOTS) & 1);
        if (!__all_sync(0xffffffffu, ok && !*abort_flag)) { *abort_flag = 1; break; }
        uint32_t top = 0;
        if (lane < 28) {                     // slots 7 and 8 of a row of the map and an octet of channels: leading pieces, which are never negative
          const uint4* v = reinterpret_cast<const uint4*>(p1s + p1_slot * P1X_BYTES + ((lane >> 1) + 1) * P1X_ROW + (lane & 1) * 256 + 7 * 16);
#pragma unroll
          for (int i = 0; i < 2; ++i) top |= (v[i].x + 0x00800080u) | (v[i].y + 0x00800080u) | (v[i].z + 0x00800080u) | (v[i].w + 0x00800080u);
        }
        const bool any = __any_sync(0xffffffffu, (top & 0x80008000u) != 0);
        if (lane == 0) infinite[st] = any;
      }
#pragma unroll 1
      for (int e = lt; e < 4 * 49; e += 128) {
        const int o8 = e / 49, p = e - o8 * 49, py = p / 7, px = p - py * 7;
        uint8_t* d = smem + st * D_G_BYTES + 2 * py * D_G_ROW + o8 * 256 + px * 16;
        place_g2(rp, o8, p, [&](int j, int q, uint4 v) { *reinterpret_cast<uint4*>(d + (j >> 1) * D_G_ROW + q * 1024 + (j & 1) * 128) = v; });
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&g_full[st]);
      if (warp == 3) {
        const float* g = reinterpret_cast<const float*>(rp) + lane * 49;
        const uint8_t* code = rp + FLAT * 4 + (lane >> 2) * 196 + (lane & 3);
        float t[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int p = 0; p < 49; ++p) t[p % 7] += code[p * 4] < 4 ? g[p] : 0.f;
        gb += ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + t[6]);
        if (row + 1 == r1 || row + 1 == wend || row + 1 == send) {
          ws.part2[((int64_t)s * slots + (seg - (s * a.b) / seg_len)) * C2_GRAD + 4608 + lane] = gb;
          gb = 0.f;
          if (row + 1 == wend) { ++s; wend += a.b; }
          if (row + 1 == send) { ++seg; send += seg_len; }
        }
        __syncwarp();
      }
      if (lane == 0) mbar_arrive(&raw_empty[slot]);
    }
  } else {
    const int piece = warp & 3, kx = (warp >> 2) - 1;
    int s = r0 / a.b, wend = (s + 1) * a.b, seg = blockIdx.x * segs, send = r0 + seg_len;
    float sum[48];                           // (ky, input channel); lane = output channel
#pragma unroll
    for (int i = 0; i < 48; ++i) sum[i] = 0.f;
    bool ok = true;
    for (int n = 0; n < n_samples; ++n) {
      const int row = r0 + n;
      ok = ok && warp_wait(&acc_full[kx], n & 1, abort_flag);
      if (ok) {
        tc_fence_after();
        const uint32_t at = tmem + ((uint32_t)(piece * 32) << 16) + (uint32_t)(kx * 144);
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
          uint32_t h[16], m[16], l[16];
          tmem_ld16(at + ky * 48, h);
          if (piece < 2) tmem_ld16(at + ky * 48 + 16, m);
          if (piece < 1) tmem_ld16(at + ky * 48 + 32, l);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float v = piece == 0 ? join3(__uint_as_float(h[i]), __uint_as_float(m[i]) + __uint_as_float(l[i]))
                                       : (piece == 1 ? __uint_as_float(h[i]) + __uint_as_float(m[i]) : __uint_as_float(h[i]));
            sum[ky * 16 + i] += v;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[kx]);
      }
      if (!ok) *abort_flag = 1;              // and on to the write-out, where all nine warps stop
      if (row + 1 == r1 || row + 1 == wend || row + 1 == send) {
        // the nine warps meet: the pieces' sums of a filter column, then all columns' taps in the order of the output
        float* x = xchg + kx * (2 * 48 * 32);
        if (piece > 0) {
#pragma unroll
          for (int i = 0; i < 48; ++i) x[((piece - 1) * 48 + i) * 32 + lane] = sum[i];
        }
        if (!warps_agree<1, D_READERS>(ok)) break;
        if (piece == 0) {
#pragma unroll
          for (int i = 0; i < 48; ++i) sum[i] = join3(sum[i], x[i * 32 + lane] + x[(48 + i) * 32 + lane]);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(D_READERS) : "memory");
        if (piece == 0) {
#pragma unroll
          for (int i = 0; i < 48; ++i) xchg[lane * D_OUT_PITCH + (i & 15) * 9 + (i >> 4) * 3 + kx] = sum[i];
        }
        asm volatile("bar.sync 1, %0;" ::"n"(D_READERS) : "memory");
        float* part = ws.part2 + ((int64_t)s * slots + (seg - (s * a.b) / seg_len)) * C2_GRAD;
#pragma unroll
        for (int k = 0; k < 4608 / D_READERS; ++k) {
          const int i = k * D_READERS + (kx * 3 + piece) * 32 + lane;
          part[i] = xchg[i + i / 144];                       // D_OUT_PITCH = 144 + 1
        }
        asm volatile("bar.sync 1, %0;" ::"n"(D_READERS) : "memory");       // and has been read before the next write-out
#pragma unroll
        for (int i = 0; i < 48; ++i) sum[i] = 0.f;
        if (row + 1 == wend) { ++s; wend += a.b; }
        if (row + 1 == send) { ++seg; send += seg_len; }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) { tc_fence_after(); tmem_free_all(tmem); }
  if (tid == 0 && *abort_flag) report_abort(ws.status);
}

}  // namespace

#define TIMED(id, launch) do { if (prof) prof->begin(id, st); launch; if (prof) prof->end(st); } while (0)

int configure_x3_conv2_kernels() {
  const bool ok = allow_smem((const void*)conv2_fwd_x3, F_SMEM) == cudaSuccess && allow_smem((const void*)conv2_dx_x3, X_SMEM) == cudaSuccess &&
                  allow_smem((const void*)conv2_dw_x3, D_SMEM) == cudaSuccess;
  return ok ? 0 : -1;
}

const Bank3Taps& conv2_fwd_x3_taps() { return fold_tables().taps; }

void launch_conv2_fwd_x3(const GradStepArgs& a, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  int len;
  const int n = plan_row_ranges(gt, a.b, g_sm_count, 2, &len);
  TIMED(K_CONV2_FWD, launch_pdl(conv2_fwd_x3, dim3(n), F_THREADS, F_SMEM, st, a, gt, ws, len, fold_tables().fold));
}

void launch_conv2_dx_x3(const GradStepArgs& a, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  int len;
  const int n = plan_row_ranges(gt, a.b, g_sm_count, 1, &len);
  TIMED(K_CONV2_BWD, launch_pdl(conv2_dx_x3, dim3(n), X_THREADS, X_SMEM, st, a, gt, ws, len));
}

// Returns the number of partial-sum slots reserved per worker (the stride of part2) and, in *seg_len, the rows of a partial
// sum.  The workspace holds one slot per four samples of a worker and eight more.
// A CTA's rows are summed up to DW_SEG at a time: what single precision loses grows with a sum's length.
constexpr int DW_SEG = 16;
int launch_conv2_dw_x3(const GradStepArgs& a, const Workspace& ws, cudaStream_t st, Profiler* prof, int* seg_len) {
  const int total = a.W * a.b, most = (a.b + CONV_SPB - 1) / CONV_SPB + 8;
  const int rows = (total + g_sm_count - 1) / g_sm_count, segs = (rows + DW_SEG - 1) / DW_SEG;
  int len = (rows + segs - 1) / segs;
  while ((a.b - 1) / len + 2 > most) ++len;
  const int slots = (a.b - 1) / len + 2;
  TIMED(K_CONV2_DW, (conv2_dw_x3<<<(total + segs * len - 1) / (segs * len), D_THREADS, D_SMEM, st>>>(a, ws, segs, len, slots)));
  *seg_len = len;
  return slots;
}

}  // namespace psk
