// Second convolution (16 -> 32 channels, 3x3, pad 1, 14x14 maps) of the FP32 path: forward with ReLU and 2x2 max
// pooling, the gradient with respect to its input, and its filter / bias gradient, on the FP32 pipes.
//
// All three are 903,168 multiply-adds per sample, so what counts is how many of them a thread does per value it reads
// from shared memory (the FP32 pipes take 128 multiply-adds per clock and SM, shared memory gives 32 words):
//   - forward and input gradient: a thread owns a 2x2 block of output positions and 16 output channels (64 sums).
//     Per input channel it reads the 4x4 patch under its block (16 words) and, per tap, 16 filters as four 16-byte
//     loads that are the same for the whole warp (one wavefront each): 52 loads for 576 multiply-adds.
//   - filter gradient: a thread owns 8 output channels x 1 input channel x 9 taps (72 sums) and slides along an image
//     row: per position three new input words and two 16-byte loads of gradients for 72 multiply-adds.
// The multiply-adds are packed pairs over output channels (half the instructions; the pipe's rate is the same).
//
// Measured (B200, 128 workers x 128 samples, 29.6 GFLOP per product, 0.40 ms at the pipe's rate): forward 1.25 -> 0.70 ms;
// input and filter gradient together 8.40 -> 0.64 + 0.65 ms (the former kernel did both with one multiply-add per word
// read and skipped zero gradients with a branch that the lanes of a warp took differently).  At 2 x 8: 57 -> 13 us and
// 402 -> 15 + 15 us.  The FP32 pipe is busy 66 - 69 % of the time (ncu, half the samples); scalar multiply-adds instead: 0.78 / 0.72 /
// 0.67 ms; three blocks of 8-channel threads per SM: 0.77 / 0.66 ms.
#include "bf16x3.cuh"
#include "device_common.cuh"
#include "kernels.h"

namespace psk {

namespace {

// ------------------------------------------------------------------------------------------------
// Forward (FWD) and input gradient.  A block takes up to SPB samples that share a weight snapshot and NC of the output
// channels (blockIdx.y).  The input of CH channels at a time lies in zero-bordered planes (position (y, x) at row
// y + 1, column x + 2: pairs of columns stay 8-byte aligned), double-buffered unless one chunk holds all channels.  The
// input gradient's input is the gradient at the convolution's output: the pooled gradient put back at the pooling winners.
// ------------------------------------------------------------------------------------------------
constexpr int CV_PITCH = 22;                       // words per plane row (17 used); 2 x 22 = 12 mod 32 spreads the rows of a warp's patches
constexpr int CV_PLANE = 16 * CV_PITCH;
template <bool FWD> struct ConvShape { static constexpr int KIN = FWD ? C1 : C2, NOUT = FWD ? C2 : C1; };
template <bool FWD, int NC, int SPB, int CH> constexpr int conv_smem_bytes() {
  return 4 * (ConvShape<FWD>::KIN * 9 * NC + (CH < ConvShape<FWD>::KIN ? 2 : 1) * SPB * CH * CV_PLANE);
}
template <int SPB> __host__ __device__ constexpr int conv_threads() { return (49 * SPB + 31) / 32 * 32; }

template <bool FWD, int NC, int SPB, int CH>
__global__ void __launch_bounds__(conv_threads<SPB>(), SPB > 1 ? 2 : 1) conv2_direct(GradStepArgs a, GroupTable gt, Workspace ws) {
  constexpr int KIN = ConvShape<FWD>::KIN, THREADS = conv_threads<SPB>();
  constexpr int N_CHUNKS = KIN / CH, BUF = SPB * CH * CV_PLANE;
  extern __shared__ __align__(16) float sm[];
  float* w = sm;                                   // [input channel][tap][NC]
  float* planes = sm + KIN * 9 * NC;               // [buffer][sample][channel][16][CV_PITCH]
  const int tid = threadIdx.x, n0 = blockIdx.y * NC;
  int g, r0, r1;
  if (!locate_row_range(gt, a.b, SPB, blockIdx.x, g, r0, r1)) return;
  const int n_s = r1 - r0;
  const float* theta = gt.theta[g];

  // input staging: element e of a chunk
  constexpr int ITEMS = FWD ? SPB * CH * 98 : SPB * CH * 49, PER = (ITEMS + THREADS - 1) / THREADS;
  float gv[FWD ? 1 : PER];
  uint32_t gc[FWD ? 1 : PER];
  auto fetch = [&](int c, int buf) {
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int e = tid + k * THREADS;
      if (FWD) {        // two columns of a row of the first convolution's output, straight into the plane
        const int sp = e / (CH * 98), rem = e - sp * (CH * 98), ch = rem / 98, q = rem - ch * 98, y = q / 7, x2 = q - y * 7;
        if (sp < n_s)
          cp_async8(planes + buf * BUF + (sp * CH + ch) * CV_PLANE + (y + 1) * CV_PITCH + 2 * x2 + 2,
                    ws.p1 + (int64_t)(r0 + sp) * P1_ELEMS + (c * CH + ch) * 196 + 2 * q);
      } else {          // a pooled gradient and its decision, into registers
        const int sp = e / (CH * 49), rem = e - sp * (CH * 49);
        const int64_t at = (int64_t)(r0 + sp) * FLAT + c * CH * 49 + rem;
        const bool in = sp < n_s;
        gv[k] = in ? ws.dp2[at] : 0.f;
        gc[k] = in ? ws.code2[at] : 4u;
      }
    }
    if (FWD) cp_async_commit();
  };
  auto place = [&](int buf) {      // input gradient: the fetched elements' windows, losers cleared
    if constexpr (!FWD) {
#pragma unroll
      for (int k = 0; k < PER; ++k) {
        const int e = tid + k * THREADS;
        const int sp = e / (CH * 49), rem = e - sp * (CH * 49), ch = rem / 49, p = rem - ch * 49, py = p / 7, px = p - py * 7;
        if (e < ITEMS) {
          float* d = planes + buf * BUF + (sp * CH + ch) * CV_PLANE + (2 * py + 1) * CV_PITCH + 2 * px + 2;
          *reinterpret_cast<float2*>(d) = make_float2(gc[k] == 0u ? gv[k] : 0.f, gc[k] == 1u ? gv[k] : 0.f);
          *reinterpret_cast<float2*>(d + CV_PITCH) = make_float2(gc[k] == 2u ? gv[k] : 0.f, gc[k] == 3u ? gv[k] : 0.f);
        }
      }
    }
  };

  for (int t = tid; t < (N_CHUNKS > 1 ? 2 : 1) * BUF / 2; t += THREADS) reinterpret_cast<float2*>(planes)[t] = make_float2(0.f, 0.f);
  // filters of the block's output channels: forward w[ic][tap][oc]; input gradient w[oc][8 - tap][ic] (the tap that
  // reads a position shifted the other way)
  for (int t = tid; t < KIN * 9 * NC; t += THREADS) {
    const int n = t % NC, rest = t / NC, tap = rest % 9, k = rest / 9;
    w[t] = FWD ? theta[OFF_C2W + ((n0 + n) * C1 + k) * 9 + tap] : theta[OFF_C2W + (k * C1 + n0 + n) * 9 + 8 - tap];
  }
  __syncthreads();                                 // the borders are in place before copies land beside them
  pdl_enter();
  fetch(0, 0);
  place(0);
  const int sp = tid / 49, pos = tid - sp * 49, py = pos / 7, px = pos - py * 7;
  const bool active = sp < n_s;
  u64 acc[NC / 2][4];                              // channel pair x window element
#pragma unroll
  for (int o = 0; o < NC / 2; ++o) {
    const u64 bias = FWD ? pack2(theta[OFF_C2B + n0 + 2 * o], theta[OFF_C2B + n0 + 2 * o + 1]) : 0ull;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[o][j] = bias;
  }
  for (int c = 0; c < N_CHUNKS; ++c) {
    const int buf = c & 1;
    if (FWD) cp_async_wait<0>();
    __syncthreads();                               // chunk c is complete; the other buffer is no longer read
    if (c + 1 < N_CHUNKS) fetch(c + 1, buf ^ 1);
    if (active) {
      const float* src0 = planes + buf * BUF + sp * CH * CV_PLANE + 2 * py * CV_PITCH + 2 * px + 1;
      const float* w0 = w + c * CH * 9 * NC;
#pragma unroll 1
      for (int ch = 0; ch < CH; ++ch) {
        const float* src = src0 + ch * CV_PLANE;
        u64 patch[4][4];                           // every value in both halves
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float v0 = src[r * CV_PITCH], v3 = src[r * CV_PITCH + 3];
          const float2 v12 = *reinterpret_cast<const float2*>(src + r * CV_PITCH + 1);
          patch[r][0] = pack2(v0, v0); patch[r][1] = pack2(v12.x, v12.x); patch[r][2] = pack2(v12.y, v12.y); patch[r][3] = pack2(v3, v3);
        }
        const float4* wr = reinterpret_cast<const float4*>(w0 + ch * 9 * NC);
#pragma unroll
        for (int tap = 0; tap < 9; ++tap)
#pragma unroll
          for (int q = 0; q < NC / 4; ++q) {
            const float4 wv = wr[tap * (NC / 4) + q];
            const u64 wa = pack2(wv.x, wv.y), wb = pack2(wv.z, wv.w);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const u64 v = patch[(j >> 1) + tap / 3][(j & 1) + tap % 3];
              acc[2 * q][j] = ffma2(wa, v, acc[2 * q][j]);
              acc[2 * q + 1][j] = ffma2(wb, v, acc[2 * q + 1][j]);
            }
          }
      }
    }
    if (c + 1 < N_CHUNKS) place(buf ^ 1);
  }
  if (!active) return;
  const int64_t row = r0 + sp;
#pragma unroll
  for (int o = 0; o < NC / 2; ++o) {
    float v[2][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) unpack2(acc[o][j], v[0][j], v[1][j]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int n = n0 + 2 * o + h;
      if (FWD) {
        float best = fmaxf(v[h][0], 0.f);
        uint32_t bi = 0;
#pragma unroll
        for (int j = 1; j < 4; ++j) {
          const float r = fmaxf(v[h][j], 0.f);
          if (r > best) { best = r; bi = j; }
        }
        const Bf16x3 s = split3(best, 0.f);        // its readers are the dense layer's products
#pragma unroll
        for (int p = 0; p < PIECES; ++p) ws.p2x[((int64_t)p * a.W * a.b + row) * FLAT + n * 49 + pos] = (uint16_t)s.p[p];
        ws.code2[row * FLAT + n * 49 + pos] = best > 0.f ? (uint8_t)bi : (uint8_t)4;
      } else {
        float* d = ws.dp1 + row * P1_ELEMS + n * 196 + 2 * py * 14 + 2 * px;
        *reinterpret_cast<float2*>(d) = make_float2(v[h][0], v[h][1]);
        *reinterpret_cast<float2*>(d + 14) = make_float2(v[h][2], v[h][3]);
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Filter and bias gradient: dW[oc][ic][ky][kx] = sum over samples and positions of g2[oc][y][x] * p1pad[ic][y+ky][x+kx].
// A block of eight warps walks over a contiguous range of rows (sorted worker, sample) and writes a partial sum every
// seg_len rows and where the range leaves a worker.  Warp w: output-channel octets 2 (w & 1) and + 1 (one per half warp; lane % 16 = input
// channel), quarter w / 2 of the 196 positions (seven half rows of seven).  The next sample's inputs arrive (cp.async
// for the planes, registers for the gradients) while the current one is accumulated.
// ------------------------------------------------------------------------------------------------
constexpr int DW_THREADS = 256;
constexpr int DW_PITCH = 18, DW_PLANE = 16 * DW_PITCH + 2;       // 290 = 2 mod 32: sixteen planes, sixteen banks
constexpr int DW_BUF = 16 * DW_PLANE + 196 * 32;                 // planes, then gradients [position][32 output channels]
constexpr int DW_SMEM = 4 * (2 * DW_BUF + C2_GRAD);
static_assert(2 * DW_SMEM <= 227 * 1024, "two blocks per SM");
static_assert(DW_BUF % 4 == 0 && (16 * DW_PLANE) % 4 == 0, "16-byte aligned gradients");

__global__ void __launch_bounds__(DW_THREADS, 2) conv2_dw_direct(GradStepArgs a, Workspace ws, int segs, int seg_len, int slots) {
  extern __shared__ __align__(16) float sm[];
  float* red = sm + 2 * DW_BUF;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int total = a.W * a.b, r0 = blockIdx.x * segs * seg_len, r1 = min(r0 + segs * seg_len, total);
  const int ic = lane & 15, oct = 2 * (warp & 1) + (lane >> 4), quarter = warp >> 1;
  constexpr int PER_P = (C1 * 98 + DW_THREADS - 1) / DW_THREADS, PER_G = (FLAT + DW_THREADS - 1) / DW_THREADS;
  float gv[PER_G], gb = 0.f;
  uint32_t gc[PER_G];
  auto fetch = [&](int row, int buf) {
    float* pl = sm + buf * DW_BUF;
#pragma unroll
    for (int k = 0; k < PER_P; ++k) {
      const int e = tid + k * DW_THREADS, ch = e / 98, q = e - ch * 98, y = q / 7, x2 = q - y * 7;
      if (e < C1 * 98) cp_async8(pl + ch * DW_PLANE + (y + 1) * DW_PITCH + 2 * x2 + 2, ws.p1 + (int64_t)row * P1_ELEMS + 2 * e);
    }
    cp_async_commit();
#pragma unroll
    for (int k = 0; k < PER_G; ++k) {              // lane = output channel: its stores below meet no bank twice
      const int e = tid + k * DW_THREADS, oc = e & 31, p = e >> 5;
      gv[k] = e < FLAT ? ws.dp2[(int64_t)row * FLAT + oc * 49 + p] : 0.f;
      gc[k] = e < FLAT ? ws.code2[(int64_t)row * FLAT + oc * 49 + p] : 4u;
    }
  };
  auto place = [&](int buf) {
    float* gr = sm + buf * DW_BUF + 16 * DW_PLANE;
#pragma unroll
    for (int k = 0; k < PER_G; ++k) {
      const int e = tid + k * DW_THREADS, oc = e & 31, p = e >> 5, py = p / 7, px = p - py * 7;
      if (e < FLAT) {
        float* d = gr + (2 * py * 14 + 2 * px) * 32 + oc;
        d[0] = gc[k] == 0u ? gv[k] : 0.f;
        d[32] = gc[k] == 1u ? gv[k] : 0.f;
        d[14 * 32] = gc[k] == 2u ? gv[k] : 0.f;
        d[15 * 32] = gc[k] == 3u ? gv[k] : 0.f;
        if (gc[k] < 4u) gb += gv[k];
      }
    }
  };
  for (int t = tid; t < 16 * DW_PLANE; t += DW_THREADS) sm[t] = sm[DW_BUF + t] = 0.f;
  __syncthreads();
  fetch(r0, 0);
  place(0);
  u64 acc[9][4];                                   // tap x output-channel pair
#pragma unroll
  for (int t = 0; t < 9; ++t)
#pragma unroll
    for (int o = 0; o < 4; ++o) acc[t][o] = 0ull;
  int s = r0 / a.b, wend = (s + 1) * a.b, seg = blockIdx.x * segs, send = r0 + seg_len;
  for (int row = r0; row < r1; ++row) {
    const int buf = (row - r0) & 1;
    cp_async_wait<0>();
    __syncthreads();
    const bool more = row + 1 < r1;
    const bool flush = !more || row + 1 == wend || row + 1 == send;
    if (more) fetch(row + 1, buf ^ 1);
    const float* pl = sm + buf * DW_BUF + ic * DW_PLANE;
    const float* gr = sm + buf * DW_BUF + 16 * DW_PLANE + oct * 8;
#pragma unroll 1
    for (int i = 0; i < 7; ++i) {
      const int hr = quarter * 7 + i, y = hr >> 1, x0 = (hr & 1) * 7;
      const float* src = pl + y * DW_PITCH + x0 + 1;
      const float4* gp = reinterpret_cast<const float4*>(gr + (y * 14 + x0) * 32);
      u64 col[3][3];                               // [column mod 3][row]
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) { const float v = src[ky * DW_PITCH + k]; col[k][ky] = pack2(v, v); }
#pragma unroll
      for (int xx = 0; xx < 7; ++xx) {
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) { const float v = src[ky * DW_PITCH + xx + 2]; col[(xx + 2) % 3][ky] = pack2(v, v); }
        const float4 ga = gp[xx * 8], gq = gp[xx * 8 + 1];
        const u64 g2[4] = {pack2(ga.x, ga.y), pack2(ga.z, ga.w), pack2(gq.x, gq.y), pack2(gq.z, gq.w)};
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
          for (int kx = 0; kx < 3; ++kx)
#pragma unroll
            for (int o = 0; o < 4; ++o) acc[ky * 3 + kx][o] = ffma2(g2[o], col[(xx + kx) % 3][ky], acc[ky * 3 + kx][o]);
      }
    }
    if (more && !flush) place(buf ^ 1);
    if (flush) {
      // the four position quarters are added in order; the bias sums (one output channel per lane) in warp order
      float* part = ws.part2 + ((int64_t)s * slots + (seg - (s * a.b) / seg_len)) * C2_GRAD;
      for (int q = 0; q < 4; ++q) {
        if (quarter == q) {
#pragma unroll
          for (int o = 0; o < 4; ++o)
#pragma unroll
            for (int t = 0; t < 9; ++t) {
              float lo, hi;
              unpack2(acc[t][o], lo, hi);
              float* d = red + ((oct * 8 + 2 * o) * 16 + ic) * 9 + t;
              d[0] = q ? d[0] + lo : lo;
              d[144] = q ? d[144] + hi : hi;
            }
        }
        __syncthreads();
      }
      for (int q = 0; q < 8; ++q) {
        if (warp == q) red[4608 + lane] = q ? red[4608 + lane] + gb : gb;
        __syncthreads();
      }
      for (int t = tid; t < C2_GRAD; t += DW_THREADS) part[t] = red[t];
#pragma unroll
      for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[t][o] = 0ull;
      gb = 0.f;
      if (row + 1 == wend) { ++s; wend += a.b; }
      if (row + 1 == send) { ++seg; send += seg_len; }
      __syncthreads();                             // the sums have been read before the next flush overwrites them
      if (more) place(buf ^ 1);
    }
  }
}

template <bool FWD, int NC, int SPB, int CH>
bool set_smem() {
  return allow_smem((const void*)(conv2_direct<FWD, NC, SPB, CH>), conv_smem_bytes<FWD, NC, SPB, CH>()) == cudaSuccess;
}

template <bool FWD, int NC, int SPB, int CH>
void run_conv(const GradStepArgs& a, const GroupTable& gt, const Workspace& ws, cudaStream_t st) {
  launch_pdl(conv2_direct<FWD, NC, SPB, CH>, dim3(group_tiles(gt, a.b, SPB), ConvShape<FWD>::NOUT / NC), conv_threads<SPB>(),
             conv_smem_bytes<FWD, NC, SPB, CH>(), st, a, gt, ws);
}

}  // namespace

#define TIMED(id, launch) do { if (prof) prof->begin(id, st); launch; if (prof) prof->end(st); } while (0)

int configure_fp32_conv2_kernels() {
  const bool ok = set_smem<true, 16, 5, 4>() && set_smem<true, 8, 5, 4>() && set_smem<true, 4, 1, 16>() && set_smem<false, 16, 5, 4>() &&
                  set_smem<false, 8, 5, 4>() && set_smem<false, 4, 1, 32>() &&
                  allow_smem((const void*)(conv2_dw_direct), DW_SMEM) == cudaSuccess;
  return ok ? 0 : -1;
}

void launch_conv2_direct(bool fwd, const GradStepArgs& a, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  const int rows = a.W * a.b;
  const int id = fwd ? K_CONV2_FWD : K_CONV2_BWD;
  // Few rows: one sample and 4 channels per block of 64 threads, so that 16 samples make 128 (64) blocks; then 5 samples
  // x 8 channels; then 5 samples x 16 channels.  Forward + input gradient in us (with ~6 us of event overhead each) at
  // 64 / 128 / 256 / 1024 / 1536 / 2048 rows: 4 channels 30 / 38 / 62 / 176 / 251 / 322; 8 channels 42 / 42 / 50 / 113 /
  // 166 / 203; 16 channels 66 / 66 / 66 / 124 / 180 / 197.
  const int variant = rows <= 128 ? 2 : (rows <= 1536 ? 1 : 0);
  if (fwd) {
    if (variant == 2) TIMED(id, (run_conv<true, 4, 1, 16>(a, gt, ws, st)));
    else if (variant == 1) TIMED(id, (run_conv<true, 8, 5, 4>(a, gt, ws, st)));
    else TIMED(id, (run_conv<true, 16, 5, 4>(a, gt, ws, st)));
  } else {
    if (variant == 2) TIMED(id, (run_conv<false, 4, 1, 32>(a, gt, ws, st)));
    else if (variant == 1) TIMED(id, (run_conv<false, 8, 5, 4>(a, gt, ws, st)));
    else TIMED(id, (run_conv<false, 16, 5, 4>(a, gt, ws, st)));
  }
}

// Returns the number of partial-sum slots reserved per worker (the stride of part2) and, in *seg_len, the rows of a partial
// sum.  The workspace holds one slot per four samples of a worker and eight more.
// Two blocks per SM share the rows, and a block's rows are summed up to DW_SEG at a time: a thread's sum runs over a quarter of
// the positions of that many samples, and what single precision loses grows with its length.  Relative error of a worker's
// filter gradient at 128 x 128 (55 rows per block) with one sum per block: 2.5e-7; with up to
// 32, 16 and 8 rows: 1.7e-7, 1.4e-7 and 1.3e-7, for 11, 19 and 30 us more in a tick of 3.9 ms.  Four samples at a time, as the
// former kernel summed them: 1.5e-7.
constexpr int DW_SEG = 16;
int launch_conv2_dw_direct(const GradStepArgs& a, const Workspace& ws, cudaStream_t st, Profiler* prof, int* seg_len) {
  const int total = a.W * a.b, most = (a.b + CONV_SPB - 1) / CONV_SPB + 8;
  const int rows = (total + 2 * g_sm_count - 1) / (2 * g_sm_count), segs = (rows + DW_SEG - 1) / DW_SEG;
  int len = (rows + segs - 1) / segs;
  while ((a.b - 1) / len + 2 > most) ++len;
  const int slots = (a.b - 1) / len + 2;
  TIMED(K_CONV2_DW, (conv2_dw_direct<<<(total + segs * len - 1) / (segs * len), DW_THREADS, DW_SMEM, st>>>(a, ws, segs, len, slots)));
  *seg_len = len;
  return slots;
}

}  // namespace psk
