// Worker-side gradient step, FP32 path (the second convolution is in grad_kernels_x3_conv2.cu, the dense layer in grad_kernels_x3_gemm.cu): the paper's small CNN (model endnote),
// forward and backward, for W workers that may hold different weight snapshots.
//
// Rows of every activation buffer are (sorted worker s, sample i) -> s*b + i, where the sorted
// order places workers that share a snapshot next to each other, so that a group's samples form
// one contiguous row range and the dense layers can run one tiled product per group.
//
// Every reduction is taken in a fixed order (no floating-point atomics), so that two runs on the
// same inputs give the same bits.
#include "bf16x3.cuh"
#include "device_common.cuh"
#include "kernels.h"

namespace psk {

namespace {

// ---- conv1 (1->16, 3x3, pad 1) + ReLU + 2x2 max pool, and its filter gradient.  (FP32 path; the tensor-core path has its own kernels.)
// A thread owns a quad of four output channels, packed multiply-adds over channel pairs, and takes seven of a sample's 784 items
// (pooled position, quad) in turn: per item it reads the 4x4 input patch under its pooling window once.  The next sample's
// image is fetched into registers meanwhile.
// Measured (~6 us of event overhead included) at 128 x 128 (3.7 GFLOP, 58 us at the packed multiply-add's rate) / 16 x 64: forward 193 / 20.1 us
// with scalar multiply-adds and all sixteen channels of a position in one thread, 162 / 17 now, 187 with six blocks per SM (80 registers);
// filter gradient 171 / 19.0 with one multiply-add per pixel read, 146 / 19.0 now (170 / 24 with an item's gradients fetched one item
// ahead).  The FMA pipe is busy for half of the cycles, the issue slots likewise: four blocks of four warps leave latencies open.
constexpr int CONV1_SPB = 8;            // most samples per block, forward
constexpr int CONV1_ITEMS = 112;        // items taken at a time: 28 positions (two rows of 14) x 4 quads
constexpr int CONV1_THREADS = 128;      // the last sixteen have none
constexpr int CONV1_PITCH = 32, CONV1_IMAGE = 30 * CONV1_PITCH;      // zero-bordered image, column x at x + 1

// The thread's seven pixels of an image; where they go.
struct ImagePart {
  float v[7];
  __device__ __forceinline__ void load(const float* x, int tid) {
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = tid < CONV1_ITEMS ? x[tid + CONV1_ITEMS * k] : 0.f;
  }
  __device__ __forceinline__ void store(float* image, int tid) const {      // 112 pixels = four rows
    float* d = image + (tid / IMG + 1) * CONV1_PITCH + tid % IMG + 1;
    if (tid < CONV1_ITEMS) {
#pragma unroll
      for (int k = 0; k < 7; ++k) d[4 * k * CONV1_PITCH] = v[k];
    }
  }
  // Is one of them infinite or NaN?
  __device__ __forceinline__ bool odd() const {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 7; ++k) t = fmaf(v[k], 0.f, t);
    return t != t;
  }
};
// The 4x4 patch under the pooling window at (py, px), every value in both halves.
__device__ __forceinline__ void load_patch(const float* image, int py, int px, u64 (&dup)[4][4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float2 lo = *reinterpret_cast<const float2*>(image + (2 * py + r) * CONV1_PITCH + 2 * px);
    const float2 hi = *reinterpret_cast<const float2*>(image + (2 * py + r) * CONV1_PITCH + 2 * px + 2);
    dup[r][0] = pack2(lo.x, lo.x); dup[r][1] = pack2(lo.y, lo.y); dup[r][2] = pack2(hi.x, hi.x); dup[r][3] = pack2(hi.y, hi.y);
  }
}

// The second convolution's filters of a weight group as its kernels' operands, one row of eight values (in pieces) per thread.
// Blocks of conv1_fwd beyond its workers do it, so that the next kernel finds them without a launch or a fork of their own.
// Behind them come, in an evaluation, W1_UNITS blocks per weight group for the dense layer's.
constexpr int BANK3_ROWS = 2 * BANK3_FWD_ROWS + 12 * 48, BANK3_UNITS = (BANK3_ROWS + CONV1_THREADS - 1) / CONV1_THREADS;      // blocks per weight group
constexpr int W1_UNITS = W1_ELEMS / (8 * CONV1_THREADS);
static_assert(W1_ELEMS % (8 * CONV1_THREADS) == 0, "whole blocks");
__device__ __forceinline__ void build_bank3(const float* __restrict__ theta, uint8_t* __restrict__ bank, int e, const Bank3Taps& taps) {
  if (e >= BANK3_ROWS) return;
  float v[8];
  uint8_t* d;
  int piece_bytes;
  if (e < 2 * BANK3_FWD_ROWS) {      // forward: [piece][octet of input channels][row = block, output channel]
    const int oct = e / BANK3_FWD_ROWS, row = e - oct * BANK3_FWD_ROWS, oc = row & 31, tap = taps.tap[row >> 5];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = theta[OFF_C2W + (oc * 16 + oct * 8 + i) * 9 + tap];
    d = bank + e * 16;
    piece_bytes = 2 * BANK3_FWD_ROWS * 16;
  } else {                           // input gradient: [filter row][octet of output channels][piece][column = kx, input channel]
    const int u = e - 2 * BANK3_FWD_ROWS, ko = u / 48, col = u - ko * 48, ky = ko >> 2, o8 = ko & 3, kx = col >> 4, ic = col & 15;
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = theta[OFF_C2W + ((o8 * 8 + i) * 16 + ic) * 9 + ky * 3 + kx];
    d = bank + BANK3_FWD_BYTES + (ko * PIECES * 48 + col) * 16;
    piece_bytes = 48 * 16;
  }
  const float more = e < 2 * BANK3_FWD_ROWS ? LOST_CONV2 : 0.f;
  const Bf16x3 s[4] = {split3(v[0], v[1], more), split3(v[2], v[3], more), split3(v[4], v[5], more), split3(v[6], v[7], more)};
#pragma unroll
  for (int p = 0; p < PIECES; ++p) *reinterpret_cast<uint4*>(d + p * piece_bytes) = make_uint4(s[0].p[p], s[1].p[p], s[2].p[p], s[3].p[p]);
}

__global__ void __launch_bounds__(CONV1_THREADS, 4) conv1_fwd(GradStepArgs a, WorkerTable wt, GroupTable gt, Workspace ws, int spb, int w1_units, const __grid_constant__ Bank3Taps taps) {
  __shared__ __align__(16) float xs[2][CONV1_IMAGE];
  const int s = blockIdx.y, tid = threadIdx.x;
  if (s >= a.W) {
    const int u = (s - a.W) * gridDim.x + blockIdx.x, u1 = u - gt.n_groups * BANK3_UNITS;
    pdl_enter();
    if (u1 < 0) {
      const int g = u / BANK3_UNITS;
      build_bank3(gt.theta[g], ws.bank2 + (int64_t)g * BANK3_BYTES, (u - g * BANK3_UNITS) * CONV1_THREADS + tid, taps);
    } else if (u1 < gt.n_groups * w1_units) {
      const int g = u1 / W1_UNITS;
      split_w1(gt.theta[g], ws.w1x, g, ((u1 - g * W1_UNITS) * CONV1_THREADS + tid) * 8);
    }
    return;
  }
  const float* theta = group_theta(wt, gt, s);
  for (int t = tid; t < 2 * CONV1_IMAGE; t += CONV1_THREADS) (&xs[0][0])[t] = 0.f;
  const int cg = tid & 3, px = (tid >> 2) % 14, py0 = (tid >> 2) / 14;
  const int i0 = blockIdx.x * spb, i1 = min(i0 + spb, a.b);
  const float* x = a.x + (int64_t)wt.src[s] * a.b * (IMG * IMG);
  pdl_enter();       // the weights may come from the apply just before
  ImagePart next;
  next.load(x + (int64_t)i0 * (IMG * IMG), tid);
  u64 wp[2][10];     // wp[cp][k] = tap k of channels 4 cg + 2 cp and + 1; k = 9 is the bias
#pragma unroll
  for (int cp = 0; cp < 2; ++cp) {
    const int c0 = 4 * cg + 2 * cp;
#pragma unroll
    for (int k = 0; k < 9; ++k) wp[cp][k] = pack2(theta[OFF_C1W + c0 * 9 + k], theta[OFF_C1W + (c0 + 1) * 9 + k]);
    wp[cp][9] = pack2(theta[OFF_C1B + c0], theta[OFF_C1B + c0 + 1]);
  }
  __syncthreads();
  next.store(xs[0], tid);
  for (int i = i0; i < i1; ++i) {
    const int cur = (i - i0) & 1;
    __syncthreads();                       // image `cur` is complete; image `cur^1` is no longer read
    if (i + 1 < i1) next.load(x + (int64_t)(i + 1) * (IMG * IMG), tid);
    if (tid < CONV1_ITEMS) {
      const int64_t row = (int64_t)s * a.b + i;
      // a position's channel quad in pieces, half of a 16-byte slot each; Y and X in the bordered map
      uint8_t* out = ws.p1x + row * P1X_BYTES + (cg >> 1) * 256 + (cg & 1) * 8;
      auto slot = [&](int Y, int X) { return out + Y * P1X_ROW + ((X & 1) * 8 + (X >> 1)) * 16; };
      {                                    // the zeros at either end of the fourteen image rows: whole runs leave
        uint8_t* d = slot((tid >> 3) + 1, ((tid >> 2) & 1) * 15);
#pragma unroll
        for (int p = 0; p < PIECES; ++p) *reinterpret_cast<uint2*>(d + p * 512) = make_uint2(0u, 0u);
      }
#pragma unroll 1
      for (int k = 0; k < 7; ++k) {
        const int py = py0 + 2 * k;
        u64 dup[4][4], acc[2][4];
        load_patch(xs[cur], py, px, dup);
#pragma unroll
        for (int cp = 0; cp < 2; ++cp)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[cp][j] = wp[cp][9];
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
          for (int kx = 0; kx < 3; ++kx)
#pragma unroll
            for (int cp = 0; cp < 2; ++cp)
#pragma unroll
              for (int j = 0; j < 4; ++j) acc[cp][j] = ffma2(wp[cp][ky * 3 + kx], dup[(j >> 1) + ky][(j & 1) + kx], acc[cp][j]);
        float v[4][4];     // [channel][window element]
#pragma unroll
        for (int cp = 0; cp < 2; ++cp)
#pragma unroll
          for (int j = 0; j < 4; ++j) unpack2(acc[cp][j], v[2 * cp][j], v[2 * cp + 1][j]);
        // ReLU then max = max then ReLU; the winner is the first window element that reaches the maximum.  The maximum is taken
        // against the smallest positive number: no element of a dead window equals it, and its pieces are zeros.
        float best[4];
        uint32_t codes = 0u;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float m = fmaxf(fmaxf(fmaxf(v[c][0], v[c][1]), fmaxf(v[c][2], v[c][3])), __int_as_float(1));
          best[c] = m;
          uint32_t e = v[c][3] == m ? 3u << (8 * c) : 4u << (8 * c);
          e = v[c][2] == m ? 2u << (8 * c) : e;
          e = v[c][1] == m ? 1u << (8 * c) : e;
          codes |= v[c][0] == m ? 0u : e;
        }
        const Bf16x3 q0 = split3(best[0], best[1]), q1 = split3(best[2], best[3]);
        uint8_t* d = slot(py + 1, px + 1);
#pragma unroll
        for (int p = 0; p < PIECES; ++p) *reinterpret_cast<uint2*>(d + p * 512) = make_uint2(q0.p[p], q1.p[p]);
        reinterpret_cast<uint32_t*>(ws.code1 + row * P1_ELEMS)[cg * 196 + py * 14 + px] = codes;
      }
    }
    next.store(xs[cur ^ 1], tid);
  }
}

// ---- backward through pool1, ReLU and conv1 (filter / bias gradients only: the input needs none): per window element the pooled
// gradients of the channels that it won, all others cleared, times the patch.  A sample's gradients and decisions arrive by
// asynchronous copies while the sample before is added up.  A cleared gradient times a pixel that is not finite is NaN, and no part of the
// gradient, which is a sum over the winners' patches: an image with such a pixel takes its products one by one.
constexpr int CONV1B_SPB = 16;            // most samples per block
__global__ void __launch_bounds__(CONV1_THREADS, 4) conv1_bwd(GradStepArgs a, WorkerTable wt, Workspace ws, int spb, int n_chunks) {
  __shared__ __align__(16) float xs[2][CONV1_IMAGE];
  __shared__ __align__(16) float4 gs[2][7][CONV1_ITEMS];
  __shared__ uint32_t cs[2][7][CONV1_ITEMS];
  float (*red)[C1_GRAD] = reinterpret_cast<float (*)[C1_GRAD]>(&gs[0][0][0]);      // the warps' sums take their place
  const int s = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cg = tid & 3, pos0 = tid >> 2, px = pos0 % 14, py0 = pos0 / 14;
  const bool active = tid < CONV1_ITEMS;
  for (int t = tid; t < 2 * CONV1_IMAGE; t += CONV1_THREADS) (&xs[0][0])[t] = 0.f;
  const int i0 = blockIdx.x * spb, i1 = min(i0 + spb, a.b);
  const float* x = a.x + (int64_t)wt.src[s] * a.b * (IMG * IMG);
  const int64_t row0 = (int64_t)s * a.b;
  u64 gw[2][9];                             // channel pair x tap
  float gb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int cp = 0; cp < 2; ++cp)
#pragma unroll
    for (int k = 0; k < 9; ++k) gw[cp][k] = 0ull;
  // a thread's items of a sample, in its own places: dp1 and the decisions are [quad][position][4 channels]
  auto fetch = [&](int i) {
    if (active) {
      const int buf = (i - i0) & 1;
      const float4* g = reinterpret_cast<const float4*>(ws.dp1 + (row0 + i) * P1_ELEMS) + cg * 196 + pos0;
      const uint32_t* c = reinterpret_cast<const uint32_t*>(ws.code1 + (row0 + i) * P1_ELEMS) + cg * 196 + pos0;
#pragma unroll
      for (int k = 0; k < 7; ++k) {
        cp_async16(&gs[buf][k][tid], g + 28 * k, true);
        cp_async4(&cs[buf][k][tid], c + 28 * k);
      }
    }
    cp_async_commit();
  };
  ImagePart next;
  next.load(x + (int64_t)i0 * (IMG * IMG), tid);
  __syncthreads();
  next.store(xs[0], tid);
  pdl_enter();
  fetch(i0);
  for (int i = i0; i < i1; ++i) {
    const int cur = (i - i0) & 1;
    const bool odd = __syncthreads_or(next.odd());      // image `cur`, which `next` still holds, is complete; image `cur^1` is no longer read
    if (i + 1 < i1) {
      next.load(x + (int64_t)(i + 1) * (IMG * IMG), tid);
      fetch(i + 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    if (odd) {
#pragma unroll 1
      for (int k = 0; k < 7 && active; ++k) {
        const float4 g4 = gs[cur][k][tid];
        const uint32_t code = cs[cur][k][tid];
        const float g[4] = {g4.x, g4.y, g4.z, g4.w};
        const float* window = xs[cur] + 2 * (py0 + 2 * k) * CONV1_PITCH + 2 * px;
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          const uint32_t c = (code >> (8 * ch)) & 255u;
          if (c > 3u) continue;
          gb[ch] += g[ch];
          const float* patch = window + (c >> 1) * CONV1_PITCH + (c & 1);
#pragma unroll
          for (int t = 0; t < 9; ++t) {
            float v[2];
            unpack2(gw[ch >> 1][t], v[0], v[1]);
            v[ch & 1] = fmaf(g[ch], patch[t / 3 * CONV1_PITCH + t % 3], v[ch & 1]);
            gw[ch >> 1][t] = pack2(v[0], v[1]);
          }
        }
      }
    }
#pragma unroll 1
    for (int k = odd ? 7 : 0; k < 7; ++k) {
      const float4 g4 = active ? gs[cur][k][tid] : make_float4(0.f, 0.f, 0.f, 0.f);
      const uint32_t code = active ? cs[cur][k][tid] : 0x04040404u;
      const float g[4] = {g4.x, g4.y, g4.z, g4.w};
      u64 dup[4][4];
      load_patch(xs[cur], active ? py0 + 2 * k : 0, px, dup);
      uint32_t c[4];
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        c[ch] = (code >> (8 * ch)) & 255u;
        gb[ch] += c[ch] < 4u ? g[ch] : 0.f;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
          const u64 gj = pack2(c[2 * cp] == j ? g[2 * cp] : 0.f, c[2 * cp + 1] == j ? g[2 * cp + 1] : 0.f);
#pragma unroll
          for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) gw[cp][ky * 3 + kx] = ffma2(gj, dup[(j >> 1) + ky][(j & 1) + kx], gw[cp][ky * 3 + kx]);
        }
    }
    next.store(xs[cur ^ 1], tid);
  }
  __syncthreads();
  // fixed-order sums: the eight lanes of a quad, then the four warps
  auto over_lanes = [](float v) {
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
#pragma unroll
  for (int cp = 0; cp < 2; ++cp)
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      float lo, hi;
      unpack2(gw[cp][k], lo, hi);
      lo = over_lanes(lo);
      hi = over_lanes(hi);
      if (lane < 4) {
        red[warp][(4 * cg + 2 * cp) * 9 + k] = lo;
        red[warp][(4 * cg + 2 * cp + 1) * 9 + k] = hi;
      }
    }
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    const float t = over_lanes(gb[ch]);
    if (lane < 4) red[warp][144 + 4 * cg + ch] = t;
  }
  __syncthreads();
  float* part = ws.part1 + ((int64_t)s * n_chunks + blockIdx.x) * C1_GRAD;
  for (int o = tid; o < C1_GRAD; o += CONV1_THREADS) part[o] = (red[0][o] + red[1][o]) + (red[2][o] + red[3][o]);
}

// ---- sums the per-block partial gradients in a fixed order, finishes the loss and zeroes the padding.
// part1 and part2 hold n_chunks / n_chunks2 slots per worker; all of them are summed when seg_len == 0, otherwise one
// for every range of seg_len rows that meets the worker's b rows.
// A worker's outputs are numbered conv2 (4640), conv1 (160), output layer (5642), loss, padding; a block takes
// `per_block` of them.  With few workers the time is a thread's chain of loads, so its terms are fetched eight at a time.
constexpr int RED_OUTPUTS = C2_GRAD + C1_GRAD + (NCLS * HID + HID + NCLS) + 1 + (P_PAD - P);

// p[0] + p[stride] + ... (n terms), eight loads in flight.  Eight terms are added in pairs before they join the sum: it rounds
// an eighth as often, and the error of a few hundred terms stays near a single rounding.
__device__ __forceinline__ float sum_slots(const float* p, int n, int64_t stride) {
  float t = 0.f;
  for (int c = 0; c < n; c += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = c + u < n ? p[(c + u) * stride] : 0.f;
    t += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
  }
  return t;
}
// slots of worker s in use
__device__ __forceinline__ int used_slots(int s, int b, int seg_len, int n_chunks) {
  return seg_len > 0 ? (s * b + b - 1) / seg_len - (s * b) / seg_len + 1 : n_chunks;
}

__global__ void __launch_bounds__(256) conv_grad_reduce(GradStepArgs a, WorkerTable wt, Workspace ws, int per_block, int n_chunks, int seg_len1,
                                                        int n_chunks2, int seg_len) {
  const int s = blockIdx.x, b = a.b, split = fc2_split(a.W, b);
  float* grad = wt.grad[s];
  pdl_enter();
  const int used2 = used_slots(s, b, seg_len, n_chunks2), used1 = used_slots(s, b, seg_len1, n_chunks);
  for (int v = blockIdx.y * per_block + threadIdx.x; v < min(RED_OUTPUTS, ((int)blockIdx.y + 1) * per_block); v += 256) {
    int o = v;
    if (o < C2_GRAD) {
      grad[OFF_C2W + o] = sum_slots(ws.part2 + (int64_t)s * n_chunks2 * C2_GRAD + o, used2, C2_GRAD);
      continue;
    }
    o -= C2_GRAD;
    if (o < C1_GRAD) {
      grad[OFF_C1W + o] = sum_slots(ws.part1 + (int64_t)s * n_chunks * C1_GRAD + o, used1, C1_GRAD);
      continue;
    }
    o -= C1_GRAD;
    if (o <= NCLS * HID + HID + NCLS) {
      const float t = sum_slots(ws.partf + (int64_t)s * split * FC_PART + o, split, FC_PART);
      if (o < NCLS * HID) grad[OFF_F2W + o] = t;
      else if (o < NCLS * HID + HID) grad[OFF_F1B + o - NCLS * HID] = t;
      else if (o < NCLS * HID + HID + NCLS) grad[OFF_F2B + o - NCLS * HID - HID] = t;
      else a.loss[wt.src[s]] = t * (1.0f / (float)b);
      continue;
    }
    o -= NCLS * HID + HID + NCLS + 1;
    grad[P + o] = 0.f;
  }
}

// ---- the summed step's final reduction: ONE gradient vector, the sum over all workers (who share one weight
// snapshot).  The 512-unit layer's weight gradient arrives as n_super partial vectors (one per group of workers whose
// samples went through one product), every other tensor as the per-worker, per-block partial sums the per-worker
// reduction also reads; everything is added in a fixed order.  Blocks 0 .. FUSED_W1_BLOCKS - 1 take the float4 columns of
// the big tensor, the rest 32 small outputs each: warp w of eight adds the partial sums of workers w, w + 8, ... in four sums
// taken in turn (lane = output, so a warp's loads are consecutive), then the four and the warps' sums are added in pairs: no
// sum is longer than those of one lane in 32 were when a warp shared an output.
constexpr int FUSED_W1_VEC = HID * FLAT / 4;                                 // 200,704 float4
constexpr int FUSED_W1_BLOCKS = (FUSED_W1_VEC + 255) / 256;                  // 784
constexpr int FUSED_SMALL = C2_GRAD + C1_GRAD + (NCLS * HID + HID + NCLS) + (P_PAD - P);
constexpr int FUSED_SMALL_BLOCKS = (FUSED_SMALL + 31) / 32;
__global__ void __launch_bounds__(256) fused_finish(GradStepArgs a, WorkerTable wt, Workspace ws, const float* __restrict__ super_part,
                                                    int n_super, float* __restrict__ grad_sum, int n_chunks, int seg_len1,
                                                    int n_chunks2, int seg_len) {
  __shared__ float warp_sum[8][32];
  pdl_enter();
  const int b = a.b, split = fc2_split(a.W, b);
  if (blockIdx.x < FUSED_W1_BLOCKS) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= FUSED_W1_VEC) return;
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int g0 = 0; g0 < n_super; g0 += 8) {
      float4 v[8];
#pragma unroll
      for (int g = 0; g < 8; ++g)
        v[g] = g0 + g < n_super ? reinterpret_cast<const float4*>(super_part + (int64_t)(g0 + g) * P_PAD + OFF_F1W)[i] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int g = 0; g < 8; ++g) { t.x += v[g].x; t.y += v[g].y; t.z += v[g].z; t.w += v[g].w; }
    }
    reinterpret_cast<float4*>(grad_sum + OFF_F1W)[i] = t;
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int o = (blockIdx.x - FUSED_W1_BLOCKS) * 32 + lane;
  if (blockIdx.x == FUSED_W1_BLOCKS && threadIdx.x < a.W)        // the per-worker losses ride along (W <= 256)
    a.loss[wt.src[threadIdx.x]] = sum_slots(ws.partf + (int64_t)threadIdx.x * split * FC_PART + NCLS * HID + HID + NCLS, split, FC_PART) * (1.0f / (float)b);
  auto sum_workers = [&](auto worker_sum) {
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    for (int s = warp; s < a.W; s += 32) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (s + 8 * u < a.W) v[u] += worker_sum(s + 8 * u);
    }
    return (v[0] + v[1]) + (v[2] + v[3]);
  };
  float t = 0.f;
  float* dst = nullptr;
  if (o < C2_GRAD) {
    t = sum_workers([&](int s) { return sum_slots(ws.part2 + (int64_t)s * n_chunks2 * C2_GRAD + o, used_slots(s, b, seg_len, n_chunks2), C2_GRAD); });
    dst = grad_sum + OFF_C2W + o;
  } else if (o < C2_GRAD + C1_GRAD) {
    const int oo = o - C2_GRAD;
    t = sum_workers([&](int s) { return sum_slots(ws.part1 + (int64_t)s * n_chunks * C1_GRAD + oo, used_slots(s, b, seg_len1, n_chunks), C1_GRAD); });
    dst = grad_sum + OFF_C1W + oo;
  } else if (o < C2_GRAD + C1_GRAD + NCLS * HID + HID + NCLS) {
    const int oo = o - C2_GRAD - C1_GRAD, n = a.W * split, per = (n + 7) / 8;      // all workers' slots lie end to end
    const int c0 = min(n, warp * per), c1 = min(n, c0 + per);
    t = sum_slots(ws.partf + (int64_t)c0 * FC_PART + oo, c1 - c0, FC_PART);
    dst = oo < NCLS * HID ? grad_sum + OFF_F2W + oo : (oo < NCLS * HID + HID ? grad_sum + OFF_F1B + oo - NCLS * HID : grad_sum + OFF_F2B + oo - NCLS * HID - HID);
  } else if (o < FUSED_SMALL) {
    dst = grad_sum + P + (o - C2_GRAD - C1_GRAD - NCLS * HID - HID - NCLS);      // padding: zero
  }
  warp_sum[warp][lane] = t;
  __syncthreads();
  if (warp != 0 || !dst) return;
  *dst = ((warp_sum[0][lane] + warp_sum[1][lane]) + (warp_sum[2][lane] + warp_sum[3][lane])) +
         ((warp_sum[4][lane] + warp_sum[5][lane]) + (warp_sum[6][lane] + warp_sum[7][lane]));
}

// ---- evaluation: per worker, the mean loss from the output-layer kernel's partial sums and the number of samples
// whose predicted label equals the given one (an integer count, summed in a fixed order).
__global__ void __launch_bounds__(128) eval_finish(GradStepArgs a, WorkerTable wt, Workspace ws, int32_t* __restrict__ correct) {
  __shared__ int warp_hits[4];
  const int s = blockIdx.x, src = wt.src[s], split = fc2_split(a.W, a.b);
  int hits = 0;
  pdl_enter();
  for (int i = threadIdx.x; i < a.b; i += 128) {
    const int64_t r = (int64_t)src * a.b + i;
    hits += a.argmax[r] == a.y[r] ? 1 : 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hits += __shfl_xor_sync(0xffffffffu, hits, o);
  if ((threadIdx.x & 31) == 0) warp_hits[threadIdx.x >> 5] = hits;
  __syncthreads();
  if (threadIdx.x == 0) {
    correct[src] = warp_hits[0] + warp_hits[1] + warp_hits[2] + warp_hits[3];
    float t = 0.f;
    for (int c = 0; c < split; ++c) t += ws.partf[((int64_t)s * split + c) * FC_PART + NCLS * HID + HID + NCLS];
    a.loss[src] = t * (1.0f / (float)a.b);
  }
}

// ---- the keep mask on its own: thread e/4 draws the four words of elements 4*(e/4) .. +3.
__global__ void __launch_bounds__(256) dropout_mask(uint64_t seed, uint32_t worker, uint64_t step, int n_quads,
                                                    uint32_t thresh, uchar4* __restrict__ keep) {
  int q = blockIdx.x * 256 + threadIdx.x;
  if (q >= n_quads) return;
  uint4 r = philox4x32_10(make_uint4((uint32_t)q, worker, (uint32_t)step, (uint32_t)(step >> 32)),
                          make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
  keep[q] = make_uchar4(r.x >= thresh, r.y >= thresh, r.z >= thresh, r.w >= thresh);
}

}  // namespace

#define TIMED(id, launch) do { if (prof) prof->begin(id, st); launch; if (prof) prof->end(st); } while (0)

int launch_dropout_mask(uint64_t seed, uint32_t worker, uint64_t step, int b, uint32_t thresh,
                        uint8_t* keep, cudaStream_t st, Profiler* prof) {
  int n_quads = b * HID / 4;
  TIMED(K_DROPOUT_MASK, (dropout_mask<<<(n_quads + 255) / 256, 256, 0, st>>>(seed, worker, step, n_quads, thresh,
                                                                            reinterpret_cast<uchar4*>(keep))));
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

// Samples of a block follow one another, so blocks take fewer of them while all blocks fit on the chip (eight per SM):
// at 2 x 8 the forward kernel went from 22 to 10 us and the filter-gradient kernel from 19 to 13, at 16 x 64 from 26 to
// 19 and from 33 to 19 (~6 us of event overhead included).
static int samples_per_block(int rows, int least, int most) {
  int spb = least;
  while (spb < most && (rows + spb - 1) / spb > 8 * g_sm_count) spb *= 2;
  return spb;
}
static void launch_conv1_fwd(bool with_w1, const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  const int spb = samples_per_block(a.W * a.b, 1, CONV1_SPB);
  const int w1_units = with_w1 ? W1_UNITS : 0, chunks = (a.b + spb - 1) / spb, more = (gt.n_groups * (BANK3_UNITS + w1_units) + chunks - 1) / chunks;
  TIMED(K_CONV1_FWD, launch_pdl_if(!a.after_wait, conv1_fwd, dim3(chunks, a.W + more), CONV1_THREADS, 0, st, a, wt, gt, ws, spb, w1_units, conv2_fwd_x3_taps()));
}

// Evaluation pass: the forward kernels of the grad step with the dropout switched off, then the per-worker loss and hit
// count.  FP32 path: there is no side stream here for the pieces of W1, and a launch of their own costs more than spare blocks of conv1_fwd
// (us per pass, own launch / spare blocks: 1 x 1 27.9 / 25.0, 2 x 8 29.8 / 25.5, 16 x 8 32.0 / 28.6, 80 x 125 354 / 349).
int launch_eval(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, int32_t* correct,
                cudaStream_t st, Profiler* prof) {
  int launches = 0;
  if (a.precision != 0) {
    if (!a.skip_prep_w1) launches += launch_prep_w1(gt, ws, st, prof);
    if (launch_conv1_fwd_planes(true, a, wt, gt, ws, st, prof) < 0) return -1;
    launch_conv2_fwd_tc5(true, a, wt, gt, ws, st, prof);
    const int n = launch_fc1_fwd_tc5(a, wt, gt, ws, st, prof);
    if (n < 0) return -1;
    launches += 2 + n;
  } else {
    launch_conv1_fwd(true, a, wt, gt, ws, st, prof);
    launch_conv2_fwd_x3(a, gt, ws, st, prof);
    if (launch_fc1_fwd_x3(a, wt, gt, ws, st, prof, false) < 0) return -1;
    launches += 3;
  }
  launch_output_layer(true, a, wt, gt, ws, st, prof);
  TIMED(K_EVAL_FINISH, launch_pdl(eval_finish, dim3(a.W), 128, 0, st, a, wt, ws, correct));
  launches += 2;
  return cudaGetLastError() == cudaSuccess ? launches : -1;
}

// Launch order of one grad step.  On the tensor-core path the copies of the dense layer's weights are made on a
// side stream while the convolutions run; on both paths the backward pass forks (FP32 path, us per tick with no side stream / the second
// only / both: 2 x 8 75 / 66 / 67, 8 x 16 94 / 79 / 82, 8 x 64 135 / 122 / 116, 16 x 64 171 / 166 / 160, 32 x 64 263 / 259 / 252, 128 x 128 1,546 / 1,544 /
// 1,551: the branches fill each other's last waves): once the output
// layer's backward has produced da1, the dense layer's per-worker weight gradient (bound by its 3.2 MB
// per worker of writes) runs on a side stream next to the input-gradient chain, and once dp2 exists the
// second convolution's filter gradient runs on another side stream next to its input gradient and the
// first convolution's backward (tensor-core path: at some numbers of rows only, by the rule below).  Everything joins before the final reduction.
int launch_grad_step(const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws,
                     cudaStream_t st, const SideStreams& side, Profiler* prof, const SummedStep* sum) {
  const bool tc = a.precision != 0;
  // one output of the final reduction per thread while the blocks are few: 8.6 against 10.7 us at 8 and 16 workers; four from
  // 64 workers on: 12.7 against 14.1 us at 128
  const int red_per_block = a.W >= 64 ? 1024 : 256;
  const int spb1b = samples_per_block(a.W * a.b, CONV_SPB, CONV1B_SPB);      // at least as many as the partial-sum slots allow
  const int n_chunks1b = (a.b + spb1b - 1) / spb1b;
  int launches = 0, n_chunks2 = 0, seg_len = 0;
  // Summed step: the 512-unit layer's weight gradient is taken over groups of workers at once ("super-workers" of
  // W / n_super workers: their samples are consecutive rows, so the product only sees a longer batch) and written to
  // n_super partial vectors instead of one vector per worker.
  GradStepArgs a_dw = a;
  WorkerTable wt_dw = wt;
  if (sum) {
    a_dw.W = sum->n_super;
    a_dw.b = a.b * (a.W / sum->n_super);
    for (int g = 0; g < sum->n_super; ++g) wt_dw.grad[g] = sum->super_part + (int64_t)g * P_PAD;
  }
  if (tc) {
    // The second convolution's filter gradient has a stream of its own only while its blocks are few but its chain of samples
    // counts; from 512 rows on it and the input gradient fill the chip one after the other and the fork and join only cost, at
    // up to 64 rows the host's event calls cost more than the overlap gives.  us per tick, side stream / in line: 2 x 8 60 / 56,
    // 4 x 32 61 / 62, 5 x 37 80 / 82, 8 x 64 83.2 / 82.3, 16 x 64 107 / 105, 32 x 64 171 / 168, 64 x 32 241 / 239, 128 x 128 687 / 681.
    const bool own_stream = side.s2 && a.W * a.b > 64 && a.W * a.b < 512;
    cudaStream_t s1 = side.s1 ? side.s1 : st, s2 = own_stream ? side.s2 : st;
    // the copies of W1 are not needed before the dense layer: they are made next to the convolutions
    if (!a.skip_prep_w1) {
      if (side.s1) { cudaEventRecord(side.fork1, st); cudaStreamWaitEvent(s1, side.fork1, 0); }
      launches += launch_prep_w1(gt, ws, s1, prof);
      if (side.s1) cudaEventRecord(side.join1, s1);
    }
    if (launch_conv1_fwd_planes(false, a, wt, gt, ws, st, prof) < 0) return -1;
    launch_conv2_fwd_tc5(false, a, wt, gt, ws, st, prof);
    if (!a.skip_prep_w1 && side.s1) cudaStreamWaitEvent(st, side.join1, 0);
    int n = launch_fc1_fwd_tc5(a, wt, gt, ws, st, prof, side.s1 && !a.skip_prep_w1);
    if (n < 0) return -1;
    launches += 2 + n;
    launch_output_layer(false, a, wt, gt, ws, st, prof);
    launches += 1;
    if (side.s1) { cudaEventRecord(side.fork1, st); cudaStreamWaitEvent(s1, side.fork1, 0); }
    n = sum ? launch_fc1_dw_tc5(a_dw, wt_dw, gt, ws, s1, prof) : launch_fc1_dw_tc5(a, wt, gt, ws, s1, prof);
    if (n < 0) return -1;
    launches += n;
    if (side.s1) cudaEventRecord(side.join1, s1);
    n = launch_fc1_dx_tc5(a, wt, gt, ws, st, prof);
    if (n < 0) return -1;
    launches += n;
    if (own_stream) { cudaEventRecord(side.fork2, st); cudaStreamWaitEvent(s2, side.fork2, 0); }
    n_chunks2 = launch_conv2_dw_tc5(a, wt, ws, s2, prof, &seg_len, !own_stream);
    if (own_stream) cudaEventRecord(side.join2, s2);
    launch_conv2_dx_tc5(a, wt, gt, ws, st, prof);
    int seg_len1 = 0;
    const int n_chunks1t = launch_conv1_dw_tc5(a, wt, ws, st, prof, &seg_len1);
    if (n_chunks1t < 0) return -1;
    if (side.s1) cudaStreamWaitEvent(st, side.join1, 0);
    if (own_stream) cudaStreamWaitEvent(st, side.join2, 0);
    if (sum) TIMED(K_CONV_GRAD_REDUCE, (fused_finish<<<dim3(FUSED_W1_BLOCKS + FUSED_SMALL_BLOCKS), 256, 0, st>>>(a, wt, ws, sum->super_part, sum->n_super, sum->grad_sum, n_chunks1t, seg_len1, n_chunks2, seg_len)));
    else TIMED(K_CONV_GRAD_REDUCE, (conv_grad_reduce<<<dim3(a.W, (RED_OUTPUTS + red_per_block - 1) / red_per_block), 256, 0, st>>>(a, wt, ws, red_per_block, n_chunks1t, seg_len1, n_chunks2, seg_len)));
    launches += 4;
  } else {
    cudaStream_t s1 = side.s1 ? side.s1 : st, s2 = side.s2 ? side.s2 : st;
    // the pieces of W1 are made next to the convolutions
    if (side.s1) { cudaEventRecord(side.fork1, st); cudaStreamWaitEvent(s1, side.fork1, 0); }
    launch_prep_w1_x3(gt, ws, s1, prof);
    if (side.s1) cudaEventRecord(side.join1, s1);
    launch_conv1_fwd(false, a, wt, gt, ws, st, prof);
    launch_conv2_fwd_x3(a, gt, ws, st, prof);
    if (side.s1) cudaStreamWaitEvent(st, side.join1, 0);
    if (launch_fc1_fwd_x3(a, wt, gt, ws, st, prof, side.s1 != nullptr) < 0) return -1;
    launch_output_layer(false, a, wt, gt, ws, st, prof);
    if (side.s1) { cudaEventRecord(side.fork1, st); cudaStreamWaitEvent(s1, side.fork1, 0); }
    if (launch_fc1_dw_x3(sum ? a_dw : a, sum ? wt_dw : wt, gt, ws, s1, prof) < 0) return -1;
    if (side.s1) cudaEventRecord(side.join1, s1);
    if (launch_fc1_dx_x3(a, wt, gt, ws, st, prof) < 0) return -1;
    if (side.s2) { cudaEventRecord(side.fork2, st); cudaStreamWaitEvent(s2, side.fork2, 0); }
    n_chunks2 = launch_conv2_dw_x3(a, ws, s2, prof, &seg_len);
    if (side.s2) cudaEventRecord(side.join2, s2);
    launch_conv2_dx_x3(a, gt, ws, st, prof);
    TIMED(K_CONV1_BWD, launch_pdl(conv1_bwd, dim3(n_chunks1b, a.W), CONV1_THREADS, 0, st, a, wt, ws, spb1b, n_chunks1b));
    if (side.s1) cudaStreamWaitEvent(st, side.join1, 0);
    if (side.s2) cudaStreamWaitEvent(st, side.join2, 0);
    if (sum) TIMED(K_CONV_GRAD_REDUCE, (fused_finish<<<dim3(FUSED_W1_BLOCKS + FUSED_SMALL_BLOCKS), 256, 0, st>>>(a, wt, ws, sum->super_part, sum->n_super, sum->grad_sum, n_chunks1b, 0, n_chunks2, seg_len)));
    else TIMED(K_CONV_GRAD_REDUCE, (conv_grad_reduce<<<dim3(a.W, (RED_OUTPUTS + red_per_block - 1) / red_per_block), 256, 0, st>>>(a, wt, ws, red_per_block, n_chunks1b, 0, n_chunks2, seg_len)));
    launches = 11;
  }
  return cudaGetLastError() == cudaSuccess ? launches : -1;
}

}  // namespace psk
