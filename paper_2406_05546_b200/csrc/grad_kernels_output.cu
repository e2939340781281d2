// The output layer (512 -> 10) of both paths, FP32: logits, softmax cross-entropy, argmax, and the backward pass down to the
// gradient with respect to the 512-unit layer's pre-activation, with the layer's weight / bias gradients and the 512-unit
// layer's bias gradient as partial sums of the block.
//
// fc2_split(W, b) blocks of 16 warps per worker, each with its share of the worker's samples.  Per chunk of up to 128 of
// them: first four samples per warp at a time (a lane owns 16 hidden units; the 40 partial logits are summed over the
// lanes by an exchange that halves what a lane carries at every step), the logits' gradients going to shared memory; then
// thread = hidden unit, its ten weights and ten gradient sums in registers, walks over the chunk's samples: from a sample's
// activation and its ten logits gradients it takes both the unit's pre-activation gradient and its share of the sums, so
// the weights are read from shared memory once per pass of four samples and nothing but the activations is read again.
//
// Measured (B200, ~6 us of event overhead included; before: one block per worker, pre-activation gradients written by the
// first part and read back by the second): 14.5 -> 9 us at 2 x 8, 21.5 -> 10.7 at 8 x 64, 37 -> 33 at 128 x 128 (two blocks
// per worker).  One and two samples per warp instead of four, at twice the blocks per SM: 10.5 / 10.7 / 41 and 10.7 / 11.8 / 35.
#include "bf16x3.cuh"
#include "device_common.cuh"
#include "kernels.h"

namespace psk {

namespace {

constexpr int FC2_THREADS = 512;
constexpr int NS = 4, LPS = 32 / NS;   // samples per warp and pass, lanes that end up with a sample
constexpr int DZ_CHUNK = 128;      // samples whose logits gradients are held in shared memory at a time
constexpr int W2T_PITCH = 12;      // 48-byte rows: 16-byte loads of consecutive rows fall on distinct banks
static_assert(FC2_THREADS == HID, "thread = hidden unit");

template <bool EVAL, bool FP32>
__global__ void __launch_bounds__(FC2_THREADS, 1) output_layer(GradStepArgs a, WorkerTable wt, GroupTable gt, Workspace ws) {
  __shared__ __align__(16) float w2t[HID][W2T_PITCH];     // w2t[j][c] = W2[c][j]; the two pad columns are zero
  __shared__ __align__(16) float dzs[DZ_CHUNK][W2T_PITCH];   // logits gradients of a chunk of samples
  __shared__ float b2[NCLS];
  __shared__ float warp_loss[FC2_THREADS / 32];
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* theta = group_theta(wt, gt, s);
  const int src = wt.src[s];
  const int per = (a.b + gridDim.y - 1) / gridDim.y;
  const int i_lo = min(a.b, (int)blockIdx.y * per), i_hi = min(a.b, i_lo + per);
#pragma unroll
  for (int c = 0; c < NCLS; ++c) w2t[tid][c] = theta[OFF_F2W + c * HID + tid];
  w2t[tid][NCLS] = w2t[tid][NCLS + 1] = 0.f;
  if (tid < NCLS) b2[tid] = theta[OFF_F2B + tid];
  __syncthreads();
  pdl_enter();
  const float scale = 1.0f / (1.0f - a.drop_p);
  const float inv_b = 1.0f / (float)a.b;
  const bool hi16 = lane & 16, hi8 = lane & 8, hi4 = lane & 4;
  const int my_u = lane / LPS, sub = lane % LPS;          // after the reduction a lane works for sample my_u of the pass
  float loss_acc = 0.f, gb1 = 0.f, gb2 = 0.f;
  u64 gwk[NCLS / 2];
#pragma unroll
  for (int k = 0; k < NCLS / 2; ++k) gwk[k] = 0ull;
  for (int c0 = i_lo; c0 < i_hi; c0 += DZ_CHUNK) {
    const int n = min(DZ_CHUNK, i_hi - c0);
    for (int i0 = NS * warp; i0 < n; i0 += NS * (FC2_THREADS / 32)) {
      const int n_s = min(NS, n - i0);                    // warp-uniform
      const bool mine = my_u < n_s;
      // the weights are re-read from shared memory on every pass: 160 of them per lane would not fit in the
      // registers of a 512-thread block, so their address is made to look pass-dependent
      uint32_t opaque_zero;
      asm volatile("mov.u32 %0, 0;" : "=r"(opaque_zero));
      const float4* w2p = reinterpret_cast<const float4*>(&w2t[0][0] + opaque_zero);
      const int64_t row0 = (int64_t)s * a.b + c0 + i0;
      // the label is asked for now: by the time the softmax needs it, it has arrived
      int label = a.y[(int64_t)src * a.b + c0 + i0 + (mine ? my_u : 0)];
      // classes in pairs, one packed multiply-add per pair: zp[u][k] = logits 2k and 2k + 1 of sample u
      u64 zp[NS][NCLS / 2];
#pragma unroll
      for (int u = 0; u < NS; ++u)
#pragma unroll
        for (int k = 0; k < NCLS / 2; ++k) zp[u][k] = 0ull;
#pragma unroll
      for (int h = 0; h < 2; ++h) {                       // the units in two halves, to bound the registers
        float dv[NS][8];
#pragma unroll
        for (int u = 0; u < NS; ++u)
#pragma unroll
          for (int t = 0; t < 8; ++t) dv[u][t] = ws.d[(row0 + (u < n_s ? u : 0)) * HID + lane + 32 * (8 * h + t)];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const float4* wr = w2p + (lane + 32 * (8 * h + t)) * (W2T_PITCH / 4);
          const float4 q0 = wr[0], q1 = wr[1], q2 = wr[2];
          const u64 wk[NCLS / 2] = {pack2(q0.x, q0.y), pack2(q0.z, q0.w), pack2(q1.x, q1.y), pack2(q1.z, q1.w), pack2(q2.x, q2.y)};
#pragma unroll
          for (int u = 0; u < NS; ++u) {
            const u64 du = pack2(dv[u][t], dv[u][t]);
#pragma unroll
            for (int k = 0; k < NCLS / 2; ++k) zp[u][k] = ffma2(wk[k], du, zp[u][k]);
          }
        }
      }
      // Sum over the lanes.  Each exchange halves what a lane goes on with: after the first two a lane holds the ten
      // partial logits of sample lane / 8 only, after the third five of them; two plain exchanges finish the sums and a
      // last one brings the two halves of the classes together.
      float v[NS * NCLS];
#pragma unroll
      for (int u = 0; u < NS; ++u)
#pragma unroll
        for (int k = 0; k < NCLS / 2; ++k) unpack2(zp[u][k], v[u * NCLS + 2 * k], v[u * NCLS + 2 * k + 1]);
      float w20[2 * NCLS], x10[NCLS], y5[NCLS / 2], z[NCLS];
#pragma unroll
      for (int k = 0; k < 2 * NCLS; ++k) {
        const float keep = hi16 ? v[2 * NCLS + k] : v[k], send = hi16 ? v[k] : v[2 * NCLS + k];
        w20[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
      }
#pragma unroll
      for (int k = 0; k < NCLS; ++k) {
        const float keep = hi8 ? w20[NCLS + k] : w20[k], send = hi8 ? w20[k] : w20[NCLS + k];
        x10[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
      }
#pragma unroll
      for (int k = 0; k < NCLS / 2; ++k) {
        const float keep = hi4 ? x10[NCLS / 2 + k] : x10[k], send = hi4 ? x10[k] : x10[NCLS / 2 + k];
        y5[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
        y5[k] += __shfl_xor_sync(0xffffffffu, y5[k], 2);
        y5[k] += __shfl_xor_sync(0xffffffffu, y5[k], 1);
      }
#pragma unroll
      for (int k = 0; k < NCLS / 2; ++k) {
        const float other = __shfl_xor_sync(0xffffffffu, y5[k], 4);
        z[k] = (hi4 ? other : y5[k]) + b2[k];
        z[NCLS / 2 + k] = (hi4 ? y5[k] : other) + b2[NCLS / 2 + k];
      }
      // softmax, loss and logits gradient of the lane's sample (the eight lanes of a sample do the same work)
      float zmax = z[0];
      int am = 0;
#pragma unroll
      for (int c = 1; c < NCLS; ++c)
        if (z[c] > zmax) { zmax = z[c]; am = c; }
      float ez[NCLS], se = 0.f;
#pragma unroll
      for (int c = 0; c < NCLS; ++c) { ez[c] = expf(z[c] - zmax); se += ez[c]; }
      const float lse = zmax + logf(se), inv_se = 1.0f / se;
      if (label < 0 || label >= NCLS) {
        if (mine && sub == 0) atomicOr(ws.status, STATUS_BAD_LABEL);
        label = 0;
      }
      float zy = 0.f, e0 = 0.f, e1 = 0.f;                 // lane sub of a sample stores elements 2 sub and 2 sub + 1 of its padded row
#pragma unroll
      for (int c = 0; c < NCLS; ++c) {
        if (c == label) zy = z[c];
        const float g = (ez[c] * inv_se - (c == label ? 1.f : 0.f)) * inv_b;     // softmax from the exponentials already taken
        if (sub == c / 2) { if (c & 1) e1 = g; else e0 = g; }
      }
      if (mine) {
        loss_acc += lse - zy;
        if (sub == 0) a.argmax[(int64_t)src * a.b + c0 + i0 + my_u] = am;
        if (!EVAL && sub < W2T_PITCH / 2) *reinterpret_cast<float2*>(&dzs[i0 + my_u][2 * sub]) = make_float2(e0, e1);
      }
    }
    if (EVAL) continue;
    __syncthreads();
    u64 wk[NCLS / 2];
    {
      const float4* wr = reinterpret_cast<const float4*>(&w2t[tid][0]);
      const float4 q0 = wr[0], q1 = wr[1], q2 = wr[2];
      wk[0] = pack2(q0.x, q0.y); wk[1] = pack2(q0.z, q0.w); wk[2] = pack2(q1.x, q1.y); wk[3] = pack2(q1.z, q1.w); wk[4] = pack2(q2.x, q2.y);
    }
    const float* dp = ws.d + ((int64_t)s * a.b + c0) * HID + tid;
    float* da1p = ws.da1 + ((int64_t)s * a.b + c0) * HID + tid;
    uint16_t* da1x = ws.da1x + ((int64_t)s * a.b + c0) * HID + tid;
    const int64_t piece = (int64_t)a.W * a.b * HID;
    constexpr int U = 8;                                  // activations in flight per thread
    for (int i0 = 0; i0 < n; i0 += U) {
      float dval[U];
#pragma unroll
      for (int u = 0; u < U; ++u) dval[u] = dp[(int64_t)min(i0 + u, n - 1) * HID];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (i0 + u >= n) break;
        const float4* zr = reinterpret_cast<const float4*>(&dzs[i0 + u][0]);
        const float4 z0 = zr[0], z1 = zr[1], z2 = zr[2];
        const u64 dzk[NCLS / 2] = {pack2(z0.x, z0.y), pack2(z0.z, z0.w), pack2(z1.x, z1.y), pack2(z1.z, z1.w), pack2(z2.x, z2.y)};
        const u64 dd = pack2(dval[u], dval[u]);
        u64 e = 0ull;                                     // even classes in the low half, odd classes in the high half
#pragma unroll
        for (int k = 0; k < NCLS / 2; ++k) {
          e = ffma2(wk[k], dzk[k], e);
          gwk[k] = ffma2(dzk[k], dd, gwk[k]);
        }
        float lo, hi;
        unpack2(e, lo, hi);
        float o = dval[u] > 0.f ? (lo + hi) * scale : 0.f;   // the unit passed ReLU and dropout
        // it feeds tensor-core products only: as TF32, or (FP32 path) as three BF16 pieces
        if (!FP32) {
          o = round_tf32(o);
          da1p[(int64_t)(i0 + u) * HID] = o;
        } else {
          const Bf16x3 sp = split3(o, 0.f);
#pragma unroll
          for (int p = 0; p < PIECES; ++p) da1x[p * piece + (int64_t)(i0 + u) * HID] = (uint16_t)sp.p[p];
        }
        gb1 += o;
      }
    }
    if (tid < NCLS)
      for (int i = 0; i < n; ++i) gb2 += dzs[i][tid];
    __syncthreads();                                      // the chunk's gradients have been read
  }
  // the eight lanes of a sample hold the same loss: one of each, in lane order
  float loss = __shfl_sync(0xffffffffu, loss_acc, 0);
#pragma unroll
  for (int u = 1; u < NS; ++u) loss += __shfl_sync(0xffffffffu, loss_acc, u * LPS);
  if (lane == 0) warp_loss[warp] = loss;
  __syncthreads();
  float* part = ws.partf + ((int64_t)s * gridDim.y + blockIdx.y) * FC_PART;
  if (tid == 0) {
    float t = 0.f;
    for (int w = 0; w < FC2_THREADS / 32; ++w) t += warp_loss[w];
    part[NCLS * HID + HID + NCLS] = t;
  }
  if constexpr (!EVAL) {
#pragma unroll
    for (int k = 0; k < NCLS / 2; ++k) {
      float lo, hi;
      unpack2(gwk[k], lo, hi);
      part[2 * k * HID + tid] = lo;
      part[(2 * k + 1) * HID + tid] = hi;
    }
    part[NCLS * HID + tid] = gb1;
    if (tid < NCLS) part[NCLS * HID + HID + tid] = gb2;
  }
}

}  // namespace

#define TIMED(id, launch) do { if (prof) prof->begin(id, st); launch; if (prof) prof->end(st); } while (0)

void launch_output_layer(bool eval, const GradStepArgs& a, const WorkerTable& wt, const GroupTable& gt, const Workspace& ws, cudaStream_t st, Profiler* prof) {
  const dim3 grid(a.W, fc2_split(a.W, a.b));
  if (eval) TIMED(K_FC2_FWD_BWD, launch_pdl(output_layer<true, false>, dim3(grid), FC2_THREADS, 0, st, a, wt, gt, ws));
  else if (a.precision == 0) TIMED(K_FC2_FWD_BWD, launch_pdl(output_layer<false, true>, dim3(grid), FC2_THREADS, 0, st, a, wt, gt, ws));
  else TIMED(K_FC2_FWD_BWD, launch_pdl(output_layer<false, false>, dim3(grid), FC2_THREADS, 0, st, a, wt, gt, ws));
}

}  // namespace psk
