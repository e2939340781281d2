// Single precision on the tensor cores: every FP32 operand as the sum of three BF16 pieces.
//
// x = h + m + l with h = bf16(x), m = bf16(x - h), l = bf16(x - h - m): 3 x 8 significant bits hold all 24 of a float, and BF16 has
// its exponent range (only below 2^-110 do the last pieces run out of it).  Of the nine products of two such sums six are
// taken: h h, then h m, m h, h l, m m, l h, which are 2^-8 and 2^-16 of it; the three left out (m l, l m, l l) are 2^-24 of it and
// of either sign.  A product of two BF16 values is exact in the tensor core.
//
// What limits the precision is its accumulator, which drops the low bits of every sum (it does not round to nearest), so that
// the error grows with the number of instructions added up, always towards zero.  Hence
//   - the five small products have an accumulator of their own, where the same loss is 2^-8 as large, and
//   - the leading products are added up over a bounded number of values of k, then added to a sum in registers, which rounds: 64 in the
//     dense layer's forward product, 128 in its gradients, 80 and 64 in the second convolution forward (in two accumulators), 96 in its input
//     gradient, 224 in its filter gradient.  (The small products over all of k: their loss is 2^-8 of it.)
// Error relative to float64, 2-norm, of 512 x 128 sums over K = 1,600 of N(0, 1) x N(0, 0.05^2), rectified: one chain of fused
// multiply-adds 4.9e-7; all six products in one accumulator 1.0e-5; two accumulators 1.1e-6; leading products over 512,
// 256, 128 and 64 values of k at a time 2.9e-7, 1.5e-7, 1.1e-7 and 1.1e-7.  K = 512: chain 2.6e-7, 128 at a time 0.8e-7;
// K = 128: 1.4e-7 and 0.8e-7.
//
// Infinities and NaN: such a value is its own first piece and the others are zero, and where the sum of the leading products is not
// finite the small ones (infinity times a piece of either sign) are left out, so that it is what FP32 gives.
#pragma once
#include <stdint.h>

#include "device_common.cuh"
#include "kernels.h"

namespace psk {

constexpr int PIECES = 3;

// The part of a leading sum that truncation takes from it on average: (n - 1) / 2 times 1.3e-8 to 1.6e-8 for n instructions, whatever the
// operands' signs (partial sums grow towards the whole in the mean).  It is the same for every sample, so that it does not average out in a
// sum over samples as rounding does.  In the forward products, on which every gradient depends, sums are short (4 or 5 instructions) and the
// weights' last pieces are larger by as much (the dense layer's input gradient, of 8 instructions, has the same operand).  Mean relative
// error without / with both: second convolution -6.4e-8 (one sum of 9 instructions) / -0.04e-8, dense layer -4.7e-8 (8) / -0.01e-8, its input
// gradient -4.3e-8 / -2.1e-8.  fc2.w of a summed step of 128 x 128 against float64, 2-norm: 2.1e-7 / 0.8e-7, as multiply-adds that round give it.
constexpr float LOST_CONV2 = 2.35e-8f, LOST_FC1 = 2.3e-8f;

struct Bf16x3 { uint32_t p[PIECES]; };      // two values: BF16 pairs, the first value in the low halves

// One value that rounds past the largest BF16, or none: the piece is cut off instead.
__device__ __forceinline__ void split3_huge(float x, uint32_t shift, Bf16x3& o) {
  const uint32_t u = __float_as_uint(x);
  const bool finite = (u & 0x7F800000u) != 0x7F800000u;
  const uint32_t h = (u >> 16) | (x != x ? 0x40u : 0u);
  const float r = finite ? x - __uint_as_float(u & 0xFFFF0000u) : 0.f;
  const uint32_t m = bf16_bits(r), l = bf16_bits(r - __uint_as_float(m << 16));
  const uint32_t keep = 0xFFFF0000u >> shift;
  o.p[0] = (o.p[0] & keep) | (h << shift);
  o.p[1] = (o.p[1] & keep) | (m << shift);
  o.p[2] = (o.p[2] & keep) | (l << shift);
}

// more: the part of a value that is added to its last piece
__device__ __forceinline__ Bf16x3 split3(float a, float b, float more = 0.f) {
  constexpr float MOST = 3.3895313892515355e38f;      // the largest BF16
  Bf16x3 o;
  o.p[0] = bf16_pair(a, b);
  float ra = a - __uint_as_float(o.p[0] << 16), rb = b - __uint_as_float(o.p[0] & 0xFFFF0000u);
  o.p[1] = bf16_pair(ra, rb);
  ra -= __uint_as_float(o.p[1] << 16);
  rb -= __uint_as_float(o.p[1] & 0xFFFF0000u);
  if (more != 0.f) {
    ra = fmaf(a, more, ra);
    rb = fmaf(b, more, rb);
  }
  o.p[2] = bf16_pair(ra, rb);
  if (!(fabsf(a) <= MOST)) split3_huge(a, 0, o);
  if (!(fabsf(b) <= MOST)) split3_huge(b, 16, o);
  return o;
}

// Eight values of the dense layer's weights, i onwards, of weight group g: [group][piece][512][1568].
constexpr int W1_ELEMS = HID * FLAT;
__device__ __forceinline__ void split_w1(const float* __restrict__ theta, uint16_t* __restrict__ w1x, int g, int i) {
  const float4* src = reinterpret_cast<const float4*>(theta + OFF_F1W + i);
  const float4 v0 = src[0], v1 = src[1];
  const Bf16x3 s0 = split3(v0.x, v0.y, LOST_FC1), s1 = split3(v0.z, v0.w, LOST_FC1), s2 = split3(v1.x, v1.y, LOST_FC1), s3 = split3(v1.z, v1.w, LOST_FC1);
#pragma unroll
  for (int p = 0; p < PIECES; ++p)
    *reinterpret_cast<uint4*>(w1x + ((int64_t)g * PIECES + p) * W1_ELEMS + i) = make_uint4(s0.p[p], s1.p[p], s2.p[p], s3.p[p]);
}

// The sum of the leading products with that of the small ones.
__device__ __forceinline__ float join3(float lead, float small) { return fabsf(lead) <= 3.402823466e38f ? lead + small : lead; }

}  // namespace psk
