// Kernel 1, the arithmetic: block-Hadamard rotation + MXFP4 quantisation of one MX group (paper Sec. 4.3 Eq. 1, Sec. 4.1),
// shared by the kernels that move the bytes (rotate_quantize_direct.cuh, rotate_quantize_wide.cuh, rotate_quantize_global.cuh
// and the split-K GEMM).
//
//  * A thread owns whole MX groups (32 consecutive channels of one row): the 5 butterfly stages of the 32-point
//    Walsh-Hadamard transform run entirely in registers.
//  * fp32 arithmetic in exactly this order: butterflies (a+b, a-b) with ascending stride, one
//    multiply by c = fp32(1/sqrt(block)), amax over the group, shared exponent
//    E = max(expfield(amax) - 2, 0) - 127, r = y * 2^-E, round-to-nearest-even to E2M1 with
//    saturation.  The multiply by c and the exact scaling by 2^-E are merged into one multiply by
//    c*2^-E whenever that product is a normal fp32 (bit-identical result); otherwise the two
//    multiplies are done separately.
#pragma once

#include <cuda_fp16.h>

#include "bro_common.cuh"

namespace bro {
namespace rq {

// Zero tiled scales for the rows that pad the last block of 128, by all threads of a grid; whole lines by each warp.
__device__ __forceinline__ void clear_padding(void* scales, int64_t M, int64_t kblocks, int64_t thread, int64_t threads) {
  const int rest = (int)(M & 127);
  if (rest == 0) return;
  uint32_t* block = reinterpret_cast<uint32_t*>(scales) + (M >> 7) * kblocks * 128;
  for (int64_t i = thread; i < kblocks * 128; i += threads) {
    const int slot = (int)(i & 127), row = ((slot & 3) << 5) | (slot >> 2);
    if (row >= rest) block[i] = 0u;
  }
}

// x diag(s): flip the bf16 sign bits of a 16-byte chunk of x where the sign vector is negative.
// One three-input logic operation per 32-bit word (x ^ (s & 0x80008000)); exact.
__device__ __forceinline__ uint4 apply_signs(uint4 q, uint4 sg) {
  q.x ^= sg.x & 0x80008000u;
  q.y ^= sg.y & 0x80008000u;
  q.z ^= sg.z & 0x80008000u;
  q.w ^= sg.w & 0x80008000u;
  return q;
}

__device__ __forceinline__ uint32_t pack_e2m1x8(float r0, float r1, float r2, float r3, float r4,
                                                float r5, float r6, float r7) {
  // cvt.rn.satfinite.e2m1x2.f32 d, a, b : a -> bits 4..7, b -> bits 0..3 (nearest even, +-6 clamp)
  uint32_t w;
  asm("{ .reg .b8 b0, b1, b2, b3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n\t"
      "mov.b32 %0, {b0, b1, b2, b3}; }"
      : "=r"(w)
      : "f"(r0), "f"(r1), "f"(r2), "f"(r3), "f"(r4), "f"(r5), "f"(r6), "f"(r7));
  return w;
}

// the same for 4 values, in the low 16 bits (and once more in the high ones)
__device__ __forceinline__ uint32_t pack_e2m1x4(float r0, float r1, float r2, float r3) {
  uint32_t w;
  asm("{ .reg .b8 b0, b1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
      "mov.b32 %0, {b0, b1, b0, b1}; }"
      : "=r"(w)
      : "f"(r0), "f"(r1), "f"(r2), "f"(r3));
  return w;
}

// c = fp32 nearest 1/sqrt(2^LOG2B)
template <int LOG2B>
__device__ __forceinline__ constexpr uint32_t norm_bits() {
  // even exponent: exact power of two; odd: fp32(sqrt 2) = 0x3FB504F3 scaled by a power of two
  return (LOG2B % 2 == 0) ? (uint32_t)(127 - LOG2B / 2) << 23
                          : 0x3FB504F3u - ((uint32_t)((LOG2B + 1) / 2) << 23);
}

// the same for a run-time log2b
__host__ __device__ inline uint32_t norm_bits_of(int log2b) {
  return (log2b % 2 == 0) ? (uint32_t)(127 - log2b / 2) << 23 : 0x3FB504F3u - ((uint32_t)((log2b + 1) / 2) << 23);
}

// ---- packed fp32x2 arithmetic (sm_100): one issue slot for two IEEE round-to-nearest results.
// A group's 32 values live in 16 register pairs; pair k holds elements (2k, 2k+1).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t shfl_xor2(uint64_t v, int lane_mask) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  lo = __shfl_xor_sync(0xFFFFFFFFu, lo, lane_mask);
  hi = __shfl_xor_sync(0xFFFFFFFFu, hi, lane_mask);
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}

// The two values of a word, lo and hi -> lo + hi and lo - hi.  The sum of a bf16 and an fp32 is one instruction (exact operands, one
// rounding), so the low value needs no unpacking: 16 instructions of a group's 300 less, [16384, 4096] block 32 28.7 -> 28.1 us (at the power cap
// 31.1 -> 30.2), block 128 30.6 -> 29.9, the full dimension 50.8 -> 50.0, the gated producer [4096, 14336] 45.8 -> 44.8.
__device__ __forceinline__ void stage1(uint32_t word, float& sum, float& diff) {
  const float hi = __uint_as_float(word & 0xFFFF0000u);
  asm("{ .reg .b16 l, h; mov.b32 {l, h}, %2;\n\t"
      "add.rn.f32.bf16 %0, l, %3;\n\t"
      "sub.rn.f32.bf16 %1, l, %3; }"
      : "=f"(sum), "=f"(diff)
      : "r"(word), "f"(hi));
}

// 8 bf16 (one 16-byte chunk) -> 4 pairs, fused with butterfly stage h = 1, which pairs the two
// halves of one 32-bit word: (lo, hi) -> (lo + hi, lo - hi).
__device__ __forceinline__ void unpack_stage1(const uint4& q, uint64_t* P) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float sum, diff;
    stage1(w[k], sum, diff);
    P[k] = pack2(sum, diff);
  }
}

// Butterfly stages h = 2, 4, 8, 16 on pairs (ascending stride): pair k meets pair k ^ (h/2).
__device__ __forceinline__ void fwht32_stages_2_to_16(uint64_t (&P)[16]) {
#pragma unroll
  for (int hp = 1; hp < 16; hp <<= 1) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if ((k & hp) == 0) {
        const uint64_t a = P[k], b = P[k + hp];
        P[k] = add2(a, b);
        P[k + hp] = sub2(a, b);
      }
    }
  }
}

// The same for a rotation inside the MX group (blocks of 2..16 channels: LOG2B = 1..4): the stages of
// stride 2 .. B/2 only (stage h = 1 is in unpack_stage1).
template <int LOG2B>
__device__ __forceinline__ void fwht32_stages_below(uint64_t (&P)[16]) {
  static_assert(LOG2B >= 1 && LOG2B <= 4, "blocks of 2..16");
#pragma unroll
  for (int hp = 1; hp < (1 << (LOG2B - 1)); hp <<= 1) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if ((k & hp) == 0) {
        const uint64_t a = P[k], b = P[k + hp];
        P[k] = add2(a, b);
        P[k + hp] = sub2(a, b);
      }
    }
  }
}

// ---- blocks of 64 / 128 channels: cross-lane stages that exchange HALF of each lane's values --------
// The 2 (or 4) MX groups of a block sit in neighbouring lanes.  A butterfly stage between two lanes
// needs, for every element i, a + b in one lane and a - b in the other.  Instead of every lane
// fetching all 32 partner values and producing 32 results, each lane keeps 16 of its values, sends
// the other 16, and produces BOTH the sum and the difference for the 16 elements it kept: half the
// shuffles, and the arithmetic stays on packed pairs.  Afterwards a lane holds 16 values of one output
// group and 16 values of another (two 8-byte code stores instead of one 16-byte store; the group
// maximum takes one more shuffle).
//
// So that both lanes of a pair run the same instructions on the same registers, the odd lane loads
// its 64 bytes with the two 32-byte halves exchanged (register pair k holds true pair k ^ 8): every
// lane then keeps registers 0..7 and sends registers 8..15.  Stages h = 1..8 never cross the halves;
// stage h = 16 does, and is written as two fused multiply-adds with the lane's sign s (+1 even lane,
// -1 odd lane), which yields a + b and a - b in the registers where this lane expects them:
//   P'[k]   = s * P[k]   + P[k+8]      P'[k+8] = -s * P[k+8] + P[k]
// Each is ONE rounding of the exact sum or difference (a product with +-1 is exact), i.e. bit-identical
// to the add / subtract of the contract, including the sign of an exact zero (x - y == x + (-y)).
__device__ __forceinline__ void fwht32_stages_2_to_8(uint64_t (&P)[16]) {
#pragma unroll
  for (int hp = 1; hp < 8; hp <<= 1) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if ((k & hp) == 0) {
        const uint64_t a = P[k], b = P[k + hp];
        P[k] = add2(a, b);
        P[k + hp] = sub2(a, b);
      }
    }
  }
}
__device__ __forceinline__ void stage16_halves_exchanged(uint64_t (&P)[16], uint64_t s2, uint64_t ns2) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint64_t a = P[k], b = P[k + 8];
    P[k] = fma2(a, s2, b);
    P[k + 8] = fma2(b, ns2, a);
  }
}

// amax of the 16 values held in 8 pairs (three-input maximum of absolute values, two chains).
__device__ __forceinline__ float amax_pairs8(const uint64_t (&P)[8]) {
  float m = 0.f, m2 = 0.f;
#pragma unroll
  for (int k = 0; k < 8; k += 2) {
    float lo, hi, lo2, hi2;
    unpack2(P[k], lo, hi);
    unpack2(P[k + 1], lo2, hi2);
    asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(lo), "f"(hi));
    asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m2) : "f"(lo2), "f"(hi2));
  }
  return fmaxf(m, m2);
}
// Scale byte of a group from its pre-normalisation amax, and the 16 codes of the half group in P
// (same arithmetic as quantize_group).
__device__ __forceinline__ uint32_t encode_pairs8(const uint64_t (&P)[8], float amax, uint32_t cbits, uint32_t (&w)[2]) {
  const float c = __uint_as_float(cbits);
  const uint32_t ef = __float_as_uint(__fmul_rn(amax, c)) >> 23;
  const uint32_t s = ef > 2u ? ef - 2u : 0u;
  float r[16];
  if (ef >= 27u && ef <= 250u) {
    const float c2 = __uint_as_float(cbits + ((127u - s) << 23));
    const uint64_t cc = pack2(c2, c2);
#pragma unroll
    for (int k = 0; k < 8; ++k) unpack2(mul2(P[k], cc), r[2 * k], r[2 * k + 1]);
  } else {
    const float p2 = __uint_as_float((254u - s) << 23);
    const uint64_t cc = pack2(c, c), pp = pack2(p2, p2);
#pragma unroll
    for (int k = 0; k < 8; ++k) unpack2(mul2(mul2(P[k], cc), pp), r[2 * k], r[2 * k + 1]);
  }
#pragma unroll
  for (int j = 0; j < 2; ++j)
    w[j] = pack_e2m1x8(r[8 * j], r[8 * j + 1], r[8 * j + 2], r[8 * j + 3], r[8 * j + 4], r[8 * j + 5],
                       r[8 * j + 6], r[8 * j + 7]);
  return s;
}

// A group in four neighbouring lanes, 8 values each: the lane's 8 codes, and the group's scale byte in every lane (same arithmetic as
// quantize_group).
__device__ __forceinline__ uint32_t encode_pairs4(const uint64_t (&P)[4], uint32_t cbits, uint32_t& scale) {
  float v[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) unpack2(P[k], v[2 * k], v[2 * k + 1]);
  float m = 0.f, m2 = 0.f;
  asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(v[0]), "f"(v[1]));
  asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m2) : "f"(v[2]), "f"(v[3]));
  asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(v[4]), "f"(v[5]));
  asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m2) : "f"(v[6]), "f"(v[7]));
  m = fmaxf(m, m2);
  m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, 1));
  m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, 2));
  const float c = __uint_as_float(cbits);
  const uint32_t ef = __float_as_uint(__fmul_rn(m, c)) >> 23;
  const uint32_t s = ef > 2u ? ef - 2u : 0u;
  scale = s;
  if (ef >= 27u && ef <= 250u) {
    const float c2 = __uint_as_float(cbits + ((127u - s) << 23));
    const uint64_t cc = pack2(c2, c2);
#pragma unroll
    for (int k = 0; k < 4; ++k) unpack2(mul2(P[k], cc), v[2 * k], v[2 * k + 1]);
  } else {
    const float p2 = __uint_as_float((254u - s) << 23);
    const uint64_t cc = pack2(c, c), pp = pack2(p2, p2);
#pragma unroll
    for (int k = 0; k < 4; ++k) unpack2(mul2(mul2(P[k], cc), pp), v[2 * k], v[2 * k + 1]);
  }
  return pack_e2m1x8(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
}

// The cross-lane stages of a 64- or 128-channel block on the registers described above, then the
// quantisation of the two half groups this lane ends up with.
//   lane & 1   which 16 elements of a group this lane keeps (0: elements 0..15, 1: 16..31)
//   lane & 2   (blocks of 128) which pair of groups: 0 -> groups 0 / 2 of the block, 1 -> groups 1 / 3
// Outputs: wx / sx = codes of this lane's 16 elements and scale byte of group X, wy / sy of group Y, with
//   block 64 : X = group 0, Y = group 1 of the block;   block 128 : X = group (lane>>1)&1, Y = X + 2.
// P must hold the values after stages h = 1..8 (odd lanes: halves exchanged).
template <int LOG2B>
__device__ __forceinline__ void cross_lane_split(uint64_t (&P)[16], int lane, uint32_t cbits, uint32_t (&wx)[2],
                                                 uint32_t& sx, uint32_t (&wy)[2], uint32_t& sy) {
  static_assert(LOG2B == 6 || LOG2B == 7, "blocks of 64 or 128 channels");
  const float s0 = (lane & 1) ? -1.f : 1.f;
  const uint64_t s0p = pack2(s0, s0), ns0p = pack2(-s0, -s0);
  stage16_halves_exchanged(P, s0p, ns0p);
  uint64_t X[8], Y[8];
  if (LOG2B == 6) {
    // stage h = 32 with lane ^ 1: kept K = P[0..7], received R = partner's P[8..15] (the same elements)
    //   even lane: X = K + R, Y = K - R;   odd lane: X = R + K, Y = R - K
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint64_t R = shfl_xor2(P[8 + k], 1);
      X[k] = add2(P[k], R);
      Y[k] = fma2(P[k], s0p, mul2(R, ns0p));
    }
  } else {
    // stage h = 32 with lane ^ 1, written so that lanes of the second group pair (lane & 2) get sum and
    // difference in exchanged registers: they keep the difference and send the sum in stage h = 64.
    const bool second = (lane & 2) != 0;
    const float one = 1.f;
    const uint64_t c1 = second ? s0p : pack2(one, one), c2 = second ? ns0p : pack2(one, one);
    const uint64_t c3 = second ? pack2(one, one) : s0p, c4 = second ? pack2(one, one) : ns0p;
    const float s1 = second ? -1.f : 1.f;
    const uint64_t s1p = pack2(s1, s1), ns1p = pack2(-s1, -s1);
    uint64_t U[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint64_t R = shfl_xor2(P[8 + k], 1);
      U[k] = fma2(P[k], c1, mul2(R, c2));            // kept for stage h = 64
      const uint64_t V = fma2(P[k], c3, mul2(R, c4)); // sent
      const uint64_t R2 = shfl_xor2(V, 2);
      X[k] = add2(U[k], R2);
      Y[k] = fma2(U[k], s1p, mul2(R2, ns1p));
    }
  }
  float mx = amax_pairs8(X), my = amax_pairs8(Y);
  mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
  my = fmaxf(my, __shfl_xor_sync(0xFFFFFFFFu, my, 1));
  sx = encode_pairs8(X, mx, cbits, wx);
  sy = encode_pairs8(Y, my, cbits, wy);
}

// One butterfly stage across two lanes that hold the low / high half of the pairs.
// low lane: a + b ; high lane: a - b = own * (-1) + other (exact, one rounding).
__device__ __forceinline__ void cross_lane_stage(uint64_t (&P)[16], int lane_mask, bool is_high) {
  const float sgn = is_high ? -1.f : 1.f;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    float lo, hi;
    unpack2(P[k], lo, hi);
    const float olo = __shfl_xor_sync(0xFFFFFFFFu, lo, lane_mask);
    const float ohi = __shfl_xor_sync(0xFFFFFFFFu, hi, lane_mask);
    P[k] = pack2(__fmaf_rn(lo, sgn, olo), __fmaf_rn(hi, sgn, ohi));
  }
}

// Quantise the 32 fp32 values held in P (pre-normalisation: y = v*c) of one MX group.
// Returns the scale byte; writes 4 code words.
__device__ __forceinline__ uint32_t quantize_group(const uint64_t (&P)[16], uint32_t cbits, uint32_t (&w)[4]) {
  // amax with the three-input maximum of absolute values (one instruction per pair); two
  // accumulators halve the dependent chain
  float m = 0.f, m2 = 0.f;
#pragma unroll
  for (int k = 0; k < 16; k += 2) {
    float lo, hi, lo2, hi2;
    unpack2(P[k], lo, hi);
    unpack2(P[k + 1], lo2, hi2);
    asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(lo), "f"(hi));
    asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m2) : "f"(lo2), "f"(hi2));
  }
  m = fmaxf(m, m2);
  const float c = __uint_as_float(cbits);
  // amax of y: rounding is monotonic, so max_i fl(|v_i| c) = fl(max_i |v_i| * c)
  const uint32_t ef = __float_as_uint(__fmul_rn(m, c)) >> 23;
  const uint32_t s = ef > 2u ? ef - 2u : 0u;
  float r[32];
  if (ef >= 27u && ef <= 250u) {
    // c * 2^-E is a normal fp32: one multiply, bit-identical to (v*c)*2^-E
    const float c2 = __uint_as_float(cbits + ((127u - s) << 23));
    const uint64_t cc = pack2(c2, c2);
#pragma unroll
    for (int k = 0; k < 16; ++k) unpack2(mul2(P[k], cc), r[2 * k], r[2 * k + 1]);
  } else {
    const float p2 = __uint_as_float((254u - s) << 23);   // 2^-E, E = s - 127
    const uint64_t cc = pack2(c, c), pp = pack2(p2, p2);
#pragma unroll
    for (int k = 0; k < 16; ++k) unpack2(mul2(mul2(P[k], cc), pp), r[2 * k], r[2 * k + 1]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
    w[j] = pack_e2m1x8(r[8 * j], r[8 * j + 1], r[8 * j + 2], r[8 * j + 3], r[8 * j + 4], r[8 * j + 5],
                       r[8 * j + 6], r[8 * j + 7]);
  return s;
}

// Scale byte only: the E8M0 byte quantize_group would assign to the group held in P.
constexpr int kFormatScaleOnly = 4;     // `format` value of the analysis kernels that selects this output
__device__ __forceinline__ uint32_t group_scale_byte(const uint64_t (&P)[16], uint32_t cbits) {
  float m = 0.f, m2 = 0.f;
#pragma unroll
  for (int k = 0; k < 16; k += 2) {
    float lo, hi, lo2, hi2;
    unpack2(P[k], lo, hi);
    unpack2(P[k + 1], lo2, hi2);
    asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(lo), "f"(hi));
    asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(m2) : "f"(lo2), "f"(hi2));
  }
  m = fmaxf(m, m2);
  const uint32_t ef = __float_as_uint(__fmul_rn(m, __uint_as_float(cbits))) >> 23;
  return ef > 2u ? ef - 2u : 0u;
}

// Quantisation error of one group of 32 (paper Sec. 4.1-4.2: block-level error under the shared
// scale; Sec. 3.2 / Fig. 2-3 for the formats compared): mean over the group of (y - deq(Q(y)))^2 with
// y = v * c the rotated values.  `format`: 0 MXFP4 (E2M1, scale 2^E, E = floor(log2 amax) - 2),
// 1 BFP4 (E2M1, scale fp16(amax / 6)), 2 MXINT4 (k/4 with |k| <= 7, scale 2^floor(log2 amax)),
// 3 BINT4 (|k| <= 7, scale fp16(amax / 7)); round to nearest even, saturating.
// E2M1 codes come from the same conversion instruction as in quantize_group and are decoded again
// in hardware (e2m1x2 -> f16x2).  With a power-of-two scale the difference is exact in the scaled
// domain; with an fp16 scale it is one fused multiply-add.  Squares and their sum are fp32.
__device__ __forceinline__ float group_error_any(const uint64_t (&P)[16], uint32_t cbits, int format) {
  const float c = __uint_as_float(cbits);
  const uint64_t cc = pack2(c, c);
  float y[32];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    unpack2(mul2(P[k], cc), y[2 * k], y[2 * k + 1]);
    y[2 * k] = fabsf(y[2 * k]);             // every format is symmetric: work on magnitudes
    y[2 * k + 1] = fabsf(y[2 * k + 1]);
  }
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 32; ++i) m = fmaxf(m, y[i]);
  const uint32_t ef = __float_as_uint(m) >> 23;
  auto e2m1 = [](float r0, float r1, float& q0, float& q1) {
    uint32_t h;
    asm("{ .reg .b8 b; cvt.rn.satfinite.e2m1x2.f32 b, %2, %1; cvt.rn.f16x2.e2m1x2 %0, b; }" : "=r"(h) : "f"(r0), "f"(r1));
    q0 = __half2float(__ushort_as_half((unsigned short)(h & 0xFFFFu)));
    q1 = __half2float(__ushort_as_half((unsigned short)(h >> 16)));
  };
  float acc = 0.f;
  if (format == 0 || format == 2) {
    const uint32_t s = format == 0 ? (ef > 2u ? ef - 2u : 0u) : ef;
    const float inv = __uint_as_float(s <= 253u ? ((254u - s) << 23) : 0x00400000u);   // 2^-E, E = s - 127 (2^-127 is subnormal)
    const float pe = __uint_as_float(s >= 1u ? (s << 23) : 0x00400000u);    // 2^E (2^-127 is subnormal)
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
      const float r0 = __fmul_rn(y[i], inv), r1 = __fmul_rn(y[i + 1], inv);
      float q0, q1;
      if (format == 0) {
        e2m1(r0, r1, q0, q1);
      } else {
        q0 = 0.25f * (float)min(__float2int_rn(__fmul_rn(r0, 4.f)), 7);
        q1 = 0.25f * (float)min(__float2int_rn(__fmul_rn(r1, 4.f)), 7);
      }
      const float d0 = __fsub_rn(r0, q0), d1 = __fsub_rn(r1, q1);
      acc = __fadd_rn(acc, __fmul_rn(d0, d0));
      acc = __fadd_rn(acc, __fmul_rn(d1, d1));
    }
    return __fmul_rn(__fmul_rn(__fmul_rn(acc, 0.03125f), pe), pe);
  }
  // fp16 scale: the fp32 quotient amax / qmax rounded to nearest-even fp16, saturating
  float sc;
  {
    const float quot = __fdiv_rn(m, format == 1 ? 6.f : 7.f);
    unsigned short hb;
    asm("cvt.rn.satfinite.f16.f32 %0, %1;" : "=h"(hb) : "f"(quot));
    sc = __half2float(__ushort_as_half(hb));
  }
#pragma unroll
  for (int i = 0; i < 32; i += 2) {
    float q0 = 0.f, q1 = 0.f;
    if (sc != 0.f) {
      const float r0 = __fdiv_rn(y[i], sc), r1 = __fdiv_rn(y[i + 1], sc);
      if (format == 1) {
        e2m1(r0, r1, q0, q1);
      } else {
        q0 = (float)min(__float2int_rn(r0), 7);
        q1 = (float)min(__float2int_rn(r1), 7);
      }
    }
    const float d0 = __fmaf_rn(-q0, sc, y[i]), d1 = __fmaf_rn(-q1, sc, y[i + 1]);
    acc = __fadd_rn(acc, __fmul_rn(d0, d0));
    acc = __fadd_rn(acc, __fmul_rn(d1, d1));
  }
  return __fmul_rn(acc, 0.03125f);
}

// The same with a short form for MXFP4 away from the ends of the exponent range, on packed pairs: c * 2^-E in one multiply
// as in quantize_group, squares added by fused multiply-adds in two chains of pairs.  ([16384, 4096], block 32: 37 -> 31 us.)
__device__ __forceinline__ float group_error(const uint64_t (&P)[16], uint32_t cbits, int format) {
  const float c = __uint_as_float(cbits);
  if (format == 0) {
    float m = 0.f, m2 = 0.f;
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
      float a, b, a2, b2;
      unpack2(P[k], a, b);
      unpack2(P[k + 1], a2, b2);
      asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(a), "f"(b));
      asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(m2) : "f"(a2), "f"(b2));
    }
    asm("max.NaN.f32 %0, %0, %1;" : "+f"(m) : "f"(m2));
    if (m == 0.f) return 0.f;             // (zeros need not wait for the general form)
    const uint32_t ef = __float_as_uint(__fmul_rn(m, c)) >> 23;
    if (ef >= 27u && ef <= 250u) {
      const float c2 = __uint_as_float(cbits + ((129u - ef) << 23)), pe = __uint_as_float((ef - 2u) << 23);
      const uint64_t cc = pack2(c2, c2);
      uint64_t acc[2] = {0ull, 0ull};
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const uint64_t r = mul2(P[k], cc);
        float r0, r1;
        unpack2(r, r0, r1);
        uint32_t h;
        asm("{ .reg .b8 b; cvt.rn.satfinite.e2m1x2.f32 b, %2, %1; cvt.rn.f16x2.e2m1x2 %0, b; }" : "=r"(h) : "f"(r0), "f"(r1));
        const uint64_t d = sub2(r, pack2(__half2float(__ushort_as_half((unsigned short)(h & 0xFFFFu))),
                                         __half2float(__ushort_as_half((unsigned short)(h >> 16)))));
        acc[k & 1] = fma2(d, d, acc[k & 1]);
      }
      float s0, s1;
      unpack2(add2(acc[0], acc[1]), s0, s1);
      return __fmul_rn(__fmul_rn(__fmul_rn(__fadd_rn(s0, s1), 0.03125f), pe), pe);
    }
  }
  return group_error_any(P, cbits, format);
}

}  // namespace rq
}  // namespace bro
