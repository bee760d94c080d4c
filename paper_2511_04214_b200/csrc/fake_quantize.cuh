// Simulated ("fake") quantisation: rotate, quantise to one of the compared 4-bit formats, dequantise.
// The paper evaluates every method this way (Sec. 3.1, experimental setup: MX quantisation is
// simulated, no native FP4 GEMM is run), and its format study (Sec. 3.2 / Fig. 2, Sec. 4.1 / Fig. 3)
// compares MXFP4 with BFP4, MXINT4 and BINT4 on the same tensors.  This kernel gives those tensors at
// full bandwidth: out[m, k] = deq(Q_format((x R)[m, :]))_k as fp32, in the rotated domain.
//
// One thread owns one MX group of 32 channels (64 bytes of bf16), a warp 32 consecutive groups of a
// row; the rotation is the same fixed-order fp32 butterfly as in the quantising kernels (stages of
// stride 1..16 in registers, stride 32 / 64 through one / two shuffles for blocks of 64 / 128), or
// none at all (LOG2B = 0: the identity, "before rotation"), or a rotation inside the MX group
// (LOG2B = 1..4: blocks of 2..16 channels — the paper's Sec. 5.2 sweeps the rotation dimension below as
// well as above the MX group), which simply stops the butterfly early.  Every dequantised value is exactly
// representable in fp32 (a 3-bit element times a power of two or an 11-bit fp16 scale), so the result
// can be compared bit for bit with an evaluation in higher precision.
//
// An analysis path: 2 bytes read and 4 written per element.  A thread's 128 output bytes go through a
// per-warp shared-memory buffer (16-byte pieces XOR-swizzled with the lane, conflict-free both ways) so
// that every store instruction of the warp writes 512 contiguous bytes of the row.
#pragma once

#include <type_traits>

#include "bro_common.cuh"
#include "rotate_quantize.cuh"

namespace bro {
namespace fq {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// The 32 values of one group (P holds the un-normalised butterfly output, y = P * c) dequantised
// under `format`: 0 MXFP4 (E2M1, scale 2^E, E = floor(log2 amax) - 2), 1 BFP4 (E2M1, scale
// fp16(amax / 6)), 2 MXINT4 (k / 4, |k| <= 7, scale 2^E, E = floor(log2 amax)), 3 BINT4 (|k| <= 7,
// scale fp16(amax / 7)).  Decisions are taken exactly as in rq::group_error: magnitudes scaled by an
// exact power of two, or divided by the fp16 scale in fp32, then rounded to nearest even, saturating.
__device__ __forceinline__ void group_dequant_any(const uint64_t (&P)[16], uint32_t cbits, int format, float (&out)[32]) {
  const float c = __uint_as_float(cbits);
  const uint64_t cc = rq::pack2(c, c);
  float y[32];
#pragma unroll
  for (int k = 0; k < 16; ++k) rq::unpack2(rq::mul2(P[k], cc), y[2 * k], y[2 * k + 1]);
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 32; ++i) m = fmaxf(m, fabsf(y[i]));
  const uint32_t ef = __float_as_uint(m) >> 23;
  auto e2m1 = [](float r0, float r1, float& q0, float& q1) {
    uint32_t h;
    asm("{ .reg .b8 b; cvt.rn.satfinite.e2m1x2.f32 b, %2, %1; cvt.rn.f16x2.e2m1x2 %0, b; }" : "=r"(h) : "f"(r0), "f"(r1));
    q0 = __half2float(__ushort_as_half((unsigned short)(h & 0xFFFFu)));
    q1 = __half2float(__ushort_as_half((unsigned short)(h >> 16)));
  };
  if (format == 0 || format == 2) {
    const uint32_t s = format == 0 ? (ef > 2u ? ef - 2u : 0u) : ef;
    // 2^-E and 2^E with E = s - 127 (2^-127 is a subnormal)
    const float inv = __uint_as_float(s <= 253u ? ((254u - s) << 23) : 0x00400000u);
    const float pe = __uint_as_float(s >= 1u ? (s << 23) : 0x00400000u);
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
      const float r0 = __fmul_rn(fabsf(y[i]), inv), r1 = __fmul_rn(fabsf(y[i + 1]), inv);
      float q0, q1;
      if (format == 0) {
        e2m1(r0, r1, q0, q1);
      } else {
        q0 = 0.25f * (float)min(__float2int_rn(__fmul_rn(r0, 4.f)), 7);
        q1 = 0.25f * (float)min(__float2int_rn(__fmul_rn(r1, 4.f)), 7);
      }
      out[i] = copysignf(__fmul_rn(q0, pe), y[i]);
      out[i + 1] = copysignf(__fmul_rn(q1, pe), y[i + 1]);
    }
    return;
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
    if (sc == 0.f) {                 // (a scale that rounds to zero gives an all-zero group)
      out[i] = 0.f;
      out[i + 1] = 0.f;
      continue;
    }
    const float r0 = __fdiv_rn(fabsf(y[i]), sc), r1 = __fdiv_rn(fabsf(y[i + 1]), sc);
    float q0, q1;
    if (format == 1) {
      e2m1(r0, r1, q0, q1);
    } else {
      q0 = (float)min(__float2int_rn(r0), 7);
      q1 = (float)min(__float2int_rn(r1), 7);
    }
    out[i] = copysignf(__fmul_rn(q0, sc), y[i]);
    out[i + 1] = copysignf(__fmul_rn(q1, sc), y[i + 1]);
  }
}

// ---- the same on packed pairs, for ordinary numbers ------------------------------------------------------------
// What made the forms above slow were IEEE divisions (25 instructions an element) and conversions to integers and back at a
// quarter of the issue rate.  Here a quotient by the group's (row's) scale is q = y * inv, corrected once by its exact remainder,
// q + (y - q sc) inv, with inv the correctly rounded 1 / sc: correctly rounded, by Markstein ("Computation of elementary
// functions on the IBM RISC System/6000 processor", 1990), as long as nothing leaves the normal range; quotients so small that
// their remainder is subnormal round to the element 0 either way.  Integers come from adding and subtracting 1.5 * 2^23 (nearest,
// ties to even) after clamping, which commutes with rounding.  Every step rounds as in the forms above, so the values are the same
// bits.  Groups that hold an infinity or a NaN (amax_nan then is one too) and the ends of the exponent range take the forms
// above.  They are rare, but a warp that holds one waits for both forms; so groups of zeros have an answer of their own,
// and the lanes beyond the end of a row compute nothing.
// [8192, 4096], block 32, general forms -> these: BFP4 56 -> 36 us, BINT4 58 -> 36, MXFP4 39 -> 36, MXINT4 41 -> 36.
__device__ __forceinline__ float amax_nan(const uint64_t (&Y)[16]) {
  float m = 0.f, m2 = 0.f;
#pragma unroll
  for (int k = 0; k < 16; k += 2) {
    float a, b, c, d;
    rq::unpack2(Y[k], a, b);
    rq::unpack2(Y[k + 1], c, d);
    asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(a), "f"(b));
    asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(m2) : "f"(c), "f"(d));
  }
  asm("max.NaN.f32 %0, %0, %1;" : "+f"(m) : "f"(m2));
  return m;
}
__device__ __forceinline__ uint64_t both(float v) { return rq::pack2(v, v); }
__device__ __forceinline__ uint64_t quotient2(uint64_t y, uint64_t inv, uint64_t minus_sc) {
  const uint64_t q = rq::mul2(y, inv);
  return rq::fma2(rq::fma2(minus_sc, q, y), inv, q);
}
// clamp to [lo, hi] (whole numbers), round to a whole number
__device__ __forceinline__ uint64_t round2(uint64_t r, float lo, float hi) {
  float a, b;
  rq::unpack2(r, a, b);
  const uint64_t magic = both(12582912.0f);
  return rq::sub2(rq::add2(rq::pack2(fminf(fmaxf(a, lo), hi), fminf(fmaxf(b, lo), hi)), magic), magic);
}
__device__ __forceinline__ uint64_t e2m1_value2(uint64_t r) {          // nearest E2M1 values
  float a, b;
  rq::unpack2(r, a, b);
  uint32_t h;
  asm("{ .reg .b8 b; cvt.rn.satfinite.e2m1x2.f32 b, %2, %1; cvt.rn.f16x2.e2m1x2 %0, b; }" : "=r"(h) : "f"(a), "f"(b));
  return rq::pack2(__half2float(__ushort_as_half((unsigned short)(h & 0xFFFFu))), __half2float(__ushort_as_half((unsigned short)(h >> 16))));
}
// out = |v| with the sign of y (a value that rounds to zero keeps its sign)
__device__ __forceinline__ void signed_out(uint64_t v, uint64_t y, float& o0, float& o1) {
  float v0, v1, y0, y1;
  rq::unpack2(v, v0, v1);
  rq::unpack2(y, y0, y1);
  o0 = copysignf(v0, y0);
  o1 = copysignf(v1, y1);
}

// The rare path as a call, so that the ordinary one keeps its registers.  (Not for the full-dimension rotation, which has
// no registers to spare around a call: there the short forms and their call made every mode of its kernel 15 to 50 %
// slower, quantisation to codes included, and it keeps the forms above.)
__device__ __noinline__ void group_dequant_rare(const uint64_t (&P)[16], uint32_t cbits, int format, float (&out)[32]) {
  group_dequant_any(P, cbits, format, out);
}

__device__ __forceinline__ void group_dequant(const uint64_t (&P)[16], uint32_t cbits, int format, float (&out)[32]) {
  uint64_t Y[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) Y[k] = rq::mul2(P[k], both(__uint_as_float(cbits)));
  const float m = amax_nan(Y);
  if (m == 0.f) {              // zeros, which keep their signs under a power-of-two scale
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      rq::unpack2(Y[k], out[2 * k], out[2 * k + 1]);
      if (format & 1) out[2 * k] = out[2 * k + 1] = 0.f;
    }
    return;
  }
  const uint32_t ef = __float_as_uint(m) >> 23;
  // 2^-125 and up, finite; the fp16 scales not zero
  float sc = 0.f, inv = 0.f;
  if (format & 1) {
    unsigned short hb;
    asm("cvt.rn.satfinite.f16.f32 %0, %1;" : "=h"(hb) : "f"(__fdiv_rn(m, format == 1 ? 6.f : 7.f)));
    sc = __half2float(__ushort_as_half(hb));
    inv = __frcp_rn(sc);
  }
  if (ef < 8u || ef > 250u || ((format & 1) && sc == 0.f)) {          // (a NaN has exponent field 255)
    uint64_t Q[16];                            // (copies: only this path keeps arrays in memory)
    float o[32];
#pragma unroll
    for (int k = 0; k < 16; ++k) Q[k] = P[k];
    group_dequant_rare(Q, cbits, format, o);
#pragma unroll
    for (int i = 0; i < 32; ++i) out[i] = o[i];
    return;
  }
  if (format == 0) {
    const float s_inv = __uint_as_float((256u - ef) << 23), s = __uint_as_float((ef - 2u) << 23);   // 2^-E and 2^E, E = ef - 2 - 127
#pragma unroll
    for (int k = 0; k < 16; ++k) signed_out(rq::mul2(e2m1_value2(rq::mul2(Y[k], both(s_inv))), both(s)), Y[k], out[2 * k], out[2 * k + 1]);
  } else if (format == 2) {
    const float s_inv = __uint_as_float((256u - ef) << 23), s = __uint_as_float((ef - 2u) << 23);   // 4 * 2^-E and 2^E / 4, E = ef - 127
#pragma unroll
    for (int k = 0; k < 16; ++k) signed_out(rq::mul2(round2(rq::mul2(Y[k], both(s_inv)), -7.f, 7.f), both(s)), Y[k], out[2 * k], out[2 * k + 1]);
  } else if (format == 1) {
#pragma unroll
    for (int k = 0; k < 16; ++k) signed_out(rq::mul2(e2m1_value2(quotient2(Y[k], both(inv), both(-sc))), both(sc)), Y[k], out[2 * k], out[2 * k + 1]);
  } else {
#pragma unroll
    for (int k = 0; k < 16; ++k) signed_out(rq::mul2(round2(quotient2(Y[k], both(inv), both(-sc)), -7.f, 7.f), both(sc)), Y[k], out[2 * k], out[2 * k + 1]);
  }
}

__device__ __forceinline__ void store_group(float* dst, const float (&out)[32]) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
    reinterpret_cast<float4*>(dst)[j] = make_float4(out[4 * j], out[4 * j + 1], out[4 * j + 2], out[4 * j + 3]);
}

// ---- INT4 with one scale per ROW (Sec. 3.2 / Fig. 2: per-channel symmetric weights, per-token asymmetric
// activations).  Two passes over the input: the first leaves the row's range in `rowstats`, the second
// quantises with it.  rowstats[2 * row] = bits of max(-min(row), 0), rowstats[2 * row + 1] = bits of
// max(max(row), 0): both are non-negative floats, which order like their bit patterns, so an integer
// atomicMax onto zero-initialised words is an exact, order-independent reduction.
constexpr int kFormatRowSym = 4, kFormatRowAsym = 5, kFormatNone = 6;

// The extremes of y = v c are those of v times c (rounding is monotonic): three-input minimum and maximum, a quarter of the
// instructions of a multiply and two comparisons per value.
__device__ __forceinline__ void group_range(const uint64_t (&P)[16], uint32_t cbits, float& neglo, float& hi) {
  float lo = 0.f, lo2 = 0.f, up = 0.f, up2 = 0.f;          // (0 belongs to every range)
#pragma unroll
  for (int k = 0; k < 16; k += 2) {
    float a, b, a2, b2;
    rq::unpack2(P[k], a, b);
    rq::unpack2(P[k + 1], a2, b2);
    asm("max.f32 %0, %0, %1, %2;" : "+f"(up) : "f"(a), "f"(b));
    asm("min.f32 %0, %0, %1, %2;" : "+f"(lo) : "f"(a), "f"(b));
    asm("max.f32 %0, %0, %1, %2;" : "+f"(up2) : "f"(a2), "f"(b2));
    asm("min.f32 %0, %0, %1, %2;" : "+f"(lo2) : "f"(a2), "f"(b2));
  }
  const float c = __uint_as_float(cbits);
  hi = __fmul_rn(fabsf(fmaxf(up, up2)), c);                // (fabsf: a zero of either sign is +0)
  neglo = __fmul_rn(fabsf(fminf(lo, lo2)), c);
}

// The 32 values of a group under the row's scale.  Symmetric: |k| <= 7, scale fp16(amax / 7).  Asymmetric:
// codes 0..15 over [lo, hi] (the range always contains zero): scale fp16((hi - lo) / 15), zero point
// z = rint(-lo / scale) (at most 15), q = clamp(rint(y / scale) + z, 0, 15), value (q - z) scale.  Quotients
// are IEEE fp32 divisions; every result is an integer of at most 5 bits times an fp16 number, exact in fp32.
__device__ __forceinline__ void row_dequant_any(const uint64_t (&P)[16], uint32_t cbits, bool asym, float neglo, float hi,
                                                float (&out)[32]) {
  const float c = __uint_as_float(cbits);
  const uint64_t cc = rq::pack2(c, c);
  float y[32];
#pragma unroll
  for (int k = 0; k < 16; ++k) rq::unpack2(rq::mul2(P[k], cc), y[2 * k], y[2 * k + 1]);
  const float quot = asym ? __fdiv_rn(__fadd_rn(hi, neglo), 15.f) : __fdiv_rn(fmaxf(hi, neglo), 7.f);
  unsigned short hb;
  asm("cvt.rn.satfinite.f16.f32 %0, %1;" : "=h"(hb) : "f"(quot));
  const float sc = __half2float(__ushort_as_half(hb));
  if (sc == 0.f) {                  // (a scale that rounds to zero gives an all-zero row)
#pragma unroll
    for (int i = 0; i < 32; ++i) out[i] = 0.f;
    return;
  }
  if (!asym) {
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const float q = (float)min(__float2int_rn(__fdiv_rn(fabsf(y[i]), sc)), 7);
      out[i] = copysignf(__fmul_rn(q, sc), y[i]);
    }
    return;
  }
  const int z = min(__float2int_rn(__fdiv_rn(neglo, sc)), 15);
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    int q = __float2int_rn(__fdiv_rn(y[i], sc));
    q = max(-16, min(q, 31)) + z;
    q = max(0, min(q, 15));
    out[i] = __fmul_rn((float)(q - z), sc);
  }
}

__device__ __noinline__ void row_dequant_rare(const uint64_t (&P)[16], uint32_t cbits, bool asym, float neglo, float hi,
                                              float (&out)[32]) {
  row_dequant_any(P, cbits, asym, neglo, hi, out);
}
__device__ __forceinline__ void row_dequant(const uint64_t (&P)[16], uint32_t cbits, bool asym, float neglo, float hi,
                                            float (&out)[32]) {
  uint64_t Y[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) Y[k] = rq::mul2(P[k], both(__uint_as_float(cbits)));
  const float m = amax_nan(Y);
  unsigned short hb;
  asm("cvt.rn.satfinite.f16.f32 %0, %1;" : "=h"(hb) : "f"(asym ? __fdiv_rn(__fadd_rn(hi, neglo), 15.f) : __fdiv_rn(fmaxf(hi, neglo), 7.f)));
  const float sc = __half2float(__ushort_as_half(hb));
  if (!(m < 1e38f) || sc == 0.f) {
    uint64_t Q[16];
    float o[32];
#pragma unroll
    for (int k = 0; k < 16; ++k) Q[k] = P[k];
    row_dequant_rare(Q, cbits, asym, neglo, hi, o);
#pragma unroll
    for (int i = 0; i < 32; ++i) out[i] = o[i];
    return;
  }
  const float inv = __frcp_rn(sc);
  if (asym) {        // clamp(rint(y / sc) + z, 0, 15) - z is rint(y / sc) clamped to [-z, 15 - z]
    const float z = (float)min(__float2int_rn(__fdiv_rn(neglo, sc)), 15);
#pragma unroll
    for (int k = 0; k < 16; ++k)
      rq::unpack2(rq::mul2(round2(quotient2(Y[k], both(inv), both(-sc)), -z, 15.f - z), both(sc)), out[2 * k], out[2 * k + 1]);
  } else {
#pragma unroll
    for (int k = 0; k < 16; ++k)
      signed_out(rq::mul2(round2(quotient2(Y[k], both(inv), both(-sc)), -7.f, 7.f), both(sc)), Y[k], out[2 * k], out[2 * k + 1]);
  }
}

struct Params {
  const uint16_t* x;
  int64_t M, K, ldx;
  const uint16_t* signs;        // [K] bf16 +-1 (kernels with SIGNS) or nullptr
  uint32_t* rowstats;           // [M, 2] the row ranges (see group_range): written when deq == nullptr and
                                // neither statistic is asked for, read by the per-row formats unless `whole_rows`
  float* deq;                   // [M, K] fp32, row stride ldd — or nullptr, and then one of:
  int64_t ldd;
  float* mse;                   //   [M, K/32] per-group quantisation error (rq::group_error)
  uint8_t* scale_bytes;         //   [M, K/32] E8M0 byte of each group (rq::group_scale_byte)
  int format;
  int chunks_per_row;           // ceil((K / 32) / 32): one task = one warp, 32 groups of a row
  int whole_rows;               // per-row formats of rows of at most kWarps chunks: a CTA holds whole rows
};

// Longest row of which a CTA holds every chunk in one of its warps' registers.
constexpr int64_t kWholeRowK = (int64_t)kWarps * 1024;

// LOG2B = 0: no rotation; 1..4: blocks of 2..16 inside the group; 5, 6, 7: blocks of 32, 64, 128.
// The loads of a warp's next task are issued before the current one is computed.  With `whole_rows` the warps of a CTA
// take whole rows together, exchange the chunks' ranges through shared memory and need neither the first pass nor
// its second read of x ([8192, 4096], block 32, both formats: 78 us in two passes, now 45).  Without the early loads the
// formats take 43 instead of 36 us there, with eight CTAs an SM that come and go 44.
// MODE: what the kernel writes, one of the three below.  (One kernel for all: the plain rotation paid for the registers and
// the length of the formats' code, [1000, 2176], block 32, 3.9 -> 4.4 us, now 3.6; MXFP4 there 5.4 -> 4.9.)
enum : int { kStatistics, kRotation, kFormats };
template <int LOG2B, bool SIGNS, int MODE>
__global__ void __launch_bounds__(kThreads, 2) fake_quantize_kernel(const Params p) {
  __shared__ __align__(16) float sbuf[kWarps][32 * 32];      // 4 KiB per warp
  __shared__ float2 ranges[2][kWarps];                       // whole_rows: the chunks' ranges, two rounds
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* wbuf = sbuf[warp];
  const int ng = (int)(p.K >> 5);
  constexpr uint32_t cbits = LOG2B == 0 ? 0x3F800000u : rq::norm_bits<(LOG2B == 0 ? 5 : LOG2B)>();
  const bool whole_rows = MODE == kFormats && p.whole_rows != 0;
  // row and chunk of this warp's first task, and the step to its next one
  const int c = p.chunks_per_row;
  const int rows_at_once = whole_rows ? kWarps / c : 0;
  int64_t row, step_row;
  int chunk, step_chunk = 0;
  if (whole_rows) {
    const int r = warp / c;
    chunk = warp - r * c;
    row = r < rows_at_once ? (int64_t)blockIdx.x * rows_at_once + r : p.M;      // (left-over warps only keep step)
    step_row = (int64_t)gridDim.x * rows_at_once;
  } else {
    const uint32_t task = blockIdx.x * kWarps + (uint32_t)warp, num_warps = gridDim.x * kWarps;      // (of the grid: 32 bits)
    row = task / (uint32_t)c;
    chunk = (int)(task % (uint32_t)c);
    step_row = num_warps / (uint32_t)c;
    step_chunk = (int)(num_warps % (uint32_t)c);
  }
  griddep_wait();
  griddep_launch_dependents();
  auto load = [&](int64_t r, int ch, uint4 (&v)[4]) {
    const int g = ch * 32 + lane;
    const bool in = r < p.M && g < ng;
    const uint4* src = reinterpret_cast<const uint4*>(p.x + (in ? r : 0) * p.ldx + (int64_t)(in ? g : 0) * 32);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = in ? __ldg(src + j) : make_uint4(0u, 0u, 0u, 0u);
  };
  uint4 cur[4], nxt[4];
  load(row, chunk, cur);
  int round = 0;
  for (int64_t base = whole_rows ? (int64_t)blockIdx.x * rows_at_once : row; base < p.M; ++round) {
    const int g = chunk * 32 + lane;
    const bool live = row < p.M && g < ng;         // (K is a multiple of the block, so the lanes of a block share `live`)
    int64_t nrow = row + step_row;
    int nchunk = chunk + step_chunk;
    if (nchunk >= c) { nchunk -= c; ++nrow; }
    load(nrow, nchunk, nxt);
    uint64_t P[16];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint4 q = cur[j];
      if (SIGNS && live) q = rq::apply_signs(q, __ldg(reinterpret_cast<const uint4*>(p.signs + (int64_t)g * 32) + j));
      if (LOG2B == 0) {
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          P[4 * j + k] = rq::pack2(__uint_as_float(w[k] << 16), __uint_as_float(w[k] & 0xFFFF0000u));
      } else {
        rq::unpack_stage1(q, P + 4 * j);
      }
    }
    if (LOG2B >= 5) rq::fwht32_stages_2_to_16(P);
    if (LOG2B >= 2 && LOG2B <= 4) rq::fwht32_stages_below<(LOG2B >= 2 && LOG2B <= 4) ? LOG2B : 2>(P);
    if (LOG2B >= 6) rq::cross_lane_stage(P, 1, (lane & 1) != 0);
    if (LOG2B >= 7) rq::cross_lane_stage(P, 2, (lane & 2) != 0);
    float neglo = 0.f, hi = 0.f;
    if (whole_rows || (MODE == kStatistics && !p.mse && !p.scale_bytes)) {     // the range of this chunk
      group_range(P, cbits, neglo, hi);
      // All 32 lanes hold groups of the same row; dead lanes hold zeros.  Non-negative floats order like their bits.  (In the pass over long
      // rows, which does little else, shuffles: [4096, 14336] block 128 117 us with the reduction, 112 with them.)
      if constexpr (MODE == kStatistics) {
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
          neglo = fmaxf(neglo, __shfl_xor_sync(0xFFFFFFFFu, neglo, d));
          hi = fmaxf(hi, __shfl_xor_sync(0xFFFFFFFFu, hi, d));
        }
      } else {
        neglo = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(neglo)));
        hi = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(hi)));
      }
    }
    if (whole_rows) {
      if (lane == 0) ranges[round & 1][warp] = make_float2(neglo, hi);
      __syncthreads();                             // (the buffers alternate: the round before was read before this barrier)
      for (int w = warp - chunk; w < warp - chunk + c && w < kWarps; ++w) {
        const float2 o = ranges[round & 1][w];
        neglo = fmaxf(neglo, o.x);
        hi = fmaxf(hi, o.y);
      }
    }
    if (MODE == kStatistics) {
      if (p.mse) {                                 // the statistics only
        if (live) p.mse[row * ng + g] = rq::group_error(P, cbits, p.format);
      } else if (p.scale_bytes) {
        const uint32_t sb = rq::group_scale_byte(P, cbits);
        if (live) p.scale_bytes[row * ng + g] = (uint8_t)sb;
      } else if (lane == 0) {                      // first pass of the per-row formats: the row's range
        atomicMax(p.rowstats + 2 * row, __float_as_uint(neglo));
        atomicMax(p.rowstats + 2 * row + 1, __float_as_uint(hi));
      }
    } else if (row < p.M) {
      float out[32];
      if (!live) {                                 // (beyond the row's end: these lanes must not take the rare path)
#pragma unroll
        for (int i = 0; i < 32; ++i) out[i] = 0.f;
      } else if (MODE == kRotation) {              // the rotation itself
        const uint64_t cc = rq::pack2(__uint_as_float(cbits), __uint_as_float(cbits));
#pragma unroll
        for (int k = 0; k < 16; ++k) rq::unpack2(rq::mul2(P[k], cc), out[2 * k], out[2 * k + 1]);
      } else if (p.format >= kFormatRowSym) {
        if (!whole_rows) {
          neglo = __uint_as_float(__ldcg(p.rowstats + 2 * row));
          hi = __uint_as_float(__ldcg(p.rowstats + 2 * row + 1));
        }
        row_dequant(P, cbits, p.format == kFormatRowAsym, neglo, hi, out);
      } else {
        group_dequant(P, cbits, p.format, out);
      }
      // lane l -> buffer row l (128 bytes), piece j at position j ^ (l & 7)
      __syncwarp();                                // the previous task's reads of the buffer are done
#pragma unroll
      for (int j = 0; j < 8; ++j)
        *reinterpret_cast<float4*>(wbuf + lane * 32 + ((j ^ (lane & 7)) << 2)) =
            make_float4(out[4 * j], out[4 * j + 1], out[4 * j + 2], out[4 * j + 3]);
      __syncwarp();
      // instruction i writes groups 4i .. 4i+3 of the chunk: 8 lanes per group, 16 bytes each
      const int gbase = g - lane;
      float* rowp = p.deq + row * p.ldd + (int64_t)gbase * 32;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = i * 4 + (lane >> 3), q = lane & 7;
        const float4 v = *reinterpret_cast<const float4*>(wbuf + r * 32 + ((q ^ (r & 7)) << 2));
        if (gbase + r < ng) *reinterpret_cast<float4*>(rowp + r * 32 + q * 4) = v;
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) cur[j] = nxt[j];
    row = nrow;
    chunk = nchunk;
    base = whole_rows ? base + step_row : row;
  }
}

// block: 1 (identity), 2, 4, 8, 16, 32, 64 or 128.  Exactly one of deq / mse / scale_bytes is set — or none of
// them and rowstats, for the first pass of the per-row formats; deq and a per-row format without rowstats take K up to
// kWholeRowK in one pass.
inline bro_status launch(const void* x, int64_t M, int64_t K, int64_t ldx, int block, const void* signs, int format,
                         float* deq, int64_t ldd, float* mse, uint8_t* scale_bytes, int sm_count, cudaStream_t st,
                         uint32_t* rowstats = nullptr) {
  Params p;
  p.rowstats = rowstats;
  p.x = static_cast<const uint16_t*>(x);
  p.M = M; p.K = K; p.ldx = ldx;
  p.signs = static_cast<const uint16_t*>(signs);
  p.deq = deq;
  p.ldd = ldd;
  p.mse = mse;
  p.scale_bytes = scale_bytes;
  p.format = format;
  p.chunks_per_row = (int)((K / 32 + 31) / 32);
  p.whole_rows = (deq && format >= kFormatRowSym && format != kFormatNone && !rowstats) ? 1 : 0;
  const int rows_at_once = kWarps / p.chunks_per_row;
  const int64_t want = p.whole_rows ? (M + rows_at_once - 1) / rows_at_once : (M * p.chunks_per_row + kWarps - 1) / kWarps;
  // (the formats: two CTAs an SM that stay.  The statistics need fewer registers and fit three: BFP4 error of [8192, 4096],
  // block 1, 44 us with two and 32 with three, MXFP4 of [1000, 2176] 3.3 and 2.7.  The plain rotation, which the memory alone
  // bounds, runs steadier in more and shorter ones: [16384, 4096], block 1, 72 us with two, 65 with eight, 63 with
  // sixteen, and [4096, 4096] 14.6, 16.6 and 17.7)
  const int per_sm = !deq ? 3 : (format == kFormatNone ? 8 : 2);
  const int64_t cap = (int64_t)sm_count * per_sm;
  const unsigned grid = (unsigned)(want < cap ? want : cap);
  auto go = [&](auto kernel) -> bro_status {
    return cuda_ok(launch_kernel(kernel, grid, kThreads, 0, st, 1, p), "fake_quantize launch") ? BRO_OK : BRO_ERR_CUDA;
  };
  int lg = 0;
  while ((1 << lg) < block) ++lg;
  // (with the identity the signs only flip the output signs; they are applied all the same)
  auto size = [&](auto with_signs, auto mode) -> bro_status {
    constexpr bool S = decltype(with_signs)::value;
    constexpr int MODE = decltype(mode)::value;
    switch (lg) {
      case 0: return go(fake_quantize_kernel<0, S, MODE>);
      case 1: return go(fake_quantize_kernel<1, S, MODE>);
      case 2: return go(fake_quantize_kernel<2, S, MODE>);
      case 3: return go(fake_quantize_kernel<3, S, MODE>);
      case 4: return go(fake_quantize_kernel<4, S, MODE>);
      case 5: return go(fake_quantize_kernel<5, S, MODE>);
      case 6: return go(fake_quantize_kernel<6, S, MODE>);
      default: return go(fake_quantize_kernel<7, S, MODE>);
    }
  };
  auto any = [&](auto mode) { return signs ? size(std::true_type(), mode) : size(std::false_type(), mode); };
  if (!deq) return any(std::integral_constant<int, kStatistics>());
  return format == kFormatNone ? any(std::integral_constant<int, kRotation>()) : any(std::integral_constant<int, kFormats>());
}

}  // namespace fq
}  // namespace bro
