// Kernel 1 (wide form): fused block-Hadamard rotation + MXFP4 quantisation for blocks of 32, 64 and 128 channels, K a multiple of 64;
// also the two statistics (scale byte, MXFP4 error) of the same groups.
//
// Same arithmetic contract as rotate_quantize.cuh.  What differs is who holds what: a lane owns 64 consecutive channels
// (two MX groups).  A block of 64 then needs no exchange at all and a block of 128 one stage between two neighbouring lanes, in
// which each lane keeps half of its values and sends the other half (32 shuffles for 64 values; with a lane per group the
// two stages of a block of 128 took 64 shuffles for 32 values, or 32 and three packed operations for two results).  For blocks of 32
// the two groups sit side by side in packed registers and every stage is packed, the first too.
//
// A warp task is 16 rows x 128 channels, two lanes a row, by one TMA box of 128-byte segments with the 128-byte swizzle: a lane's 64
// channels are one segment, and its eight 16-byte reads are free of bank conflicts (loaded straight from global memory they
// would be 32 lines an instruction).  The ring is the warp's own, two boxes deep: no warp waits for another.  Three
// boxes: one box more in flight, but one CTA less an SM, [16384, 4096] block 64 29.3 -> 31.9 us.
//
// Instruction issue bounds it (about 9 an element with block 128).  [16384, 4096], one group a lane -> two: block 64 33.3 -> 29.4 us, 128
// 37.2 -> 30.8 (5.5 TB/s of the 2.53 bytes an element), 32 29.1 -> 29.2, [8192, 4096] 16.4 -> 15.0; scale bytes 64 30.3 -> 24.3, 128
// 38.1 -> 25.9; error 32 32.0 -> 29.3, 64 36.2 -> 31.6, 128 42.9 -> 35.4.
#pragma once

#include <type_traits>

#include "bro_common.cuh"
#include "rotate_quantize.cuh"

namespace bro {
namespace rqw {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kRows = 16;                      // a warp task: 16 rows x 128 channels, two lanes a row
constexpr int kCols = 128;
constexpr int kBoxBytes = kRows * kCols * 2;   // 4 KiB
constexpr int kStages = 2;                     // per warp
constexpr int kBarAt = kWarps * kStages * kBoxBytes;
constexpr int kSmemBytes = kBarAt + kWarps * kStages * 8 + 1024 /*alignment*/;

enum Mode { kCodes = 0, kBytes = 1, kError = 2 };

struct Params {
  int64_t M, K;
  uint8_t* codes;               // [M, K/2]
  float* mse;                   // kError: [M, K/32]
  uint8_t* scales;
  int64_t scale_kblocks;        // tensor-core layout: 512-byte blocks per 128-row block
  int layout;                   // bro_layout
  const uint16_t* signs;        // [K] bf16 +-1 (kernels with SIGNS)
  int tiles_m, tiles_k;         // tasks: row tiles x column tiles (tensor-core layout: the scale padding included)
  int wide_stores;              // codes start on 32 bytes
};

__device__ __forceinline__ void stg256(void* dst, const uint32_t (&a)[4], const uint32_t (&b)[4]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst), "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]),
               "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3])
               : "memory");
}

// Stages h = 2 .. 16 on the two groups of a lane.
__device__ __forceinline__ void stages_2_to_16(uint64_t (&P)[32]) {
#pragma unroll
  for (int hp = 1; hp < 16; hp <<= 1) {
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      if ((k & hp) == 0) {
        const uint64_t a = P[k], b = P[k + hp];
        P[k] = rq::add2(a, b);
        P[k + hp] = rq::sub2(a, b);
      }
    }
  }
}

// ---- block 32: the two groups of a lane side by side in the halves of packed registers, P[e] = (A_e, B_e) ----
// Every stage but the first (see rq::stage1) is then packed arithmetic, and so are the multiplies by the two groups' scales.
__device__ __forceinline__ void unpack_stage1_two(const uint4& a, const uint4& b, uint64_t* P) {
  const uint32_t wa[4] = {a.x, a.y, a.z, a.w}, wb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float sa, da, sb, db;
    rq::stage1(wa[k], sa, da);
    rq::stage1(wb[k], sb, db);
    P[2 * k] = rq::pack2(sa, sb);
    P[2 * k + 1] = rq::pack2(da, db);
  }
}
__device__ __forceinline__ void stages_2_to_16_two(uint64_t (&P)[32]) {
#pragma unroll
  for (int h = 2; h < 32; h <<= 1) {
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      if ((k & h) == 0) {
        const uint64_t a = P[k], b = P[k + h];
        P[k] = rq::add2(a, b);
        P[k + h] = rq::sub2(a, b);
      }
    }
  }
}
template <bool NAN_TOO>
__device__ __forceinline__ void amax_two(const uint64_t (&P)[32], float& ma, float& mb) {
  ma = mb = 0.f;
#pragma unroll
  for (int k = 0; k < 32; k += 2) {
    float a, b, a2, b2;
    rq::unpack2(P[k], a, b);
    rq::unpack2(P[k + 1], a2, b2);
    if (NAN_TOO) {
      asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(ma) : "f"(a), "f"(a2));
      asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(mb) : "f"(b), "f"(b2));
    } else {
      asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(ma) : "f"(a), "f"(a2));
      asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(mb) : "f"(b), "f"(b2));
    }
  }
}
__device__ __forceinline__ uint32_t exp_field(float m, uint32_t cbits) { return __float_as_uint(__fmul_rn(m, __uint_as_float(cbits))) >> 23; }
__device__ __forceinline__ bool usual_range(uint32_t ef) { return ef >= 27u && ef <= 250u; }       // c * 2^-E is a normal fp32
__device__ __forceinline__ uint32_t byte_of(uint32_t ef) { return ef > 2u ? ef - 2u : 0u; }
// The arithmetic of rq::quantize_group for both groups.
__device__ __forceinline__ void quantize_two(const uint64_t (&P)[32], uint32_t cbits, uint32_t (&wa)[4], uint32_t& sa, uint32_t (&wb)[4],
                                             uint32_t& sb) {
  float ma, mb;
  amax_two<false>(P, ma, mb);
  const uint32_t ea = exp_field(ma, cbits), eb = exp_field(mb, cbits);
  sa = byte_of(ea);
  sb = byte_of(eb);
  float ra[32], rb[32];
  if (usual_range(ea) && usual_range(eb)) {
    const uint64_t cc = rq::pack2(__uint_as_float(cbits + ((127u - sa) << 23)), __uint_as_float(cbits + ((127u - sb) << 23)));
#pragma unroll
    for (int k = 0; k < 32; ++k) rq::unpack2(rq::mul2(P[k], cc), ra[k], rb[k]);
  } else {
    const float c = __uint_as_float(cbits);
    const uint64_t cc = rq::pack2(c, c), pp = rq::pack2(__uint_as_float((254u - sa) << 23), __uint_as_float((254u - sb) << 23));
#pragma unroll
    for (int k = 0; k < 32; ++k) rq::unpack2(rq::mul2(rq::mul2(P[k], cc), pp), ra[k], rb[k]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    wa[j] = rq::pack_e2m1x8(ra[8 * j], ra[8 * j + 1], ra[8 * j + 2], ra[8 * j + 3], ra[8 * j + 4], ra[8 * j + 5], ra[8 * j + 6], ra[8 * j + 7]);
    wb[j] = rq::pack_e2m1x8(rb[8 * j], rb[8 * j + 1], rb[8 * j + 2], rb[8 * j + 3], rb[8 * j + 4], rb[8 * j + 5], rb[8 * j + 6], rb[8 * j + 7]);
  }
}
// The MXFP4 error of both groups (rq::group_error, format 0).
__device__ __forceinline__ void error_two(const uint64_t (&P)[32], uint32_t cbits, float& erra, float& errb) {
  float ma, mb;
  amax_two<true>(P, ma, mb);
  const uint32_t ea = exp_field(ma, cbits), eb = exp_field(mb, cbits);
  const bool usual = usual_range(ea) && usual_range(eb);
  const float c = __uint_as_float(cbits);
  auto scale_down = [&](uint32_t ef) {
    const uint32_t s = byte_of(ef);
    return usual ? __uint_as_float(cbits + ((127u - s) << 23)) : __uint_as_float(s <= 253u ? ((254u - s) << 23) : 0x00400000u);
  };
  auto scale_up = [&](uint32_t ef) { return __uint_as_float(byte_of(ef) >= 1u ? (byte_of(ef) << 23) : 0x00400000u); };     // 2^E
  const uint64_t cc = rq::pack2(c, c), ii = rq::pack2(scale_down(ea), scale_down(eb));
  uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};                  // four chains a group, as in rq::group_error
  auto add = [&](int k, uint64_t r0, uint64_t r1) {            // elements k and k + 1 of both groups
    float a0, b0, a1, b1;
    rq::unpack2(r0, a0, b0);
    rq::unpack2(r1, a1, b1);
    uint32_t ha, hb;
    asm("{ .reg .b8 b; cvt.rn.satfinite.e2m1x2.f32 b, %2, %1; cvt.rn.f16x2.e2m1x2 %0, b; }" : "=r"(ha) : "f"(a0), "f"(a1));
    asm("{ .reg .b8 b; cvt.rn.satfinite.e2m1x2.f32 b, %2, %1; cvt.rn.f16x2.e2m1x2 %0, b; }" : "=r"(hb) : "f"(b0), "f"(b1));
    auto low = [](uint32_t h) { return __half2float(__ushort_as_half((unsigned short)(h & 0xFFFFu))); };
    auto high = [](uint32_t h) { return __half2float(__ushort_as_half((unsigned short)(h >> 16))); };
    const uint64_t d0 = rq::sub2(r0, rq::pack2(low(ha), low(hb))), d1 = rq::sub2(r1, rq::pack2(high(ha), high(hb)));
    acc[k & 2] = rq::fma2(d0, d0, acc[k & 2]);
    acc[(k & 2) + 1] = rq::fma2(d1, d1, acc[(k & 2) + 1]);
  };
  if (usual) {
#pragma unroll
    for (int k = 0; k < 32; k += 2) add(k, rq::mul2(P[k], ii), rq::mul2(P[k + 1], ii));
  } else {
#pragma unroll
    for (int k = 0; k < 32; k += 2) add(k, rq::mul2(rq::mul2(P[k], cc), ii), rq::mul2(rq::mul2(P[k + 1], cc), ii));
  }
  float sa, sb;
  rq::unpack2(rq::add2(rq::add2(acc[0], acc[1]), rq::add2(acc[2], acc[3])), sa, sb);
  erra = __fmul_rn(__fmul_rn(__fmul_rn(sa, 0.03125f), scale_up(ea)), scale_up(ea));
  errb = __fmul_rn(__fmul_rn(__fmul_rn(sb, 0.03125f), scale_up(eb)), scale_up(eb));
}

template <int LOG2B, bool SIGNS, int MODE>
__global__ void __launch_bounds__(kThreads, 2) rotate_quantize_wide_kernel(const __grid_constant__ CUtensorMap tmx, const Params p) {
  static_assert(LOG2B >= 5 && LOG2B <= 7, "blocks of 32, 64, 128");
  static_assert(LOG2B > 5 || MODE != kBytes, "scale bytes: blocks of 64 and 128");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);
  const uint32_t ring = base + (uint32_t)(warp * kStages * kBoxBytes), bars = base + kBarAt + (uint32_t)(warp * kStages * 8);
  constexpr uint32_t cbits = rq::norm_bits<LOG2B>();
  if (lane == 0) {
    for (int s = 0; s < kStages; ++s) mbar_init(bars + 8 * s, 1);
    mbar_fence_init();
    fence_proxy_async_smem();
    tma_prefetch_desc(&tmx);
  }
  __syncwarp();
  griddep_wait();               // x may be written, codes/scales still read, by the kernel before
  griddep_launch_dependents();  // (only now: see the direct form)

  // task -> (row tile, column tile), column tiles fastest; advanced incrementally
  const int num_warps = (int)gridDim.x * kWarps, first = (int)blockIdx.x * kWarps + warp;
  const int step_m = num_warps / p.tiles_k, step_k = num_warps - step_m * p.tiles_k;
  auto advance = [&](int& m, int& k) {
    m += step_m;
    k += step_k;
    if (k >= p.tiles_k) { k -= p.tiles_k; ++m; }
  };
  int tm = first / p.tiles_k, tk = first - tm * p.tiles_k;
  int am = tm, ak = tk;                                    // the next task to request
  auto request = [&](int stage) {
    if (am >= p.tiles_m) return false;
    const uint32_t bar = bars + 8 * stage;
    mbar_arrive_expect_tx_elect(bar, kBoxBytes);
    tma_load_3d_elect(ring + (uint32_t)(stage * kBoxBytes), &tmx, 0, 2 * ak, am * kRows, bar);     // (zeros outside x)
    advance(am, ak);
    return true;
  };
  int in_flight = 0;
  for (int s = 0; s < kStages; ++s) in_flight += request(s) ? 1 : 0;

  const int half = lane & 1;
  // Block 128: the odd lane loads its 64 channels with the halves exchanged (register pair k holds true pair k ^ 16), so that
  // both lanes keep registers 0..15 and send registers 16..31; see rq::cross_lane_split for the arithmetic.
  const uint32_t hswz = LOG2B == 7 && half ? 4u : 0u;
  const float s0 = LOG2B == 7 && half ? -1.f : 1.f;
  const uint64_t s2 = rq::pack2(s0, s0), ns2 = rq::pack2(-s0, -s0);
  const int ng = (int)(p.K >> 5);
  int stage = 0;
  uint32_t phase = 0;
  for (; tm < p.tiles_m; advance(tm, tk)) {
    if (!mbar_wait_warp(bars + 8 * stage, phase, SITE_RQ_FULL)) break;
    uint64_t P[32];
    {
      const uint32_t src = ring + (uint32_t)(stage * kBoxBytes) + (uint32_t)lane * 128u;
      auto chunk = [&](uint32_t j) {
        uint4 q = lds128(src + (((j ^ hswz) ^ ((uint32_t)lane & 7u)) << 4));
        if (SIGNS) {
          const int ch = tk * kCols + half * 64 + (int)(j ^ hswz) * 8;
          if (ch < (int)p.K) q = rq::apply_signs(q, __ldg(reinterpret_cast<const uint4*>(p.signs + ch)));
        }
        return q;
      };
      if constexpr (LOG2B == 5) {
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) unpack_stage1_two(chunk(j), chunk(j + 4), P + 8 * j);
      } else {
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j) rq::unpack_stage1(chunk(j), P + 4 * j);
      }
    }
    __syncwarp();
    in_flight += request(stage) ? 0 : -1;
    if (++stage == kStages) { stage = 0; phase ^= 1u; }

    uint64_t X[16], Y[16];
    if constexpr (LOG2B == 5) {
      stages_2_to_16_two(P);
    } else if constexpr (LOG2B == 6) {
      stages_2_to_16(P);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        X[k] = rq::add2(P[k], P[k + 16]);
        Y[k] = rq::sub2(P[k], P[k + 16]);
      }
    } else {
      stages_2_to_16(P);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const uint64_t keep = rq::fma2(P[k], s2, P[k + 16]), send = rq::fma2(P[k + 16], ns2, P[k]);
        const uint64_t R = rq::shfl_xor2(send, 1);
        X[k] = rq::add2(keep, R);
        Y[k] = rq::fma2(keep, s2, rq::mul2(R, ns2));
      }
    }
    // groups of this lane within the row's four: blocks of 32 / 64 2 half, 2 half + 1; block 128 half, half + 2
    const int64_t row = (int64_t)tm * kRows + (lane >> 1);
    const int g0 = tk * 4;
    const bool live = row < p.M && g0 + 2 * half < ng;
    if constexpr (MODE == kError) {
      if (live) {
        float* dst = p.mse + row * ng + g0 + (LOG2B == 7 ? half : 2 * half);
        if constexpr (LOG2B == 5) {
          error_two(P, cbits, dst[0], dst[1]);
        } else {
          dst[0] = rq::group_error(X, cbits, 0);
          dst[LOG2B == 7 ? 2 : 1] = rq::group_error(Y, cbits, 0);
        }
      }
      __syncwarp();
      continue;
    }
    uint32_t wx[4] = {}, wy[4] = {}, sx, sy;
    if constexpr (LOG2B == 5) {
      quantize_two(P, cbits, wx, sx, wy, sy);
    } else if constexpr (MODE == kBytes) {
      sx = rq::group_scale_byte(X, cbits);
      sy = rq::group_scale_byte(Y, cbits);
    } else {
      sx = rq::quantize_group(X, cbits, wx);
      sy = rq::quantize_group(Y, cbits, wy);
    }
    if (MODE == kCodes && live) {
      uint8_t* dst = p.codes + row * (p.K >> 1) + (int64_t)g0 * 16;
      if (LOG2B == 7) {
        *reinterpret_cast<uint4*>(dst + 16 * half) = make_uint4(wx[0], wx[1], wx[2], wx[3]);
        *reinterpret_cast<uint4*>(dst + 16 * half + 32) = make_uint4(wy[0], wy[1], wy[2], wy[3]);
      } else if (p.wide_stores) {
        stg256(dst + 32 * half, wx, wy);
      } else {
        *reinterpret_cast<uint4*>(dst + 32 * half) = make_uint4(wx[0], wx[1], wx[2], wx[3]);
        *reinterpret_cast<uint4*>(dst + 32 * half + 16) = make_uint4(wy[0], wy[1], wy[2], wy[3]);
      }
    }
    // the row's four scale bytes -> one 32-bit word in the even lane
    const uint32_t mine = live ? (LOG2B == 7 ? (sx | (sy << 16)) : (sx | (sy << 8))) : 0u;
    const uint32_t sb = mine | (__shfl_xor_sync(0xFFFFFFFFu, mine, 1) << (LOG2B == 7 ? 8 : 16));
    if (half == 0) {
      if (MODE == kCodes && p.layout == BRO_LAYOUT_GEMM) {
        // 512-byte block (row / 128, g / 4): byte (r % 32) * 16 + ((r % 128) / 32) * 4 + g % 4
        const int r = (int)(row & 127);
        *reinterpret_cast<uint32_t*>(p.scales + ((row >> 7) * p.scale_kblocks + tk) * 512 + (r & 31) * 16 + (r >> 5) * 4) = sb;
      } else if (row < p.M) {
        uint8_t* dst = p.scales + row * ng + g0;
        if (g0 + 4 <= ng && (reinterpret_cast<uintptr_t>(dst) & 3) == 0) {
          *reinterpret_cast<uint32_t*>(dst) = sb;
        } else {
          for (int i = 0; i < 4 && g0 + i < ng; ++i) dst[i] = (uint8_t)(sb >> (8 * i));
        }
      }
    }
  }
  // (only after a lost wait is anything left: do not leave while copies may still land, wait once more for each stage)
  for (; in_flight > 0; --in_flight) {
    mbar_wait_warp(bars + 8 * stage, phase, SITE_RQ_DRAIN);
    if (++stage == kStages) { stage = 0; phase ^= 1u; }
  }
}

// x as a 3-D tensor {64 bf16, K / 64, M rows}, box = 128 channels of 16 rows, 128-byte swizzle.
bro_status make_tile_map(CUtensorMap* map, const void* x, int64_t M, int64_t K, int64_t ldx);

template <int LOG2B, bool SIGNS, int MODE>
inline bro_status launch_one(const CUtensorMap& tmx, const Params& p, int sm_count, cudaStream_t st) {
  auto kernel = rotate_quantize_wide_kernel<LOG2B, SIGNS, MODE>;
  static DeviceOnce once;            // (one per template instantiation)
  int blocks_per_sm = 1;
  const bro_status rc = device_once(once, &blocks_per_sm, [&](int* n) {
    return cuda_ok(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes),
                   "cudaFuncSetAttribute(rotate_quantize_wide)") &&
                   cuda_ok(cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, kernel, kThreads, kSmemBytes),
                           "occupancy(rotate_quantize_wide)")
               ? BRO_OK
               : BRO_ERR_CUDA;
  });
  if (rc != BRO_OK) return rc;
  const int64_t want = ((int64_t)p.tiles_m * p.tiles_k + kWarps - 1) / kWarps, cap = (int64_t)sm_count * blocks_per_sm;
  return cuda_ok(launch_kernel(kernel, (unsigned)(want < cap ? want : cap), kThreads, kSmemBytes, st, 1, tmx, p),
                 "rotate_quantize_wide launch")
             ? BRO_OK
             : BRO_ERR_CUDA;
}

// mse set: the MXFP4 error of every group; codes not set: scale bytes only (both [M, K/32], layout canonical).
inline bro_status launch(const void* x, int64_t M, int64_t K, int64_t ldx, int log2b, const void* signs, void* codes,
                         void* scales, float* mse, bro_layout layout, int64_t scale_kblocks, int sm_count, cudaStream_t st) {
  CUtensorMap tmx;
  const bro_status rc = make_tile_map(&tmx, x, M, K, ldx);
  if (rc != BRO_OK) return rc;
  Params p;
  p.M = M; p.K = K;
  p.codes = static_cast<uint8_t*>(codes);
  p.scales = static_cast<uint8_t*>(scales);
  p.mse = mse;
  p.scale_kblocks = scale_kblocks;
  p.layout = (int)layout;
  p.signs = static_cast<const uint16_t*>(signs);
  p.tiles_m = (int)(layout == BRO_LAYOUT_GEMM ? (M + 127) / 128 * (128 / kRows) : (M + kRows - 1) / kRows);
  p.tiles_k = (int)(layout == BRO_LAYOUT_GEMM ? scale_kblocks : (K + kCols - 1) / kCols);
  p.wide_stores = (reinterpret_cast<uintptr_t>(codes) & 31) == 0 ? 1 : 0;
  auto size = [&](auto mode) -> bro_status {
    constexpr int MODE = decltype(mode)::value;
    if (log2b == 6) return signs ? launch_one<6, true, MODE>(tmx, p, sm_count, st) : launch_one<6, false, MODE>(tmx, p, sm_count, st);
    if (log2b == 7) return signs ? launch_one<7, true, MODE>(tmx, p, sm_count, st) : launch_one<7, false, MODE>(tmx, p, sm_count, st);
    // (scale bytes of blocks of 32: the register-streaming kernel is the faster one)
    if constexpr (MODE == kBytes) return BRO_ERR_UNSUPPORTED;
    else return signs ? launch_one<5, true, MODE>(tmx, p, sm_count, st) : launch_one<5, false, MODE>(tmx, p, sm_count, st);
  };
  if (mse) return size(std::integral_constant<int, kError>());
  if (!codes) return size(std::integral_constant<int, kBytes>());
  return size(std::integral_constant<int, kCodes>());
}

}  // namespace rqw
}  // namespace bro
