// Analysis kernels: the scale statistics behind the paper's regular-block / outlier-block argument
// (Sec. 4.1: blocks without / with outliers; Sec. 4.2, Fig. 6 caption: outliers are the top 0.1 % of
// the activations by absolute value; App. A.3: under global rotation most regular blocks' scales grow,
// block rotation removes most of that growth).  All of it is integer work, so results are exact and
// independent of the order in which threads add their counts.
//
//   group_scale_bytes_identity   E8M0 byte of every group of 32 of the un-rotated input
//   outlier_scan                 the k-th largest magnitude from a histogram of the largest bf16 patterns, and a
//                                code per group from which most groups' membership follows
//   outlier_group_mask           groups holding a value at or above the threshold
//   scale_histogram              256-bin histograms of the scale bytes, regular and outlier groups
//   scale_inflation              per class: groups whose byte went down / stayed / went up
#pragma once

#include "bro_common.cuh"

namespace bro {
namespace stats {

constexpr int kMagBins = 32768;                       // bf16 magnitudes: the low 15 bits
constexpr size_t kWorkspaceBytes = (size_t)kMagBins * 8 + 64;
// Behind the histogram: word 0 counts the CTAs that have merged theirs, word 1 is the smallest pattern counted.
constexpr int kTicketWord = 0, kLowestWord = 1;

// Row and group of a thread's first item and of its stride, so that the loop over a matrix divides once.  (First item and
// stride are numbers of threads and fit 32 bits, as K / 32 does: divisions in 64 bits took 0.2 us of a small launch.)
struct GroupWalk {
  int64_t row, g, step_row, step_g, ng;
  __device__ GroupWalk(uint32_t first, uint32_t step, int64_t ng_) : ng(ng_) {
    const uint32_t n = (uint32_t)ng_;
    row = first / n;
    g = first % n;
    step_row = step / n;
    step_g = step % n;
  }
  __device__ void next() {
    row += step_row;
    g += step_g;
    if (g >= ng) { g -= ng; ++row; }
  }
};

// max of the 15-bit magnitude patterns of 8 bf16 values (finite non-negative floats order like integers), both halves of
// a word at a time
__device__ __forceinline__ uint32_t max_mag8_pairs(uint4 q) {
  return __vmaxu2(__vmaxu2(q.x & 0x7FFF7FFFu, q.y & 0x7FFF7FFFu), __vmaxu2(q.z & 0x7FFF7FFFu, q.w & 0x7FFF7FFFu));
}
__device__ __forceinline__ uint32_t max_mag8(uint4 q) {
  const uint32_t m = max_mag8_pairs(q);
  return max(m & 0xFFFFu, m >> 16);
}

__device__ __forceinline__ uint32_t max_mag8_plain(uint4 q) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m = max(m, w[i] & 0x7FFFu);
    m = max(m, (w[i] >> 16) & 0x7FFFu);
  }
  return m;
}
// The largest magnitude pattern of a group, value by value: in a launch that little else fills, the two-at-a-time form
// showed in the latency (scale bytes before a rotation of [16, 8192] 1.65 -> 1.76 us, [512, 4096] 2.0 -> 2.15).
__device__ __forceinline__ uint32_t group_max_mag(const uint16_t* x, int64_t row, int64_t ldx, int64_t g) {
  const uint4* src = reinterpret_cast<const uint4*>(x + row * ldx + g * 32);
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) m = max(m, max_mag8_plain(__ldg(src + j)));
  return m;
}

// The largest magnitude pattern of every group of a run of 32 consecutive groups in memory, by a warp that reads whole lines:
// lane l holds the 16 bytes 256 j + 8 l .. of the 2 KiB in q[j], a quarter of group 8 j + l / 4.  The four lanes of a quad
// exchange maxima (both halves of a word at a time) so that lane l is left with group 8 (l mod 4) + l / 4.
__device__ __forceinline__ uint32_t quad_maxima(const uint32_t (&m)[4], int lane) {
  const bool b0 = (lane & 1) != 0, b1 = (lane & 2) != 0;
  uint32_t k0 = b0 ? m[1] : m[0], k1 = b0 ? m[3] : m[2];                 // groups j = b0 and b0 + 2
  k0 = __vmaxu2(k0, __shfl_xor_sync(0xFFFFFFFFu, b0 ? m[0] : m[1], 1));
  k1 = __vmaxu2(k1, __shfl_xor_sync(0xFFFFFFFFu, b0 ? m[2] : m[3], 1));
  const uint32_t k = __vmaxu2(b1 ? k1 : k0, __shfl_xor_sync(0xFFFFFFFFu, b1 ? k0 : k1, 2));
  return max(k & 0xFFFFu, k >> 16);
}
__device__ __forceinline__ int quad_group(int lane) { return 8 * (lane & 3) + (lane >> 2); }

// The byte is max(expfield(amax) - 2, 0) with expfield the 8-bit exponent of amax as fp32 — for a bf16 value that is
// bits 7..14 of its pattern.
__device__ __forceinline__ uint8_t scale_byte_of(uint32_t mag) {
  const uint32_t ef = mag >> 7;
  return (uint8_t)(ef > 2u ? ef - 2u : 0u);
}
// One thread per group.  (Neither this kernel nor the next signals its dependents: they are all loads, and CTAs of the next kernel that
// wait beside them cost [1000, 2112] 1.9 -> 2.3 us, [300, 14336] 2.9 -> 3.4.)
__global__ void __launch_bounds__(256) group_scale_bytes_identity(const uint16_t* x, int64_t M, int64_t K, int64_t ldx,
                                                                  uint8_t* scales) {
  griddep_wait();
  const int64_t ng = K >> 5, total = M * ng;
  // (divided per group, not walked: the walk's two divisions before the loop and its carry in it cost 0.2 us of a small
  // launch and 24.3 -> 27.2 us at [16384, 4096])
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = i / ng, g = i - row * ng;
    scales[i] = scale_byte_of(group_max_mag(x, row, ldx, g));
  }
}
// Rows without a stride are one row: 32 groups a warp and pass.
__global__ void __launch_bounds__(256) group_scale_bytes_identity_flat(const uint16_t* x, int64_t total, uint8_t* scales) {
  griddep_wait();
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)gridDim.x * 256;
  for (int64_t base = (int64_t)blockIdx.x * 256 + (threadIdx.x & ~31u); base < total; base += step) {
    const uint4* src = reinterpret_cast<const uint4*>(x + base * 32) + lane;
    uint32_t m[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool in = base + 8 * j + (lane >> 2) < total;
      m[j] = max_mag8_pairs(in ? __ldg(src + 32 * j) : make_uint4(0u, 0u, 0u, 0u));
    }
    const uint32_t mag = quad_maxima(m, lane);
    const int64_t i = base + quad_group(lane);
    if (i < total) scales[i] = scale_byte_of(mag);
  }
}

constexpr int kScanThreads = 1024;
__device__ __forceinline__ uint32_t group_code(uint32_t above_lowest) { return 1u + min(253u, above_lowest >> 3); }
constexpr int kSamples = 4 * kScanThreads;

// Counts of the 1024 threads, thread 0 first -> inclusive prefix sums.
__device__ __forceinline__ unsigned long long block_prefix(unsigned long long v, unsigned long long* warp_sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long o = __shfl_up_sync(0xFFFFFFFFu, v, d);
    if (lane >= d) v += o;
  }
  __syncthreads();
  if (lane == 31) warp_sums[warp] = v;
  __syncthreads();
  unsigned long long before = lane < warp ? warp_sums[lane] : 0ull;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, d);
  return before + v;
}

// The k-th largest of the counted magnitudes, by the whole CTA: the largest pattern t with count(patterns >= t) >= k.
// Warp w adds up the 1024 patterns of segment 31 - w; the segment in which the count from above passes k is then searched
// with one pattern per thread.  Nothing below `lowest` was counted.  Returns false if fewer than k were counted.
template <typename Count>
__device__ __forceinline__ bool find_threshold(Count&& count, unsigned long long k, uint32_t lowest, uint32_t* info,
                                               unsigned long long* warp_sums) {
  __shared__ unsigned long long segments[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, base = 1024 * (31 - warp);
  unsigned long long sum = 0;
  if (base + 1024 > (int)lowest) {
#pragma unroll
    for (int j = 0; j < 32; ++j) sum += count(base + 32 * j + lane);
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
  if (lane == 0) segments[warp] = sum;
  __syncthreads();
  unsigned long long above = 0;                       // counted above the segment searched
  int seg = 0;
  while (seg < 32 && above + segments[seg] < k) above += segments[seg++];
  if (seg == 32) return false;                        // (the same for all threads)
  const int t = 1024 * (31 - seg) + 1023 - (int)threadIdx.x;
  const unsigned long long mine = count(t), upto = above + block_prefix(mine, warp_sums);
  if (upto >= k && upto - mine < k) {
    info[0] = (uint32_t)t;
    info[1] = 0u;
    info[2] = (uint32_t)(k & 0xFFFFFFFFull);
    info[3] = (uint32_t)(k >> 32);
  }
  return true;
}

// The same for counts of 32 bits with one trip to the histogram: a warp holds the 1024 patterns of its segment, the highest with
// warp 0, and the warp in which the count from above passes k looks into what it holds.  ([300, 4096] 0.6 us less than in two trips.)
__device__ __forceinline__ bool find_threshold_narrow(const uint32_t* hist, uint32_t k, uint32_t lowest, uint32_t* info) {
  __shared__ uint32_t segments[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, base = 1024 * (31 - warp);
  uint4 c[8] = {};                                    // patterns base + 128 j + 4 lane ..
  uint32_t sum = 0;
  if (base + 1024 > (int)lowest) {
#pragma unroll
    for (int j = 0; j < 8; ++j) c[j] = __ldcg(reinterpret_cast<const uint4*>(hist + base + 128 * j) + lane);
#pragma unroll
    for (int j = 0; j < 8; ++j) sum += c[j].x + c[j].y + c[j].z + c[j].w;
  }
  const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, sum);
  if (lane == 0) segments[warp] = total;
  __syncthreads();
  uint32_t above = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? segments[lane] : 0u);      // counted above this segment
  const bool here = above < k && above + total >= k;
  if (here) {
#pragma unroll
    for (int j = 7; j >= 0; --j) {
      uint32_t upto = c[j].x + c[j].y + c[j].z + c[j].w;            // -> of this lane and those above it
      const uint32_t all = __reduce_add_sync(0xFFFFFFFFu, upto);
      if (above < k && above + all >= k) {
        const uint32_t v[4] = {c[j].x, c[j].y, c[j].z, c[j].w};
        const uint32_t mine = upto;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t o = __shfl_down_sync(0xFFFFFFFFu, upto, d);
          if (lane + d < 32) upto += o;
        }
        uint32_t count = above + upto - mine;
#pragma unroll
        for (int q = 3; q >= 0; --q) {
          if (count < k && count + v[q] >= k) {
            info[0] = (uint32_t)(base + 128 * j + 4 * lane + q);
            info[1] = 0u;
            info[2] = k;
            info[3] = 0u;
          }
          count += v[q];
        }
      }
      above += all;
    }
  }
  return __syncthreads_or(here) != 0;
}

// In front of the scan: clears the histogram and the words behind it, and lets the scan start once everything older is complete (a
// memset in its place stood between the kernel before and the scan without any overlap).
constexpr int kClearCtas = 8;
__global__ void __launch_bounds__(kScanThreads) outlier_clear(unsigned long long* hist) {
  griddep_wait();
  griddep_launch_dependents();
  uint4* dst = reinterpret_cast<uint4*>(hist);
  for (int i = (int)(blockIdx.x * kScanThreads + threadIdx.x); i < (int)(kWorkspaceBytes / 16); i += kClearCtas * kScanThreads)
    dst[i] = make_uint4(0u, 0u, 0u, 0u);
}

// The outliers are the top 0.1 % (top k of n) of the magnitudes, found exactly from a histogram of bf16 patterns; one pass
// over x.  A shared-memory atomic per value bounded it before (75 us for 67 M values and 20 us for the search in a
// launch of its own; now 36 us with the mask, of which 22 us are the pass, 134 MB at 0.93 of the copy bandwidth, and the rest a chain
// that [300, 4096], 14 us, has too: clear, sample, merge, search, mask; a warp that reads whole lines gives 35.9 as well), so only values of
// at least `lowest` are counted, a pattern that every CTA derives from the same 4096 sampled
// values such that about 4 k values (and 12 of the sample) lie at or above it: the loop reduces a group to its maximum and
// touches the histogram for the few groups that reach `lowest`.  Behind outlier_clear, which waited for everything older, it runs up
// to the merging of the histograms without waiting for the histogram to be cleared.  The last CTA to merge searches the
// threshold, without a launch of its own.  Should the sample have misled (fewer than k counted), that CTA counts everything
// by itself: slow, and exact.
// codes[g] = 0 if the group's maximum is below `lowest`, else group_code(maximum - lowest): see outlier_group_mask.
__global__ void __launch_bounds__(kScanThreads, 1) outlier_scan(const uint16_t* x, int64_t M, int64_t K, int64_t ldx,
                                                                unsigned long long k, unsigned long long* hist, uint32_t* info,
                                                                uint8_t* codes) {
  extern __shared__ uint32_t local[];                 // kMagBins counters; the sample's 1024 coarse ones first
  __shared__ unsigned long long warp_sums[32];
  __shared__ uint32_t lowest_s;
  __shared__ bool last_s;
  uint32_t* words = reinterpret_cast<uint32_t*>(hist + kMagBins);
  local[threadIdx.x] = 0u;
  if (threadIdx.x == 0) lowest_s = 0u;
  __syncthreads();
  const int64_t n = M * K;
  if (n > 16 * kSamples) {
    const unsigned long long want = 4 * ((k * kSamples + n - 1) / n) + 12;      // sampled values at or above `lowest`
#pragma unroll
    for (int j = 0; j < kSamples / kScanThreads; ++j) {
      // a fixed scattering of rows and channels (multiplicative hashing)
      const uint32_t i = (uint32_t)(j * kScanThreads) + threadIdx.x;
      const uint32_t h1 = (i + 1u) * 2654435761u, h2 = (h1 ^ (h1 >> 15)) * 2246822519u;
      const int64_t row = (int64_t)(((uint64_t)h1 * (uint64_t)M) >> 32), col = (int64_t)(((uint64_t)h2 * (uint64_t)K) >> 32);
      atomicAdd(&local[(__ldg(x + row * ldx + col) & 0x7FFFu) >> 5], 1u);
    }
    __syncthreads();
    const uint32_t mine = local[kScanThreads - 1 - threadIdx.x];
    const unsigned long long upto = block_prefix(mine, warp_sums);
    if (upto >= want && upto - mine < want) lowest_s = 32u * (uint32_t)(kScanThreads - 1 - (int)threadIdx.x);
    __syncthreads();
  }
  const uint32_t lowest = lowest_s;
  for (int i = (int)(lowest & ~1023u) + (int)threadIdx.x; i < kMagBins; i += kScanThreads) local[i] = 0u;
  __syncthreads();

  const int64_t ng = K >> 5, total = M * ng;
  // A CTA takes 1024 consecutive groups at a time and its warps change places from one time to the next: outlier channels
  // keep their place in a row, and a warp that always met them finished a third later than the others.
  const int64_t step = (int64_t)gridDim.x * kScanThreads;
  GroupWalk at(blockIdx.x * (uint32_t)kScanThreads, (uint32_t)step, ng);       // the CTA's first group
  // (ceil(2^32 / ng) does not fit 32 bits for rows of one group)
  const uint32_t magic = ng > 1 && ng < kScanThreads ? (uint32_t)((0x100000000ull + ng - 1) / ng) : 0u;
  {
    uint4 nxt[4];                                     // the next group's 64 bytes, in flight while this one is counted
    int place = (int)threadIdx.x;
    auto load = [&] {
      // (at.g + place) / ng is 0 or 1 for long rows; for short ones the product with ceil(2^32 / ng) is exact; a row of
      // one group is its own quotient
      const uint32_t v = (uint32_t)at.g + (uint32_t)place;
      const uint32_t over = magic ? __umulhi(v, magic) : (ng == 1 ? v : (v >= (uint32_t)ng ? 1u : 0u));
      const uint4* src = reinterpret_cast<const uint4*>(x + (at.row + over) * ldx + (int64_t)(v - over * (uint32_t)ng) * 32);
#pragma unroll
      for (int j = 0; j < 4; ++j) nxt[j] = __ldg(src + j);
    };
    int64_t base = (int64_t)blockIdx.x * kScanThreads;
    if (base + place < total) load();
    for (; base < total; base += step) {
      const int64_t i = base + place;
      const bool live = i < total;
      uint4 q[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) q[j] = nxt[j];
      at.next();
      place = (place + 32) & (kScanThreads - 1);
      if (base + step + place < total) load();
      if (!live) continue;
      uint32_t m4[4], reach = 0;                      // maxima of the 8-value chunks; chunks that reach `lowest`
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        m4[j] = max_mag8(q[j]);
        reach |= m4[j] >= lowest ? 1u << j : 0u;
      }
      const uint32_t m = max(max(m4[0], m4[1]), max(m4[2], m4[3]));
      codes[i] = (uint8_t)(m < lowest ? 0u : group_code(m - lowest));
      while (reach) {                                 // (mostly no chunk, or one: cheaper than a pass over all 32 values)
        const bool b0 = reach & 1u, b1 = reach & 2u, b2 = reach & 4u;
        const uint4 v = b0 ? q[0] : (b1 ? q[1] : (b2 ? q[2] : q[3]));
        reach &= reach - 1u;
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint32_t lo = w[c] & 0x7FFFu, hi = (w[c] >> 16) & 0x7FFFu;
          if (lo >= lowest) atomicAdd(&local[lo], 1u);
          if (hi >= lowest) atomicAdd(&local[hi], 1u);
        }
      }
    }
  }
  griddep_wait();                                     // the histogram is clear
  griddep_launch_dependents();
  __syncthreads();
  // Fewer than 2^32 values in all: two 32-bit counts to a 64-bit atomic (no count can carry into its neighbour), half the
  // atomics that all CTAs throw at the same few thousand bins.
  const bool wide = (n >> 32) != 0;
  for (int i = (int)(lowest & ~1023u) + 2 * (int)threadIdx.x; i < kMagBins; i += 2 * kScanThreads) {
    const uint32_t c0 = local[i], c1 = local[i + 1];
    if (wide) {
      if (c0) atomicAdd(&hist[i], (unsigned long long)c0);
      if (c1) atomicAdd(&hist[i + 1], (unsigned long long)c1);
    } else if (c0 | c1) {
      atomicAdd(&hist[i >> 1], (unsigned long long)c0 | (unsigned long long)c1 << 32);
    }
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last_s = atomicAdd(words + kTicketWord, 1u) + 1u == gridDim.x;
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  if (threadIdx.x == 0) words[kLowestWord] = lowest;
  auto counted = [&](int b) {
    return wide ? __ldcg(hist + b) : (unsigned long long)__ldcg(reinterpret_cast<const uint32_t*>(hist) + b);
  };
  if (wide ? find_threshold(counted, k, lowest, info, warp_sums)
           : find_threshold_narrow(reinterpret_cast<const uint32_t*>(hist), (uint32_t)k, lowest, info))
    return;
  // fewer than k at or above `lowest`
  for (int i = (int)threadIdx.x; i < kMagBins; i += kScanThreads) local[i] = 0u;
  __syncthreads();
  GroupWalk whole(threadIdx.x, kScanThreads, ng);
  for (int64_t i = threadIdx.x; i < total; i += kScanThreads, whole.next()) {
    const uint16_t* src = x + whole.row * ldx + whole.g * 32;
    for (int j = 0; j < 32; ++j) {
      // (a 32-bit counter of one CTA can pass 2^32 only beyond 4 G values of one pattern: carried into the global word)
      const uint32_t b = src[j] & 0x7FFFu;
      if (b < lowest && atomicAdd(&local[b], 1u) == 0xFFFFFFFFu) atomicAdd(&hist[b], 1ull << 32);   // (wide)
    }
  }
  __syncthreads();
  if (!find_threshold([&](int b) { return counted(b) + local[b]; }, k, 0u, info, warp_sums) && threadIdx.x == 0) {
    info[0] = 0u; info[1] = 0u; info[2] = (uint32_t)(k & 0xFFFFFFFFull); info[3] = (uint32_t)(k >> 32);     // (k > n)
  }
}

// mask holds outlier_scan's codes and receives 0 / 1.  A code steps by 8 patterns, a sixteenth of an octave: with t the
// threshold, a code above that of t is an outlier, one below is not, and the few groups with the same code are read again
// (all groups, should t lie below `lowest`).  2 bytes a group instead of 64: 23 us -> 2 us for 2 M groups.
__global__ void __launch_bounds__(256) outlier_group_mask(const uint16_t* x, int64_t M, int64_t K, int64_t ldx,
                                                          const uint32_t* info, const unsigned long long* hist, uint8_t* mask) {
  griddep_wait();
  griddep_launch_dependents();
  const int64_t ng = K >> 5, total = M * ng;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, threads = (int64_t)gridDim.x * blockDim.x;
  const int64_t vec = (reinterpret_cast<uintptr_t>(mask) & 15) == 0 ? total >> 4 : 0;      // 16 groups at a time
  uint4 v = tid < vec ? reinterpret_cast<uint4*>(mask)[tid] : make_uint4(0u, 0u, 0u, 0u);  // (beside the load of the threshold)
  const uint32_t t = info[0], lowest = reinterpret_cast<const uint32_t*>(hist + kMagBins)[kLowestWord];
  auto again = [&](int64_t i) { return (uint32_t)(group_max_mag(x, i / ng, ldx, i - i / ng * ng) >= t ? 1 : 0); };
  if (t < lowest) {
    for (int64_t i = tid; i < total; i += threads) mask[i] = (uint8_t)again(i);
    return;
  }
  const uint32_t code = group_code(t - lowest), code4 = code * 0x01010101u;
  for (int64_t i = tid; i < vec; i += threads) {
    if (i != tid) v = reinterpret_cast<uint4*>(mask)[i];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t r[4], open = 0;                          // one bit a group to be read again
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      r[c] = __vcmpgtu4(w[c], code4) & 0x01010101u;
      open |= (((__vcmpeq4(w[c], code4) & 0x01010101u) * 0x01020408u) >> 24 & 0xFu) << (4 * c);
    }
    for (; open; open &= open - 1u) {                 // (all 16 in one loop: as many trips to memory as the busiest lane has groups)
      const int bit = __ffs(open) - 1;
      const uint32_t one = again((i << 4) + bit) << (8 * (bit & 3));
#pragma unroll
      for (int c = 0; c < 4; ++c) r[c] |= (bit >> 2) == c ? one : 0u;
    }
    reinterpret_cast<uint4*>(mask)[i] = make_uint4(r[0], r[1], r[2], r[3]);
  }
  for (int64_t i = (vec << 4) + tid; i < total; i += threads)
    mask[i] = (uint8_t)(mask[i] == code ? again(i) : (mask[i] > code ? 1u : 0u));
}

// Counts of few groups come from one CTA, which writes them whether or not the output was zeroed (`alone`); more groups
// add to an output that clear_counts zeroes, from the whole grid.  clear_counts lets the counting kernel start once everything
// older is complete, so that it counts meanwhile and waits only before it adds; a memset in its place stood between two
// kernels without any overlap.  Groups are read 16 at a time where the pointers allow it.
constexpr int kCountThreads = 1024;
constexpr int64_t kAloneGroups = 65536;
inline bool count_alone(int64_t n_groups) { return n_groups <= kAloneGroups; }

__global__ void __launch_bounds__(512) clear_counts(unsigned long long* counts, int n) {
  griddep_wait();
  griddep_launch_dependents();
  if ((int)threadIdx.x < n) counts[threadIdx.x] = 0ull;
}

__device__ __forceinline__ bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

__global__ void __launch_bounds__(kCountThreads) scale_histogram(const uint8_t* scales, const uint8_t* mask, int64_t n, int alone,
                                                                 unsigned long long* hist) {
  __shared__ uint32_t local[512];
  for (int i = threadIdx.x; i < 512; i += kCountThreads) local[i] = 0u;
  __syncthreads();
  if (alone) griddep_wait();           // (else the scales and the mask are older than clear_counts, which waited for them)
  const int64_t tid = (int64_t)blockIdx.x * kCountThreads + threadIdx.x, threads = (int64_t)gridDim.x * kCountThreads;
  const int64_t vec = aligned16(scales) && aligned16(mask) ? n >> 4 : 0;
  for (int64_t i = tid; i < vec; i += threads) {
    const uint4 s = __ldg(reinterpret_cast<const uint4*>(scales) + i), m = __ldg(reinterpret_cast<const uint4*>(mask) + i);
    const uint32_t sw[4] = {s.x, s.y, s.z, s.w}, mw[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t b = (sw[j >> 2] >> (8 * (j & 3))) & 0xFFu;
      atomicAdd(&local[(((mw[j >> 2] >> (8 * (j & 3))) & 0xFFu) ? 256u : 0u) + b], 1u);
    }
  }
  for (int64_t i = (vec << 4) + tid; i < n; i += threads) atomicAdd(&local[(mask[i] ? 256 : 0) + scales[i]], 1u);
  if (!alone) griddep_wait();
  griddep_launch_dependents();
  __syncthreads();
  for (int i = threadIdx.x; i < 512; i += kCountThreads) {
    if (alone) hist[i] = local[i];
    else if (local[i]) atomicAdd(&hist[i], (unsigned long long)local[i]);
  }
}

__global__ void __launch_bounds__(kCountThreads) scale_inflation(const uint8_t* before, const uint8_t* after, const uint8_t* mask,
                                                                 int64_t n, int alone, unsigned long long* counts) {
  __shared__ uint32_t local[6];
  if (threadIdx.x < 6) local[threadIdx.x] = 0u;
  __syncthreads();
  if (alone) griddep_wait();           // (else: see scale_histogram)
  uint32_t mine[6] = {0, 0, 0, 0, 0, 0};
  const int64_t tid = (int64_t)blockIdx.x * kCountThreads + threadIdx.x, threads = (int64_t)gridDim.x * kCountThreads;
  const int64_t vec = aligned16(before) && aligned16(after) && aligned16(mask) ? n >> 4 : 0;
  for (int64_t i = tid; i < vec; i += threads) {
    const uint4 b4 = __ldg(reinterpret_cast<const uint4*>(before) + i), a4 = __ldg(reinterpret_cast<const uint4*>(after) + i),
                m4 = __ldg(reinterpret_cast<const uint4*>(mask) + i);
    const uint32_t b[4] = {b4.x, b4.y, b4.z, b4.w}, a[4] = {a4.x, a4.y, a4.z, a4.w}, m[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // one bit a byte: outlier group, byte went down, byte went up
      const uint32_t o = __vcmpne4(m[j], 0u) & 0x01010101u;
      const uint32_t down = __vcmpltu4(a[j], b[j]) & 0x01010101u, up = __vcmpgtu4(a[j], b[j]) & 0x01010101u;
      const uint32_t same = 0x01010101u & ~(down | up);
      mine[0] += __popc(down & ~o); mine[1] += __popc(same & ~o); mine[2] += __popc(up & ~o);
      mine[3] += __popc(down & o);  mine[4] += __popc(same & o);  mine[5] += __popc(up & o);
    }
  }
  for (int64_t i = (vec << 4) + tid; i < n; i += threads) {
    const int j = after[i] < before[i] ? 0 : (after[i] == before[i] ? 1 : 2);
    const int c = (mask[i] ? 3 : 0) + j;
#pragma unroll
    for (int q = 0; q < 6; ++q) mine[q] += (q == c) ? 1u : 0u;
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const uint32_t v = __reduce_add_sync(0xFFFFFFFFu, mine[q]);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&local[q], v);
  }
  if (!alone) griddep_wait();
  griddep_launch_dependents();
  __syncthreads();
  if (threadIdx.x < 6) {
    if (alone) counts[threadIdx.x] = local[threadIdx.x];
    else if (local[threadIdx.x]) atomicAdd(&counts[threadIdx.x], (unsigned long long)local[threadIdx.x]);
  }
}

inline unsigned grid_for(int64_t items, int threads, int sm_count, int per_sm) {
  const int64_t want = (items + threads - 1) / threads;
  const int64_t cap = (int64_t)sm_count * per_sm;
  return (unsigned)(want < 1 ? 1 : (want < cap ? want : cap));
}

}  // namespace stats
}  // namespace bro
