// Offline weight decomposition + packing (Section 5, Stage 2 -> Stage 1 -> Stage 3) and its exporter.
//
// One launch for rows up to 16384 long (`pack_kernel<FUSED>`): a CTA takes 16 rows x 2048 K, the CTAs of a thread-block cluster
// share the rows' K range, and a thread takes 128 K of one row -- 16 S-Vectors, whole Q-Vectors, so that scales need no
// exchange between threads and everything a thread produces is 4 to 16 contiguous bytes of the layout; the lanes of a warp
// are 16 consecutive rows, whose pieces make whole 128-byte lines.  W is read once, through shared memory (rows 4112 B
// apart: the 16-byte reads of 8 lanes then touch all banks once).  What needs the whole row -- the exponent (or fp32 scale) of
// the outliers, for two-level scaling the inlier factor -- is found in a first pass over the staged rows and exchanged
// through distributed shared memory.  Longer rows: `row_scale_kernel` finds it and the same kernel follows without clusters.
//
// What bounds it: the integer pipe (selections on packed keys instead of index loops took it from ~350 instructions per S-Vector
// over two passes to some 140), DRAM is at 30 %.  11008 x 4096, 1:8 + pair-wise 4:8: 189 us as one kernel with a CTA per row and a
// thread per S-Vector scattering bytes -> 20 + 42 us with the row scales in a launch of their own -> 49 us -> 42 us with the
// pairs picked by two minima and two maxima instead of six comparisons and the choices kept from the first pass.  4096 x 11008,
// 1:8 + 6:8 with channel weights: 98 us choosing in both passes -> 67.  Loops of four S-Vectors (first pass) and of one Q-Vector
// (second) instead of 16 and 4 in a row, each warp starting on its own part of the tile, the rows' maxima exchanged by counted stores
// instead of a cluster barrier, whole calls: 4096 x 11008 78.5 -> 74.9, without channel weights 64.4 -> 55.8; 16384 x 4096 with E4M3 scales
// 79.8 -> 74.7; 11008 x 4096 56.0 -> 55.6 (kernel 43.6 -> 43; with the cluster barrier and the loops only, 1 us more).
#include <cstring>
#include <type_traits>
#include <mutex>
#include <condition_variable>

#include "../../include/sdq_diag.h"
#include "sdq_codec.cuh"
#include "sdq_internal.h"
#include "sdq_layout.h"
#include "sdq_plain.h"
#include "sdq_ptx.cuh"

namespace sdq {

// ---- selections on one S-Vector of 8 weights, r[j] = elements 2 j (low half) and 2 j + 1 -----------------------------
// Ranking keys, larger = more significant.  By magnitude: magnitude bits << 16 | (7 - i), so that plain maxima resolve ties
// to the lower index.  Weighted (c != nullptr, the product |w| * c[k], one fp32 multiply): the product's bit pattern;
// comparisons resolve ties.
template <bool WGT>
__device__ __forceinline__ void rank_keys(const uint32_t (&r)[4], const float* __restrict__ c, int (&k)[8]) {
  if constexpr (!WGT) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t a = r[j] & 0x7FFF7FFFu;
      k[2 * j] = (int)prmt(a, (uint32_t)(7 - 2 * j), 0x1054u);
      k[2 * j + 1] = (int)((a & 0xFFFF0000u) | (uint32_t)(6 - 2 * j));
    }
  } else {
    const float4 c0 = __ldg(reinterpret_cast<const float4*>(c)), c1 = __ldg(reinterpret_cast<const float4*>(c) + 1);
    const float cc[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      k[2 * j] = __float_as_int(__fmul_rn(__uint_as_float((r[j] & 0x7FFFu) << 16), cc[2 * j]));
      k[2 * j + 1] = __float_as_int(__fmul_rn(__uint_as_float(r[j] & 0x7FFF0000u), cc[2 * j + 1]));
    }
  }
}
// position of the largest key of k[B .. E), ties to the lower index
template <bool WGT, int B, int E>
__device__ __forceinline__ int arg_max(const int (&k)[8]) {
  if constexpr (!WGT) {
    int best = __vimax3_s32(k[B], k[B + 1], k[B + 2]);
    if constexpr (E - B == 8) best = __vimax3_s32(__vimax3_s32(k[B + 4], k[B + 5], k[B + 6]), k[B + 7], best);
    return 7 - (max(best, k[B + 3]) & 7);
  } else {
    int best = k[B], at = B;
#pragma unroll
    for (int i = B + 1; i < E; ++i)
      if (k[i] > best) { best = k[i]; at = i; }
    return at;
  }
}
// position of the smallest key, ties to the higher index (the last in rank order)
template <bool WGT>
__device__ __forceinline__ int arg_min(const int (&k)[8]) {
  if constexpr (!WGT) {
    return 7 - (min(__vimin3_s32(__vimin3_s32(k[0], k[1], k[2]), k[3], k[4]), __vimin3_s32(k[5], k[6], k[7])) & 7);
  } else {
    int best = k[0], at = 0;
#pragma unroll
    for (int i = 1; i < 8; ++i)
      if (k[i] <= best) { best = k[i]; at = i; }
    return at;
  }
}
// Stage 2: positions of the outliers, ascending (-1: none).  order_mask turns the ranking round when the least significant
// values are taken (SDQ_ORDER_SMALL); sv4: S-Vectors of 4, one outlier in each half.
template <bool WGT, int OUTN>
__device__ __forceinline__ void pick_outliers(const int (&key)[8], int order_mask, bool sv4, int& o0, int& o1) {
  o0 = o1 = -1;
  if constexpr (OUTN > 0) {
    int k[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) k[i] = key[i];
    if (order_mask)
#pragma unroll
      for (int i = 0; i < 8; ++i) k[i] ^= order_mask;
    if (OUTN == 2 && sv4) {
      o0 = arg_max<WGT, 0, 4>(k);
      o1 = arg_max<WGT, 4, 8>(k);
    } else {
      o0 = arg_max<WGT, 0, 8>(k);
      if constexpr (OUTN == 2) {
#pragma unroll
        for (int i = 0; i < 8; ++i) k[i] = i == o0 ? -1 : k[i];
        o1 = arg_max<WGT, 0, 8>(k);
        const int lo = min(o0, o1);
        o1 = max(o0, o1);
        o0 = lo;
      }
    }
  }
}
// element `at` of the S-Vector as a float
__device__ __forceinline__ float pick_value(const uint32_t (&r)[4], int at) {
  const uint32_t sel = (uint32_t)(at & 3) * 0x2200u + 0x1000u;      // its two bytes, to the upper half
  return __uint_as_float(((at & 4) ? prmt(r[2], r[3], sel) : prmt(r[0], r[1], sel)) & 0xFFFF0000u);
}
// bf16 bits of |x|
__device__ __forceinline__ uint32_t magnitude(float x) { return __float_as_uint(x) << 1 >> 17; }
__device__ __forceinline__ uint32_t larger_half(uint32_t x) { return max(x & 0xFFFFu, x >> 16); }
// r with position `at` zeroed (at = -1: nothing)
__device__ __forceinline__ void zero_at(uint32_t (&r)[4], int at) {
  const uint32_t keep = (at & 1) ? 0x0000FFFFu : 0xFFFF0000u;
#pragma unroll
  for (int j = 0; j < 4; ++j) r[j] &= (at >> 1) == j ? keep : 0xFFFFFFFFu;
}
// r with the positions of the set `gone` (bit i: position i) zeroed: bit i of four goes to the top of byte i, whose sign is
// then spread over a half word
__device__ __forceinline__ void zero_set(uint32_t (&r)[4], uint32_t gone) {
  const uint32_t lo = (gone & 15u) * 0x10204080u, hi = ((gone >> 4) & 15u) * 0x10204080u;
  r[0] &= ~prmt(lo, 0u, 0x9988u);
  r[1] &= ~prmt(lo, 0u, 0xBBAAu);
  r[2] &= ~prmt(hi, 0u, 0x9988u);
  r[3] &= ~prmt(hi, 0u, 0xBBAAu);
}
// Stage 1, pair-wise 4:8: the 2 pairs (of 4) with the largest summed significance among the non-outliers (x: outliers
// zeroed), largest first, ties to the lower index.
// Returns the two pairs in ascending order and the pattern nibble j0 | j1 << 2.
template <bool WGT>
__device__ __forceinline__ void pick_pairs(const uint32_t (&x)[4], const int (&key)[8], int o0, int o1, uint32_t& w0, uint32_t& w1, uint32_t& nibble) {
  float s[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if constexpr (WGT) {
      const float a = (2 * j == o0 || 2 * j == o1) ? 0.0f : __int_as_float(key[2 * j]);
      const float b = (2 * j + 1 == o0 || 2 * j + 1 == o1) ? 0.0f : __int_as_float(key[2 * j + 1]);
      s[j] = __fadd_rn(a, b);
    } else {
      s[j] = __fadd_rn(fabsf(__uint_as_float(x[j] << 16)), fabsf(__uint_as_float(x[j] & 0xFFFF0000u)));
    }
  }
  // the weaker of the first two beats the stronger of the last two; or the other way round; else one of each
  const bool first = fminf(s[0], s[1]) >= fmaxf(s[2], s[3]), last = fminf(s[2], s[3]) > fmaxf(s[0], s[1]);
  const bool k0 = first || s[0] >= s[1], k2 = !last && s[2] >= s[3];
  w0 = last ? x[2] : (k0 ? x[0] : x[1]);
  w1 = first ? x[1] : (k2 ? x[2] : x[3]);
  nibble = (last ? 2u : (k0 ? 0u : 1u)) | (first ? 4u : (k2 ? 8u : 12u));
}
// Stage 1 for the patterns stored dense: the set of positions that hold +0 -- the outliers and, among the others, all but the
// keep_in most significant (of every 8, or of every 4 with grp4).  k: ranking keys.
template <bool WGT, int OUTN>
__device__ __forceinline__ uint32_t dropped_set(int (&k)[8], int o0, int o1, int keep_in, bool grp4, int order_mask) {
  uint32_t m = 0;
  if (OUTN > 0) m |= 1u << o0;
  if (OUTN > 1) m |= 1u << o1;
  if (!grp4 && keep_in + OUTN >= 7) {
    if (keep_in + OUTN == 7) {
      // exactly one value more: the last in rank order, which is no outlier unless these are the least significant
      if (OUTN > 0 && order_mask)
#pragma unroll
        for (int i = 0; i < 8; ++i) k[i] = (m >> i) & 1u ? 0x7FFFFFFF : k[i];
      m |= 1u << arg_min<WGT>(k);
    }
  } else {
    if (OUTN > 0)
#pragma unroll
      for (int i = 0; i < 8; ++i) k[i] = (m >> i) & 1u ? -1 : k[i];
    if (grp4 && keep_in == 2) {                     // two of four, as in pick_pairs (11008 x 4096, 2:4: 71.5 us ranking all four -> 65.3)
      m = 0xFFu;
#pragma unroll
      for (int g = 0; g < 8; g += 4) {
        const bool first = min(k[g], k[g + 1]) >= max(k[g + 2], k[g + 3]), last = min(k[g + 2], k[g + 3]) > max(k[g], k[g + 1]);
        const uint32_t one = k[g] >= k[g + 1] ? 1u : 2u, two = k[g + 2] >= k[g + 3] ? 4u : 8u;
        m ^= (first ? 3u : (last ? 12u : one | two)) << g;
      }
      return m;
    }
    uint32_t rank = 0;                              // nibble i: how many come before position i
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = i + 1; j < 8; ++j) {
        if ((i >> 2) == (j >> 2) || !grp4) rank += k[i] >= k[j] ? (1u << (4 * j)) : (1u << (4 * i));
      }
    m = ((rank + (uint32_t)(8 - keep_in) * 0x11111111u) >> 3) & 0x11111111u;
    m = (m | m >> 3) & 0x03030303u;                 // every fourth bit -> 8 bits
    m = (m | m >> 6) & 0x000F000Fu;
    m = (m | m >> 12) & 0xFFu;
  }
  return m;
}

// the next 16 bits of eight bytes, the next word of four: after four of them the first is the lowest
__device__ __forceinline__ void queue16(uint32_t (&q)[2], uint32_t v) { q[0] = prmt(q[0], q[1], 0x5432u); q[1] = prmt(q[1], v, 0x5432u); }
__device__ __forceinline__ void queue32(uint32_t (&q)[4], uint32_t v) { q[0] = q[1]; q[1] = q[2]; q[2] = q[3]; q[3] = v; }

struct PackParams {
  const __nv_bfloat16* W;
  int64_t N, K, ldw;
  const float* colw;           // per-channel weights of the product metric, or nullptr
  uint8_t* blob;
  PackedOffsets off;
  uint32_t* nonfinite;         // host-visible word, set to 1 when a weight (or channel weight) is not finite
  uint32_t* gave_up;           // ... when a wait for the rows' maxima gave up
  uint32_t polls;              // ... which it does after that many
  int out_n, keep_in, order_mask;
  int sv4, elem, ue, i8, b32, ceil_rule;
};

// outlier scale of a row from its largest outlier: exponent, or the bit pattern of the fp32 scale amax / 127 (int8)
__device__ __forceinline__ int row_scale(const PackParams& p, uint32_t omax) {
  const float a = bf16_bits_to_float(omax);
  return p.i8 ? __float_as_int(int8_scale(a)) : fp8_scale_exp(a);
}
// exponent of the row's inlier factor 2^t (two-level scaling)
__device__ __forceinline__ int row_factor(const PackParams& p, uint32_t imax) { return p.ue ? fp8_scale_exp(bf16_bits_to_float(imax)) : 0; }
__device__ __forceinline__ void store_row_scale(const PackParams& p, int64_t n, uint32_t omax, uint32_t imax) {
  const int e = row_scale(p, omax), tw = row_factor(p, imax);
  reinterpret_cast<int32_t*>(p.blob + p.off.osexp)[n] = e;
  reinterpret_cast<int32_t*>(p.blob + p.off.wtexp)[n] = tw;
  // the accumulator of a row is kept in units of 2^tw (the inlier scale codes leave that factor out), so the outlier
  // row scale is 2^(e - tw); the GEMM's epilogue multiplies the factor back in
  const uint32_t c = p.i8 ? 127u : (uint32_t)min(max(e - tw + 127, 0), 254);    // (int8: the epilogue applies the scales)
  *reinterpret_cast<uint32_t*>(p.blob + p.off.sfa_out + (size_t)(n / TILE_ROWS) * SF_ATOM_BYTES + sf_off((uint32_t)(n % TILE_ROWS), 0)) = c * 0x01010101u;
}
// the self-describing header, zero-filled to its reservation, by one block of at least 64 threads
__device__ __forceinline__ void store_header(const PackParams& p, const BlobHeader& hdr) {
  if (threadIdx.x < HEADER_BYTES / 4)
    reinterpret_cast<uint32_t*>(p.blob)[threadIdx.x] = threadIdx.x < sizeof(BlobHeader) / 4 ? reinterpret_cast<const uint32_t*>(&hdr)[threadIdx.x] : 0u;
}
// the choices of one S-Vector: outlier positions and values, pattern nibble and the two pairs that stay, outlier positions at +0
template <bool WGT, int OUTN>
__device__ __forceinline__ void choose_pairs(const PackParams& p, uint32_t (&r)[4], const float* c, int& o0, int& o1, float& f0, float& f1,
                                             uint32_t& w0, uint32_t& w1, uint32_t& nibble) {
  int k[8];
  rank_keys<WGT>(r, c, k);
  pick_outliers<WGT, OUTN>(k, p.order_mask, p.sv4 != 0, o0, o1);
  f0 = OUTN > 0 ? pick_value(r, o0) : 0.0f;
  f1 = OUTN > 1 ? pick_value(r, o1) : 0.0f;
  if constexpr (OUTN > 0) zero_at(r, o0);
  if constexpr (OUTN > 1) zero_at(r, o1);
  pick_pairs<WGT>(r, k, o0, o1, w0, w1, nibble);
}
// its largest outlier (and, two-level scaling, the largest inlier that stays), into running maxima
template <bool WGT, int OUTN>
__device__ __forceinline__ void group_maxima(const PackParams& p, uint32_t (&r)[4], const float* c, uint32_t& omax, uint32_t& imax) {
  int k[8], o0, o1;
  rank_keys<WGT>(r, c, k);
  pick_outliers<WGT, OUTN>(k, p.order_mask, p.sv4 != 0, o0, o1);
  if constexpr (OUTN > 0) omax = max(omax, magnitude(pick_value(r, o0)));
  if constexpr (OUTN > 1) omax = max(omax, magnitude(pick_value(r, o1)));
  if (p.ue) {                                            // pair-wise pattern
    if constexpr (OUTN > 0) zero_at(r, o0);
    if constexpr (OUTN > 1) zero_at(r, o1);
    uint32_t w0, w1, nibble;
    pick_pairs<WGT>(r, k, o0, o1, w0, w1, nibble);
    imax = max_abs2(max_abs2(imax, w0), w1);
  }
}
// two packed running maxima of the magnitudes
__device__ __forceinline__ uint32_t max_magnitudes(uint32_t m, const uint32_t (&r)[4]) {
  return max_abs2(max_abs2(max_abs2(max_abs2(m, r[0]), r[1]), r[2]), r[3]);
}
__device__ __forceinline__ bool bad_weight(float c) { return !(c >= 0.0f && c <= 3.4028234663852886e38f); }

// ---- what a row needs as a whole (K > 16384): per row the outlier scale, the inlier factor of two-level scaling, non-finite check.  One warp per row.
// SELECT = false: the outliers hold the row's largest magnitude, so nothing has to be selected (magnitude metric, most
// significant values first, no two-level scaling).
template <bool SELECT, bool WGT, int OUTN>
__global__ void __launch_bounds__(256)
row_scale_kernel(const PackParams p, const BlobHeader hdr)
{
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n = (int64_t)blockIdx.x * 8 + warp;               // N is a multiple of 128
  if (blockIdx.x == 0) store_header(p, hdr);
  const uint4* row = reinterpret_cast<const uint4*>(p.W + n * p.ldw);
  const int G = (int)(p.K / 8);
  uint32_t all2 = 0, omax = 0, imax = 0, bad = 0;                 // all2: two packed running maxima of the magnitudes
  if constexpr (!SELECT) {
    int g = (int)lane;
    for (; g + 96 < G; g += 128) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = __ldg(row + g + 32 * u);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t r[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
        all2 = max_magnitudes(all2, r);
      }
    }
    for (; g < G; g += 32) {
      const uint4 v = __ldg(row + g);
      const uint32_t r[4] = {v.x, v.y, v.z, v.w};
      all2 = max_magnitudes(all2, r);
    }
    omax = larger_half(all2);
    bad = omax >= 0x7F80u;
  } else {
#pragma unroll 2
    for (int g = (int)lane; g < G; g += 32) {
      const uint4 v = __ldg(row + g);
      uint32_t r[4] = {v.x, v.y, v.z, v.w};
      all2 = max_magnitudes(all2, r);
      if constexpr (WGT) {
#pragma unroll
        for (int i = 0; i < 8; ++i) bad |= bad_weight(__ldg(p.colw + 8 * (int64_t)g + i));
      }
      group_maxima<WGT, OUTN>(p, r, WGT ? p.colw + 8 * (int64_t)g : nullptr, omax, imax);
    }
    bad |= larger_half(all2) >= 0x7F80u;
    imax = larger_half(imax);
  }
  omax = __reduce_max_sync(0xffffffffu, omax);
  imax = __reduce_max_sync(0xffffffffu, imax);
  bad = __any_sync(0xffffffffu, bad != 0);
  if (lane == 0) {
    if (bad) *reinterpret_cast<volatile uint32_t*>(p.nonfinite) = 1u;
    store_row_scale(p, n, OUTN ? omax : 0u, imax);
  }
}

// ---- the packer
constexpr int PK_THREADS = 256, PK_ROWS = 16, PK_K = 2048;
constexpr int PK_PITCH = PK_K * 2 + 16;                  // bytes between rows of the staged tile
constexpr int PK_SMEM = PK_ROWS * PK_PITCH;              // 65792: three CTAs per SM

template <bool DENSE, bool WGT, int OUTN, bool FUSED>
__global__ void __launch_bounds__(PK_THREADS, 3)
pack_kernel(const PackParams p, const BlobHeader hdr)
{
  extern __shared__ __align__(16) uint8_t tile[];
  __shared__ uint32_t s_part[2][PK_ROWS][PK_ROWS + 1];   // [outliers / inliers][row][128-K chunk]: largest magnitudes
  __shared__ uint32_t s_all[2][8][PK_ROWS];              // [outliers / inliers][cluster rank][row], pushed by their owners
  __shared__ uint64_t s_bar;                             // ... all of which have arrived
  const uint32_t tid = threadIdx.x;
  const int T1 = (int)(p.K / K1), T2 = T1 / 2;
  const int cx = (int)((p.K + PK_K - 1) / PK_K), rank = (int)(blockIdx.x % (uint32_t)cx);   // FUSED: a cluster is the cx CTAs of these rows
  const bool first_rows = blockIdx.x < (uint32_t)cx;
  // (waited for before the first store into another CTA's shared memory: every CTA of the cluster has started by then; the fence
  // releases the barrier's set-up, and a releasing arrival would be a memory barrier for every warp)
  if constexpr (FUSED) {
    if (tid == 0) {
      ptx::mbar_init(&s_bar, 1);
      ptx::fence_barrier_init();
      ptx::mbar_expect_tx(&s_bar, (uint32_t)cx * 2u * PK_ROWS * 4u);
    }
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  }
  const int64_t n_first = (int64_t)(blockIdx.x / (uint32_t)cx) * PK_ROWS;
  {
    // 256 threads x 16 B = the 4096 B of one row per round
    const int64_t k = (int64_t)rank * PK_K + tid * 8;
    const uint8_t* src = reinterpret_cast<const uint8_t*>(p.W + n_first * p.ldw + k);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tile) + tid * 16;
    if (k < p.K) {
#pragma unroll
      for (int i = 0; i < PK_ROWS; ++i)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * PK_PITCH), "l"(src + (int64_t)i * 2 * p.ldw) : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  const uint32_t row = tid & 15u, ch = tid >> 4;         // this thread's row and 128-K chunk of the tile
  const int kc = rank * 16 + (int)ch;                    // ... and of the matrix
  const bool on = kc < T1;
  const int64_t n = n_first + row;
  uint8_t* mine = tile + row * PK_PITCH + ch * 256;
  const float* colw = WGT ? p.colw + (int64_t)kc * K1 : nullptr;
  __syncwarp();                                          // (a warp has loaded what its own threads read)

  // ---- first pass: the choices, the row's largest outlier (and inlier), non-finite check.
  // Pair-wise: everything is chosen here and the S-Vector's 16 bytes in the tile become what is left to encode, the two pairs that
  // stay and the outliers' values; positions and pattern nibbles are collected in registers, as the layout wants them (11008 x 4096
  // against choosing in the second pass: 1:8 42.3 and 45.7 us, with E4M3 scales, where both passes have to choose, 49 and 74).
  // Stored dense, with channel weights: the same, but the values stay where they are and the sets of dropped positions are
  // collected (4096 x 11008, 1:8 + 6:8: 67 and 98).  Dense by magnitude: the outliers, if the most significant, hold the row's
  // largest magnitude, this pass has nothing to choose and leaves it to the second.
  constexpr bool CHOSEN = !DENSE || WGT;
  // trips of either pass' loop in a row: one, since straight-line code waits for instructions; four where the row scales come from a launch
  // of their own, the inliers are pair-wise and the choices, made by magnitude or of two outliers or none, short (28672 x 8192, all in
  // a row, rolled -> so: 1:8 250 -> 248 us, E4M3 scales without outliers 189 -> 183, 2:8 with channel weights 607 -> 589; the others would lose: 1:8 + 6:8
  // 236 -> 259, 1:8 with channel weights 361 -> 370)
  constexpr int UNROLL = FUSED || DENSE || (WGT && OUTN == 1) ? 1 : 4;
  [[maybe_unused]] uint32_t c_o0[2] = {0, 0}, c_o1[2] = {0, 0}, c_nib[2] = {0, 0}, c_gone[4] = {0, 0, 0, 0};
  uint32_t all2 = 0, omax = 0, imax = 0, bad = 0;        // all2, imax: packed running maxima
  if constexpr (CHOSEN) {
    const bool look_at_all = WGT || OUTN == 0 || p.order_mask;    // for non-finite values: otherwise they are outliers
    if (on) {
#pragma unroll (UNROLL)
      for (int t = 0; t < 4; ++t) {                      // four S-Vectors a trip
        uint32_t n_o0 = 0, n_o1 = 0, n_nib = 0, n_gone = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint4* at = reinterpret_cast<uint4*>(mine) + 4 * t + i;
          const uint4 v = *at;
          uint32_t r[4] = {v.x, v.y, v.z, v.w};
          const float* c = WGT ? colw + 8 * (4 * t + i) : nullptr;
          int o0, o1;
          float f0, f1;
          if (look_at_all) all2 = max_magnitudes(all2, r);
          if constexpr (!DENSE) {
            uint32_t w0, w1, nibble;
            choose_pairs<WGT, OUTN>(p, r, c, o0, o1, f0, f1, w0, w1, nibble);
            if (p.ue) imax = max_abs2(max_abs2(imax, w0), w1);
            *at = make_uint4(w0, w1, __float_as_uint(f0), __float_as_uint(f1));
            n_nib |= nibble << (4 * i);
          } else {
            int k[8];
            rank_keys<WGT>(r, c, k);
            pick_outliers<WGT, OUTN>(k, p.order_mask, p.sv4 != 0, o0, o1);
            f0 = OUTN > 0 ? pick_value(r, o0) : 0.0f;
            f1 = OUTN > 1 ? pick_value(r, o1) : 0.0f;
            n_gone |= dropped_set<WGT, OUTN>(k, o0, o1, p.keep_in, p.sv4 || p.elem, p.order_mask) << (8 * i);
          }
          if constexpr (OUTN > 0) { omax = max(omax, magnitude(f0)); n_o0 |= (uint32_t)o0 << (4 * i); }
          if constexpr (OUTN > 1) { omax = max(omax, magnitude(f1)); n_o1 |= (uint32_t)o1 << (4 * i); }
        }
        queue16(c_nib, n_nib);
        queue16(c_o0, n_o0);
        queue16(c_o1, n_o1);
        queue32(c_gone, n_gone);
      }
    }
  }
  int e, tw;
  if constexpr (FUSED) {
    if (on) {
      if constexpr (!CHOSEN) {
#pragma unroll 4
        for (int i = 0; i < 16; ++i) {
          const uint4 v = *reinterpret_cast<const uint4*>(mine + i * 16);
          uint32_t r[4] = {v.x, v.y, v.z, v.w};
          all2 = max_magnitudes(all2, r);
          if (p.order_mask) group_maxima<false, OUTN>(p, r, nullptr, omax, imax);
        }
        if (!p.order_mask) omax = larger_half(all2);
      }
      imax = larger_half(imax);
      bad = max(omax, larger_half(all2)) >= 0x7F80u;
      if (WGT && first_rows)                             // the channel weights are the same for every row
        for (int i = (int)row; i < K1; i += PK_ROWS) bad |= bad_weight(__ldg(colw + i));
    }
    if (bad) *reinterpret_cast<volatile uint32_t*>(p.nonfinite) = 1u;
    s_part[0][row][ch] = OUTN ? omax : 0u;
    s_part[1][row][ch] = imax;
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    __syncthreads();
    if (tid < 2 * PK_ROWS) {
      const uint32_t which = tid >> 4, r = tid & 15u;
      uint32_t m = 0;
#pragma unroll
      for (int c = 0; c < 16; ++c) m = max(m, s_part[which][r][c]);
      const uint32_t mine_at = ptx::smem_u32(&s_all[which][rank][r]), bar = ptx::smem_u32(&s_bar);
      for (uint32_t peer = 0; peer < (uint32_t)cx; ++peer) ptx::st_async_u32(ptx::mapa_u32(mine_at, peer), m, ptx::mapa_u32(bar, peer));
    }
    // counted stores, as in the activation quantizer: a CTA waits for what it needs and for nothing else, and does not leave before all
    // pushes to it have arrived.  Where the wait gives up, peers may still push: this CTA stays until they have, or have given up as well
    if (__any_sync(0xffffffffu, !ptx::mbar_wait_cluster(&s_bar, 0, p.polls))) {
      *reinterpret_cast<volatile uint32_t*>(p.gave_up) = 1u;
      ptx::cluster_wait_for_others();
      (void)ptx::mbar_wait_cluster(&s_bar, 0);             // (what was sent last is still on its way)
    }
    omax = imax = 0;
    for (int c = 0; c < cx; ++c) { omax = max(omax, s_all[0][c][row]); imax = max(imax, s_all[1][c][row]); }
    if (rank == 0 && ch == 0) store_row_scale(p, n, omax, imax);
    if (rank == 0 && first_rows) store_header(p, hdr);
    e = row_scale(p, omax);
    tw = row_factor(p, imax);
  } else {
    e = reinterpret_cast<const int32_t*>(p.blob + p.off.osexp)[n];
    tw = p.ue ? reinterpret_cast<const int32_t*>(p.blob + p.off.wtexp)[n] : 0;
  }
  if (!on) return;

  // ---- second pass
  const int rt = (int)(n / TILE_ROWS), k2 = kc >> 1;
  const uint32_t r = (uint32_t)(n % TILE_ROWS), h = (uint32_t)kc & 1u;   // row of the row tile, 128-K half of the record
  const bool b32 = DENSE || p.b32 != 0;
  uint8_t* wi = p.blob + p.off.wi + ((size_t)rt * T2 + k2) * (size_t)wi_bytes(b32, DENSE);
  uint8_t* wo = p.blob + p.off.wo + ((size_t)rt * T1 + kc) * (size_t)WO_BYTES;
  uint8_t* wc = p.blob + p.off.wc + ((size_t)rt * T1 + kc) * (size_t)wc_bytes(OUTN);
  const float s8 = pow2_neg(e);
  const uint32_t core = (r >> 3) * 256 + (r & 7) * 16;   // this row inside a K-block of an A operand

  uint32_t in_word[2][2];                                // pair-wise inliers: the 64-K half's codes, two S-Vectors per word
  uint32_t sc = 0;                                       // scale bytes of the 128 K
  uint32_t codes[4] = {0, 0, 0, 0}, sels[4] = {0, 0, 0, 0}, metas[4] = {0, 0, 0, 0};   // outlier bytes of the 128 K
  uint32_t kept[16];                                     // pair-wise inliers of a Q-Vector of 64 K, outlier positions zeroed
  uint32_t qmax2 = 0;                                    // packed running maximum of the Q-Vector
  // (like the first pass: as straight-line code the two took a fifth of the warps' time in waits for instructions)
  constexpr int TRIP = DENSE ? 1 : 2;                    // blocks a trip (pair-wise: a Q-Vector of 64 K)
#pragma unroll (UNROLL)
  for (int b0 = 0; b0 < 4; b0 += TRIP) {
    [[maybe_unused]] const uint32_t w_o0 = b0 < 2 ? c_o0[0] : c_o0[1], w_o1 = b0 < 2 ? c_o1[0] : c_o1[1];
#pragma unroll
    for (int bi = 0; bi < TRIP; ++bi) {                   // blocks of 4 S-Vectors (32 K)
      const int b = b0 + bi, odd = DENSE ? b & 1 : bi;
      uint32_t ocode[4], ocode1[4], opos[4], opos1[4];
      uint32_t dense_codes[4], dval[16];
      [[maybe_unused]] uint32_t emeta[2] = {0, 0};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 v = *reinterpret_cast<const uint4*>(mine + (4 * b + i) * 16);
        uint32_t x[4] = {v.x, v.y, v.z, v.w};
        [[maybe_unused]] int k[8];
        int o0, o1;
        if constexpr (CHOSEN) {
          o0 = (int)((w_o0 >> (16 * odd + 4 * i)) & 7u);
          o1 = (int)((w_o1 >> (16 * odd + 4 * i)) & 7u);
        } else {
          rank_keys<false>(x, nullptr, k);
          pick_outliers<false, OUTN>(k, p.order_mask, p.sv4 != 0, o0, o1);
        }
        // Stage 3, outliers: E4M3 codes of w / 2^e, or int8 codes of w / s
        if constexpr (OUTN > 0) {
          const float f = DENSE ? pick_value(x, o0) : __uint_as_float(x[2]);
          ocode[i] = !DENSE && p.i8 ? int8_code(f, __int_as_float(e)) : e4m3x1(f * s8);
          opos[i] = (uint32_t)o0;
        }
        if constexpr (OUTN > 1) {
          const float f = DENSE ? pick_value(x, o1) : __uint_as_float(x[3]);
          ocode1[i] = !DENSE && p.i8 ? int8_code(f, __int_as_float(e)) : e4m3x1(f * s8);
          opos1[i] = (uint32_t)o1;
        }
        if constexpr (!DENSE) {
          kept[2 * (4 * odd + i)] = x[0];
          kept[2 * (4 * odd + i) + 1] = x[1];
          qmax2 = max_abs2(max_abs2(qmax2, x[0]), x[1]);
        } else {
          uint32_t gone;
          if constexpr (CHOSEN) gone = (c_gone[0] >> (8 * i)) & 255u;
          else gone = dropped_set<false, OUTN>(k, o0, o1, p.keep_in, p.sv4 || p.elem, p.order_mask);
          zero_set(x, gone);
          qmax2 = max_magnitudes(qmax2, x);
#pragma unroll
          for (int j = 0; j < 4; ++j) dval[4 * i + j] = x[j];
          if (p.elem) {
            // the kept indices (two ascending 2-bit values per group of 4) are only needed by the exporter.  Exactly two of a
            // group's four bits are set: the nibble that such a set stands for, looked up
            const uint32_t lo = (~gone) & 15u, hi = (~gone >> 4) & 15u;
            const uint32_t ml = ((lo & 8u) ? 0x000E0DC0u : 0x09804000u) >> (4 * (lo & 7u)), mh = ((hi & 8u) ? 0x000E0DC0u : 0x09804000u) >> (4 * (hi & 7u));
            emeta[i >> 1] |= ((ml & 15u) | ((mh & 15u) << 8)) << (16 * (i & 1));
          }
        }
      }

      // ---- Stage 3, inliers
      if constexpr (DENSE) {
        const uint32_t c = e8m0_scale_code_bf16(larger_half(qmax2), p.ceil_rule != 0);
        const float inv = pow2_inv_e8m0(c);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float f[8];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            f[2 * j] = __uint_as_float(dval[4 * i + j] << 16) * inv;
            f[2 * j + 1] = __uint_as_float(dval[4 * i + j] & 0xFFFF0000u) * inv;
          }
          dense_codes[i] = e2m1x8(f);
        }
        if (p.elem) *reinterpret_cast<uint2*>(p.blob + p.off.emeta + (size_t)n * (size_t)(p.K / 4) + (kc * 16 + 4 * b) * 2) = make_uint2(emeta[0], emeta[1]);
        // 16 code bytes per 32 K: K-block (64 K) 2 h + b / 2 of the record, chunk b & 1
        *reinterpret_cast<uint4*>(wi + (2 * h + (b >> 1)) * 4096 + core + odd * 128) = make_uint4(dense_codes[0], dense_codes[1], dense_codes[2], dense_codes[3]);
        sc |= c << (8 * b);
        qmax2 = 0;
      } else if (odd || b32) {
        // a Q-Vector is complete: 64 K (both blocks of the half) or 32 K (this one)
        const uint32_t key = larger_half(qmax2);
        const uint32_t c = p.ue ? ue4m3_scale_code(bf16_bits_to_float(key) * pow2_neg(tw), key != 0) : e8m0_scale_code_bf16(key, p.ceil_rule != 0);
        const float inv = p.ue ? ue4m3_scale_inverse(max(c, 1u)) : pow2_inv_e8m0(c);
#pragma unroll
        for (int hb = 0; hb < 2; ++hb) {                   // 32-K block of the half
          if (hb != odd && b32) continue;              // (one scale per 64 K: both now)
#pragma unroll
          for (int i = 0; i < 2; ++i) {                    // two S-Vectors per code word
            float f[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t w = kept[8 * hb + 4 * i + j];
              const float lo = __uint_as_float(w << 16), hi = __uint_as_float(w & 0xFFFF0000u);
              if (p.ue) {
                // (an outlier's position stays +0; the quotient of a dropped one is +0 as well)
                f[2 * j] = small_quotient(lo * pow2_neg(tw), inv);
                f[2 * j + 1] = small_quotient(hi * pow2_neg(tw), inv);
              } else {
                f[2 * j] = lo * inv;
                f[2 * j + 1] = hi * inv;
              }
            }
            in_word[hb][i] = p.ue && c == 0 ? 0u : e2m1x8(f);
          }
        }
        if (b32) { sc |= c << (8 * b); }
        else sc |= c << (8 * (b >> 1));
        qmax2 = 0;
      }
      if constexpr (!DENSE) {
        if (odd) {
          // 16 code bytes per 64 K (K-block h, chunk b / 2)
          *reinterpret_cast<uint4*>(wi + h * 4096 + core + (b >> 1) * 128) = make_uint4(in_word[0][0], in_word[0][1], in_word[1][0], in_word[1][1]);
        }
      }

      // ---- outliers of the 4 S-Vectors: compact record, and the 2:4 embedding the sparse FP8 path consumes (per 4 K two
      // ascending slot indices, unused slots hold +0)
      if constexpr (OUTN == 1) {
        // per S-Vector: position ps (0..7) sits in group of 4 number ps >> 2 at p = ps & 3, whose slots are (p, 3), the value
        // first, or (0, 3), the value second, when p = 3; the other group has slots (0, 1).  Metadata bytes and byte shifts
        // come from 8-entry tables looked up by byte-permutes, the four position nibbles being the selector.
        queue32(codes, ocode[0] | (ocode[1] << 8) | (ocode[2] << 16) | (ocode[3] << 24));
        const uint32_t sel = CHOSEN ? (w_o0 >> (16 * odd)) & 0xFFFFu : opos[0] | (opos[1] << 4) | (opos[2] << 8) | (opos[3] << 12);
        const uint32_t sh = __byte_perm(0x08000000u, 0x18101010u, sel);
        queue32(metas, __byte_perm(0x4C4E4D4Cu, 0xC4E4D4C4u, sel));
        queue32(sels, sel);
        *reinterpret_cast<uint4*>(wo + (b >> 1) * 4096 + core + odd * 128) =
            make_uint4(ocode[0] << (sh & 31u), ocode[1] << ((sh >> 8) & 31u), ocode[2] << ((sh >> 16) & 31u), ocode[3] << (sh >> 24));
      } else if constexpr (OUTN == 2) {
        uint32_t st[4], meta = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int o0 = (int)opos[i], o1 = (int)opos1[i];
          st[i] = 0;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const bool in0 = (o0 >> 2) == q, in1 = (o1 >> 2) == q;
            uint32_t s, m;
            if (in0 && in1) { s = ocode[i] | (ocode1[i] << 8); m = (uint32_t)((o0 & 3) | ((o1 & 3) << 2)); }
            else if (in0 || in1) {
              const uint32_t pp = (uint32_t)((in0 ? o0 : o1) & 3), cc = in0 ? ocode[i] : ocode1[i];
              s = pp == 3u ? cc << 8 : cc;
              m = (pp == 3u ? 0u : pp) | 12u;
            } else { s = 0; m = 4u; }
            st[i] |= s << (16 * q);
            meta |= m << (8 * i + 4 * q);
          }
        }
        *reinterpret_cast<uint4*>(wo + (b >> 1) * 4096 + core + odd * 128) = make_uint4(st[0], st[1], st[2], st[3]);
        queue32(metas, meta);
        *reinterpret_cast<uint2*>(wc + r * 32 + 8 * b) =
            make_uint2(ocode[0] | (ocode1[0] << 8) | (ocode[1] << 16) | (ocode1[1] << 24), ocode[2] | (ocode1[2] << 8) | (ocode[3] << 16) | (ocode1[3] << 24));
        *reinterpret_cast<uint32_t*>(wc + 2 * WC_CODE_BYTES + r * 16 + 4 * b) =
            opos[0] | (opos1[0] << 4) | (opos[1] << 8) | (opos1[1] << 12) | (opos[2] << 16) | (opos1[2] << 20) | (opos[3] << 24) | (opos1[3] << 28);
      }
    }
    if constexpr (DENSE && CHOSEN) queue32(c_gone, 0u);    // (the next trip's sets of dropped positions to the front)
  }
  if constexpr (!DENSE) *reinterpret_cast<uint2*>(wi + A_IN_BYTES + r * 16 + h * 8) = make_uint2(c_nib[0], c_nib[1]);
  if constexpr (OUTN > 0) *reinterpret_cast<uint4*>(wo + A_OUT_BYTES + r * 16) = make_uint4(metas[0], metas[1], metas[2], metas[3]);
  if constexpr (OUTN == 1) {
    *reinterpret_cast<uint4*>(wc + r * 16) = make_uint4(codes[0], codes[1], codes[2], codes[3]);
    *reinterpret_cast<uint2*>(wc + WC_CODE_BYTES + r * 8) = make_uint2(sels[0] | (sels[1] << 16), sels[2] | (sels[3] << 16));
  }
  // ---- inlier scales: one atom per 128-K half with four scales of 32 K, or two scales of 64 K of the one atom
  uint8_t* sf = wi + a_in_bytes(DENSE) + e_in_bytes(DENSE) + (r & 31) * 16 + (r >> 5) * 4;
  if (b32) *reinterpret_cast<uint32_t*>(sf + h * SF_ATOM_BYTES) = sc;
  else *reinterpret_cast<uint16_t*>(sf + 2 * h) = (uint16_t)sc;
}

template <bool DENSE, bool WGT, int OUTN>
static void launch_pack(const PackParams& p, const BlobHeader& hdr, cudaStream_t st)
{
  const unsigned cx = (unsigned)((p.K + PK_K - 1) / PK_K);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(cx * (unsigned)(p.N / PK_ROWS));
  lc.blockDim = dim3(PK_THREADS);
  lc.dynamicSmemBytes = PK_SMEM;
  lc.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cx;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  lc.attrs = attr;
  auto go = [&](auto kern, int n_attrs) {
    lc.numAttrs = n_attrs;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PK_SMEM) == cudaSuccess) (void)cudaLaunchKernelEx(&lc, kern, p, hdr);
  };
  if (cx <= 8) {
    go(pack_kernel<DENSE, WGT, OUTN, true>, 1);
    return;
  }
  // rows longer than a cluster of eight CTAs holds
  const unsigned rows = (unsigned)(p.N / 8);
  if (WGT || p.order_mask || p.ue) row_scale_kernel<true, WGT, OUTN><<<rows, 256, 0, st>>>(p, hdr);
  else row_scale_kernel<false, WGT, OUTN><<<rows, 256, 0, st>>>(p, hdr);
  go(pack_kernel<DENSE, WGT, OUTN, false>, 0);
}

// Host-visible words of a call in flight, where the kernels report a non-finite weight and a wait that gave up: a page of pinned
// memory, taken once per process and kept; a call holds its words until its stream has been synchronised, so calls of other threads
// and streams never share any.  More calls at once than there are words for wait for some to be given back.
class ReportWords {
 public:
  uint32_t* take() {
    std::unique_lock<std::mutex> lock(m_);
    if (!base_) {
      void* ptr = nullptr;
      if (cudaHostAlloc(&ptr, COUNT * WORDS * sizeof(uint32_t), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) return nullptr;
      base_ = (uint32_t*)ptr;
      for (int i = 0; i < COUNT; ++i) free_[i] = i;
      n_free_ = COUNT;
    }
    cv_.wait(lock, [this] { return n_free_ > 0; });
    uint32_t* w = base_ + free_[--n_free_] * WORDS;
    for (int i = 0; i < WORDS; ++i) reinterpret_cast<volatile uint32_t*>(w)[i] = 0u;
    return w;
  }
  void give_back(uint32_t* w) {
    { std::lock_guard<std::mutex> lock(m_); free_[n_free_++] = (int)(w - base_) / WORDS; }
    cv_.notify_one();
  }
 private:
  static constexpr int COUNT = 64, WORDS = 2;
  std::mutex m_;
  std::condition_variable cv_;
  uint32_t* base_ = nullptr;
  int free_[COUNT];
  int n_free_ = 0;
};
static ReportWords g_report;

// outlier t of S-Vector g of row r in row tile rt, from the compact records: code and position
__device__ __forceinline__ uint8_t wc_code(const uint8_t* blob, const PackedOffsets& off, int64_t rt, int T1, uint32_t r, int g, int out_n, int t) {
  const uint8_t* wc = blob + off.wc + ((size_t)rt * T1 + (g >> 4)) * (size_t)wc_bytes(out_n);
  return wc[r * 16 * out_n + (g & 15) * out_n + t];
}
__device__ __forceinline__ uint8_t wc_pos(const uint8_t* blob, const PackedOffsets& off, int64_t rt, int T1, uint32_t r, int g, int out_n, int t) {
  const uint8_t* wc = blob + off.wc + ((size_t)rt * T1 + (g >> 4)) * (size_t)wc_bytes(out_n);
  const int e = (g & 15) * out_n + t;
  return (uint8_t)((wc[WC_CODE_BYTES * out_n + r * 8 * out_n + (e >> 1)] >> (4 * (e & 1))) & 15);
}

// packed buffer -> canonical arrays (one code per byte)
__global__ void __launch_bounds__(128)
export_packed_kernel(const uint8_t* __restrict__ blob, int64_t N, int64_t K, sdq_config_t cfg, PackedOffsets off, sdq_canonical_t out)
{
  const int64_t n = blockIdx.x;
  const int G = (int)(K / 8), out_n = cfg.out_n;
  const int64_t rt = n / TILE_ROWS;
  const uint32_t r = (uint32_t)(n % TILE_ROWS);
  const int T1 = (int)(K / K1), T2 = (int)(K / K2);
  const bool b32 = cfg.in_block == 32, dense = is_dense_layout(cfg), elem = cfg.in_gran == SDQ_GRAN_ELEM;
  const int wib = wi_bytes(b32, dense);
  const uint8_t* wi_base = blob + off.wi + (size_t)rt * T2 * wib;
  for (int g = threadIdx.x; g < G; g += 128) {
    const uint8_t* wi = wi_base + (size_t)(g >> 5) * wib;
    if (dense) {
      const uint32_t codes = *reinterpret_cast<const uint32_t*>(wi + a_off(r, (uint32_t)(g & 31) * 4));
      if (elem) {
        // element-wise 2:4: the canonical arrays hold the two kept slots of every 4 and their indices
        uint8_t* ic = out.in_code + (size_t)n * (K / 2) + 4 * g;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t mb = blob[off.emeta + (size_t)n * (size_t)(K / 4) + 2 * g + h];
          out.in_meta[(size_t)n * (K / 4) + 2 * g + h] = (uint8_t)mb;
          ic[2 * h] = (codes >> (4 * (4 * h + (mb & 3)))) & 15;
          ic[2 * h + 1] = (codes >> (4 * (4 * h + ((mb >> 2) & 3)))) & 15;
        }
      } else {
      uint8_t* ic = out.in_code + (size_t)n * K + 8 * g;
#pragma unroll
      for (int i = 0; i < 8; ++i) ic[i] = (codes >> (4 * i)) & 15;
      }
      if ((g & 3) == 0) out.in_scale[(size_t)n * (K / 32) + (g >> 2)] = wi[a_in_bytes(true) + in_sf_off(true, r, (uint32_t)((g >> 2) & 7))];
      for (int t = 0; t < out_n; ++t) {
        out.out_code[((size_t)n * G + g) * out_n + t] = wc_code(blob, off, rt, T1, r, g, out_n, t);
        out.out_idx[((size_t)n * G + g) * out_n + t] = wc_pos(blob, off, rt, T1, r, g, out_n, t);
      }
      continue;
    }
    const uint32_t codes = *reinterpret_cast<const uint16_t*>(wi + a_off(r, (uint32_t)(g & 31) * 2));
    uint8_t* ic = out.in_code + (size_t)n * (K / 2) + 4 * g;
    ic[0] = codes & 15; ic[1] = (codes >> 4) & 15; ic[2] = (codes >> 8) & 15; ic[3] = (codes >> 12) & 15;
    const uint32_t mb = wi[A_IN_BYTES + r * 16 + ((g & 31) >> 1)];
    out.in_meta[(size_t)n * G + g] = (uint8_t)((g & 1) ? (mb >> 4) : (mb & 15));
    if (b32) { if ((g & 3) == 0) out.in_scale[(size_t)n * (K / 32) + (g >> 2)] = wi[A_IN_BYTES + E_IN_BYTES + in_sf_off(true, r, (uint32_t)((g >> 2) & 7))]; }
    else if ((g & 7) == 0) out.in_scale[(size_t)n * (K / 64) + (g >> 3)] = wi[A_IN_BYTES + E_IN_BYTES + in_sf_off(false, r, (uint32_t)((g >> 3) & 3))];
    for (int t = 0; t < out_n; ++t) {
      out.out_code[((size_t)n * G + g) * out_n + t] = wc_code(blob, off, rt, T1, r, g, out_n, t);
      out.out_idx[((size_t)n * G + g) * out_n + t] = wc_pos(blob, off, rt, T1, r, g, out_n, t);
    }
  }
  if (threadIdx.x == 0) {
    out.out_sexp[n] = reinterpret_cast<const int32_t*>(blob + off.osexp)[n];
    if (out.in_texp) out.in_texp[n] = reinterpret_cast<const int32_t*>(blob + off.wtexp)[n];
  }
}

// two ranges of a packed buffer (16-byte units) to their places in another, and its header: one pass at DRAM speed
struct CopyRange { const uint4* src; uint4* dst; size_t n; };
__global__ void __launch_bounds__(256)
compact_kernel(const CopyRange a, const CopyRange b, uint32_t* __restrict__ header, const BlobHeader hdr)
{
  if (blockIdx.x == 0 && threadIdx.x < HEADER_BYTES / 4)
    header[threadIdx.x] = threadIdx.x < sizeof(BlobHeader) / 4 ? reinterpret_cast<const uint32_t*>(&hdr)[threadIdx.x] : 0u;
  const size_t step = (size_t)gridDim.x * 256, n = a.n + b.n;
  auto from = [&](size_t i) { return i < a.n ? a.src + i : b.src + (i - a.n); };
  auto to = [&](size_t i) { return i < a.n ? a.dst + i : b.dst + (i - a.n); };
  size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  for (; i + 3 * step < n; i += 4 * step) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = __ldcs(from(i + u * step));
#pragma unroll
    for (int u = 0; u < 4; ++u) *to(i + u * step) = v[u];
  }
  for (; i < n; i += step) *to(i) = __ldcs(from(i));
}

}  // namespace sdq

using namespace sdq;

static bool cfg_ok(const sdq_config_t* c) {
  return c && c->out_n >= 0 && c->out_n <= 2 && c->in_gran >= 0 && c->in_gran <= SDQ_GRAN_3OF4 &&
         (c->out_order == SDQ_ORDER_LARGE || c->out_order == SDQ_ORDER_SMALL) &&
         (c->in_gran < SDQ_GRAN_DENSE || c->in_gran == SDQ_GRAN_3OF4 || 10 - c->in_gran > c->out_n) &&
         (c->in_gran != SDQ_GRAN_3OF4 || c->out_n != 1) &&
         (c->in_block == 32 || c->in_block == 64) && c->scale_rule >= SDQ_SCALE_OCP_FLOOR && c->scale_rule <= SDQ_SCALE_UE4M3 &&
         (c->out_fmt == SDQ_OUT_E4M3 || (c->out_fmt == SDQ_OUT_INT8 && c->scale_rule != SDQ_SCALE_UE4M3));
}
// valid configurations this kernel set does not carry out
static bool cfg_unsupported(const sdq_config_t* c) {
  return (c->in_gran >= SDQ_GRAN_DENSE && c->in_block != 32) ||
         (c->scale_rule == SDQ_SCALE_UE4M3 && !(c->in_gran == SDQ_GRAN_PAIR && c->in_block == 32)) ||
         (c->out_fmt == SDQ_OUT_INT8 && !(c->in_gran == SDQ_GRAN_PAIR && c->in_block == 64));   // int8 outliers: the primary format only
}

static void fill_header(BlobHeader* h, const sdq_packed_t& d, bool tiled) {
  h->magic = BLOB_MAGIC;
  h->version = BLOB_VERSION;
  h->header_bytes = (uint32_t)HEADER_BYTES;
  h->cfg[0] = d.cfg.out_n; h->cfg[1] = d.cfg.in_gran; h->cfg[2] = d.cfg.in_block; h->cfg[3] = d.cfg.scale_rule; h->cfg[4] = d.cfg.out_order; h->cfg[5] = d.cfg.out_fmt;
  h->tiled = tiled ? 1u : 0u;
  h->N = d.N; h->K = d.K;
  h->total = d.bytes;
  for (int i = 0; i < 8; ++i) h->off[i] = d.off[i];
}

extern "C" sdq_status_t sdq_packed_size(int64_t N, int64_t K, const sdq_config_t* cfg, size_t* bytes, size_t* algorithmic_bytes)
{
  if (!cfg_ok(cfg)) return SDQ_ERR_INVALID_ARG;
  if (cfg_unsupported(cfg)) return SDQ_ERR_UNSUPPORTED;
  if (N <= 0 || K <= 0 || N % TILE_ROWS || K % K2) return SDQ_ERR_SHAPE;
  if (bytes) *bytes = is_tensor_core_reading(*cfg) ? tiled_offsets(N, K, *cfg).total : plain_packed_offsets(N, K, *cfg).total;
  if (algorithmic_bytes) {
    // per weight: 4-bit values on half the positions (2) + index metadata (pair-wise: two 2-bit pair indices per 8 =
    // 0.5; element-wise: two 2-bit indices per 4 = 1) + one 8-bit scale per Q-Vector + out_n * (8 value + 3 index
    // bits) per 8; plus one 32-bit row scale
    // (dense storage: a 4-bit value on every position and no index metadata)
    const double inl = cfg->in_gran >= SDQ_GRAN_DENSE ? 4.0 : 2.0 + (cfg->in_gran == SDQ_GRAN_PAIR ? 0.5 : 1.0);   // 2:4: the paper's form
    const double bits = inl + 8.0 / cfg->in_block + cfg->out_n * 11.0 / 8.0;
    *algorithmic_bytes = (size_t)((double)N * (double)K * bits / 8.0) + (cfg->out_n ? (size_t)N * 4 : 0);
  }
  return SDQ_OK;
}

// polls: what a wait inside the kernel is given
static sdq_status_t decompose(const void* W, int64_t N, int64_t K, int64_t ldw, const sdq_config_t* cfg, const float* col_weight, void* packed_buf,
                              size_t packed_bytes, sdq_packed_t* out, void* stream, uint32_t polls = 1u << 22)
{
  if (!W || !packed_buf || !out || !cfg_ok(cfg)) return SDQ_ERR_INVALID_ARG;
  if (cfg_unsupported(cfg)) return SDQ_ERR_UNSUPPORTED;
  if ((uintptr_t)col_weight & 15) return SDQ_ERR_ALIGNMENT;
  if (N <= 0 || K <= 0 || N % TILE_ROWS || K % K2 || ldw < K) return SDQ_ERR_SHAPE;
  if (((uintptr_t)W & 15) || ((uintptr_t)packed_buf & 15) || (ldw % 8)) return SDQ_ERR_ALIGNMENT;
  const bool tc = is_tensor_core_reading(*cfg);
  const PackedOffsets off = tiled_offsets(N, K, *cfg);
  const PlainPackedOffsets poff = plain_packed_offsets(N, K, *cfg);
  if (packed_bytes < (tc ? off.total : poff.total)) return SDQ_ERR_BUFFER_TOO_SMALL;
  cudaStream_t st = (cudaStream_t)stream;
  out->dev = packed_buf;
  out->bytes = tc ? off.total : poff.total;
  out->N = N;
  out->K = K;
  out->cfg = *cfg;
  for (int i = 0; i < 8; ++i) out->off[i] = 0;
  if (tc) {
    out->off[0] = off.wi; out->off[1] = off.wo; out->off[2] = off.sfa_out;
    out->off[3] = off.wc; out->off[4] = 0; out->off[5] = off.osexp; out->off[6] = off.wtexp;
  } else {
    out->off[0] = poff.in_code; out->off[1] = poff.in_meta; out->off[2] = poff.in_scale;
    out->off[3] = poff.out_code; out->off[4] = poff.out_idx; out->off[5] = poff.osexp;
  }
  // the self-describing header (read back by sdq_packed_attach)
  alignas(16) unsigned char raw[HEADER_BYTES] = {0};
  BlobHeader* hdr = reinterpret_cast<BlobHeader*>(raw);
  fill_header(hdr, *out, tc);
  uint32_t* report = g_report.take();
  if (!report) return SDQ_ERR_CUDA;
  uint32_t* report_dev = nullptr;
  bool ok = cudaHostGetDevicePointer((void**)&report_dev, report, 0) == cudaSuccess;
  if (ok && tc) {
    PackParams p;
    p.W = (const __nv_bfloat16*)W; p.N = N; p.K = K; p.ldw = ldw; p.colw = col_weight;
    p.blob = (uint8_t*)packed_buf; p.off = off; p.nonfinite = report_dev; p.gave_up = report_dev + 1; p.polls = polls;
    p.out_n = cfg->out_n;
    p.sv4 = cfg->in_gran == SDQ_GRAN_3OF4;          // S-Vectors of 4: one outlier and two inliers per 4
    p.elem = cfg->in_gran == SDQ_GRAN_ELEM;         // element-wise 2:4: the 2 most significant non-outliers of every 4
    // dense family: inliers kept per group (8 - out_n without Stage 1; groups of 4: 3 minus the outlier, or 2 for 2:4)
    p.keep_in = p.elem ? 2 : (p.sv4 ? (cfg->out_n ? 2 : 3) : 10 - cfg->in_gran - cfg->out_n);
    p.order_mask = cfg->out_order == SDQ_ORDER_SMALL ? (col_weight ? 0x7FFFFFFF : 0x7FFF0000) : 0;
    p.ue = cfg->scale_rule == SDQ_SCALE_UE4M3;
    p.i8 = cfg->out_fmt == SDQ_OUT_INT8;
    p.b32 = cfg->in_block == 32;
    p.ceil_rule = cfg->scale_rule == SDQ_SCALE_CEIL_NOSAT;
    const int v = (col_weight ? 3 : 0) + cfg->out_n;
    auto pick = [&](auto dense) {
      constexpr bool D = decltype(dense)::value;
      switch (v) {
        case 0: launch_pack<D, false, 0>(p, *hdr, st); break;
        case 1: launch_pack<D, false, 1>(p, *hdr, st); break;
        case 2: launch_pack<D, false, 2>(p, *hdr, st); break;
        case 3: launch_pack<D, true, 0>(p, *hdr, st); break;
        case 4: launch_pack<D, true, 1>(p, *hdr, st); break;
        default: launch_pack<D, true, 2>(p, *hdr, st); break;
      }
    };
    if (is_dense_layout(*cfg)) pick(std::true_type{}); else pick(std::false_type{});
  } else if (ok) {
    launch_pack_plain(W, N, K, ldw, *cfg, col_weight, packed_buf, report_dev, st);
    ok = cudaMemcpyAsync(packed_buf, raw, HEADER_BYTES, cudaMemcpyHostToDevice, st) == cudaSuccess;
  }
  ok = (cudaGetLastError() == cudaSuccess) && ok;
  ok = (cudaStreamSynchronize(st) == cudaSuccess) && ok;      // also before the word goes back: no kernel writes it afterwards
  const uint32_t nonfinite = reinterpret_cast<volatile uint32_t*>(report)[0], gave_up = reinterpret_cast<volatile uint32_t*>(report)[1];
  g_report.give_back(report);
  if (!ok) return SDQ_ERR_CUDA;
  return nonfinite ? SDQ_ERR_NONFINITE : (gave_up ? SDQ_ERR_TIMEOUT : SDQ_OK);
}

extern "C" sdq_status_t sdq_decompose(const void* W, int64_t N, int64_t K, int64_t ldw, const sdq_config_t* cfg, void* packed_buf,
                                      size_t packed_bytes, sdq_packed_t* out, void* stream)
{ return decompose(W, N, K, ldw, cfg, nullptr, packed_buf, packed_bytes, out, stream); }

extern "C" sdq_status_t sdq_decompose_metric(const void* W, int64_t N, int64_t K, int64_t ldw, const sdq_config_t* cfg,
                                             const float* col_weight, void* packed_buf, size_t packed_bytes, sdq_packed_t* out,
                                             void* stream)
{ return decompose(W, N, K, ldw, cfg, col_weight, packed_buf, packed_bytes, out, stream); }

extern "C" sdq_status_t sdq_diag_decompose_timeout(const void* W, int64_t N, int64_t K, int64_t ldw, const sdq_config_t* cfg, void* packed_buf,
                                                   size_t packed_bytes, sdq_packed_t* out, void* stream)
{ return decompose(W, N, K, ldw, cfg, nullptr, packed_buf, packed_bytes, out, stream, 0); }

extern "C" sdq_status_t sdq_packed_attach(const void* dev, size_t bytes, sdq_packed_t* out, void* stream)
{
  if (!dev || !out) return SDQ_ERR_INVALID_ARG;
  if ((uintptr_t)dev & 15) return SDQ_ERR_ALIGNMENT;
  if (bytes < HEADER_BYTES) return SDQ_ERR_BUFFER_TOO_SMALL;
  alignas(16) unsigned char raw[HEADER_BYTES];
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(raw, dev, HEADER_BYTES, cudaMemcpyDeviceToHost, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
    return SDQ_ERR_CUDA;
  const BlobHeader* h = reinterpret_cast<const BlobHeader*>(raw);
  if (h->magic != BLOB_MAGIC || h->version != BLOB_VERSION || h->header_bytes != HEADER_BYTES) return SDQ_ERR_UNSUPPORTED;
  sdq_config_t cfg;
  cfg.out_n = h->cfg[0]; cfg.in_gran = h->cfg[1]; cfg.in_block = h->cfg[2]; cfg.scale_rule = h->cfg[3]; cfg.out_order = h->cfg[4]; cfg.out_fmt = h->cfg[5];
  if (!cfg_ok(&cfg) || cfg_unsupported(&cfg)) return SDQ_ERR_SHAPE;
  if (h->N <= 0 || h->K <= 0 || h->N % TILE_ROWS || h->K % K2) return SDQ_ERR_SHAPE;
  // the sections must sit where this library puts them for that configuration and shape
  const bool tc = is_tensor_core_reading(cfg);
  if ((h->tiled != 0) != tc) return SDQ_ERR_SHAPE;
  sdq_packed_t d;
  d.dev = const_cast<void*>(dev);
  d.N = h->N; d.K = h->K; d.cfg = cfg;
  for (int i = 0; i < 8; ++i) d.off[i] = 0;
  if (tc) {
    const bool compact = h->tiled == 2;
    if (h->tiled > 2 || (compact && cfg.out_n == 0)) return SDQ_ERR_SHAPE;
    const PackedOffsets off = tiled_offsets(h->N, h->K, cfg, compact);
    d.bytes = off.total;
    d.off[0] = off.wi; d.off[1] = compact ? 0 : off.wo; d.off[2] = off.sfa_out; d.off[3] = off.wc; d.off[5] = off.osexp; d.off[6] = off.wtexp;
  } else {
    const PlainPackedOffsets poff = plain_packed_offsets(h->N, h->K, cfg);
    d.bytes = poff.total;
    d.off[0] = poff.in_code; d.off[1] = poff.in_meta; d.off[2] = poff.in_scale; d.off[3] = poff.out_code; d.off[4] = poff.out_idx; d.off[5] = poff.osexp;
  }
  if (h->total != d.bytes) return SDQ_ERR_SHAPE;
  for (int i = 0; i < 8; ++i)
    if (h->off[i] != d.off[i]) return SDQ_ERR_SHAPE;
  if (bytes < d.bytes) return SDQ_ERR_BUFFER_TOO_SMALL;
  *out = d;
  return SDQ_OK;
}

extern "C" sdq_status_t sdq_packed_compact_size(int64_t N, int64_t K, const sdq_config_t* cfg, size_t* bytes)
{
  if (!cfg_ok(cfg) || !bytes) return SDQ_ERR_INVALID_ARG;
  if (cfg_unsupported(cfg) || !is_tensor_core_reading(*cfg) || cfg->out_n == 0) return SDQ_ERR_UNSUPPORTED;
  if (N <= 0 || K <= 0 || N % TILE_ROWS || K % K2) return SDQ_ERR_SHAPE;
  *bytes = tiled_offsets(N, K, *cfg, true).total;
  return SDQ_OK;
}

extern "C" sdq_status_t sdq_packed_compact(const sdq_packed_t* P, void* dst, size_t dst_bytes, sdq_packed_t* out, void* stream)
{
  if (!P || !P->dev || !dst || !out) return SDQ_ERR_INVALID_ARG;
  if (!cfg_ok(&P->cfg)) return SDQ_ERR_INVALID_ARG;
  if (!is_tensor_core_reading(P->cfg) || P->cfg.out_n == 0 || is_compact(*P)) return SDQ_ERR_UNSUPPORTED;
  if ((uintptr_t)dst & 255) return SDQ_ERR_ALIGNMENT;
  const PackedOffsets src = tiled_offsets(P->N, P->K, P->cfg), off = tiled_offsets(P->N, P->K, P->cfg, true);
  if (dst_bytes < off.total) return SDQ_ERR_BUFFER_TOO_SMALL;
  cudaStream_t st = (cudaStream_t)stream;
  const uint8_t* s = (const uint8_t*)P->dev;
  uint8_t* d = (uint8_t*)dst;
  sdq_packed_t q;
  q.dev = dst; q.bytes = off.total; q.N = P->N; q.K = P->K; q.cfg = P->cfg;
  for (int i = 0; i < 8; ++i) q.off[i] = 0;
  q.off[0] = off.wi; q.off[1] = 0; q.off[2] = off.sfa_out; q.off[3] = off.wc; q.off[5] = off.osexp; q.off[6] = off.wtexp;
  BlobHeader hdr;
  fill_header(&hdr, q, true);
  hdr.tiled = 2u;
  // every section but the 2:4 containers, each to its place in the shorter buffer
  const CopyRange a = {(const uint4*)(s + src.wi), (uint4*)(d + off.wi), (src.wo - src.wi) / 16};
  const CopyRange b = {(const uint4*)(s + src.sfa_out), (uint4*)(d + off.sfa_out), (src.total - src.sfa_out) / 16};
  const DeviceInfo* dinfo = device_info();
  if (!dinfo) return SDQ_ERR_CUDA;
  compact_kernel<<<(unsigned)(dinfo->sm_count * 8), 256, 0, st>>>(a, b, (uint32_t*)d, hdr);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return SDQ_ERR_CUDA;
  *out = q;
  return SDQ_OK;
}

extern "C" sdq_status_t sdq_packed_export(const sdq_packed_t* P, const sdq_canonical_t* out, void* stream)
{
  if (!P || !out || !P->dev || !out->in_code || !out->in_scale || !out->out_sexp) return SDQ_ERR_INVALID_ARG;
  if (!out->in_meta && P->cfg.in_gran < SDQ_GRAN_DENSE) return SDQ_ERR_INVALID_ARG;   // PAIR and ELEM record their pattern
  if (P->cfg.out_n > 0 && (!out->out_code || !out->out_idx)) return SDQ_ERR_INVALID_ARG;
  if (!is_tensor_core_reading(P->cfg)) {
    // the buffer already holds the canonical arrays
    const PlainPackedOffsets o = plain_packed_offsets(P->N, P->K, P->cfg);
    const uint8_t* b = (const uint8_t*)P->dev;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t n = (size_t)P->N, k = (size_t)P->K, on = (size_t)P->cfg.out_n;
    bool ok = cudaMemcpyAsync(out->in_code, b + o.in_code, n * k / 2, cudaMemcpyDeviceToDevice, st) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(out->in_meta, b + o.in_meta, n * (P->cfg.in_gran == SDQ_GRAN_PAIR ? k / 8 : k / 4), cudaMemcpyDeviceToDevice, st) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(out->in_scale, b + o.in_scale, n * k / (size_t)P->cfg.in_block, cudaMemcpyDeviceToDevice, st) == cudaSuccess;
    if (on) {
      ok = ok && cudaMemcpyAsync(out->out_code, b + o.out_code, n * (k / 8) * on, cudaMemcpyDeviceToDevice, st) == cudaSuccess;
      ok = ok && cudaMemcpyAsync(out->out_idx, b + o.out_idx, n * (k / 8) * on, cudaMemcpyDeviceToDevice, st) == cudaSuccess;
    }
    ok = ok && cudaMemcpyAsync(out->out_sexp, b + o.osexp, n * 4, cudaMemcpyDeviceToDevice, st) == cudaSuccess;
    return ok ? SDQ_OK : SDQ_ERR_CUDA;
  }
  const PackedOffsets off = tiled_offsets(*P);
  export_packed_kernel<<<(unsigned)P->N, 128, 0, (cudaStream_t)stream>>>((const uint8_t*)P->dev, P->N, P->K, P->cfg, off, *out);
  return cudaGetLastError() == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
}
