// Runtime activation quantization A -> A_i (E2M1 + E8M0 per 64 K) and A_o (E4M3 + per-token power-of-two
// scale), "we also quantize activations accordingly" (Section 5, Stage 3; A_o / A_i of Section 5.1).
//
// The per-token 8-bit scale needs the whole row before anything can be stored.  Rows up to 16384 long take one
// launch (`quant_act_fused_kernel`): the CTAs of a thread-block cluster split the K range of a group of 8 tokens,
// keep their elements in registers, exchange the per-token maxima through distributed shared memory and encode.
// Longer rows take two launches: `act_amax_kernel` reduces, per token, the largest magnitude of each 2048-K chunk,
// `quant_act_kernel` then encodes, one CTA per (group of 8 tokens = one row group of the operand layout, 2048-K chunk).
// In all of them (but the spread form of few tokens, see its dispatch) a warp works on one unit: 8 tokens x 256 K, i.e. what 8 tokens have in one record of the layout; 4 lanes
// per token, for each of the unit's four 64-K Q-Vectors 16 elements (two 16-byte loads) per lane.  A Q-Vector maximum is
// then a 4-lane shuffle, a token's four scales are one word, and every store instruction of codes writes whole 128-byte
// lines (8 tokens x 16 B per core matrix).  Codes come from the hardware E2M1 / E4M3 converters.
//
// Bound by DRAM traffic and the conversion instructions: 2048 x 11008 at 4.7 TB/s of algorithmic bytes (16.9 us), 8192 x 11008 at
// 5.6 TB/s (56.7), 8192 x 4096 at 5.7 (20.7), one token 2.1 us, most of it the launch.  In steps: with releasing cluster arrivals, no
// fetching ahead and an unpacking in front of every multiplication 20.1, 66.0, 23.5 us, without these 18.0, 58.3, 21.5; 4096 x 16384 with
// E4M3 scales, where 64 registers also let a fourth CTA onto the SM, 60.1 -> 45.7.  E4M3 scales and int8 codes multiply by a reciprocal
// instead of dividing every element (see sdq_codec.cuh): one int8 token 14.1 -> 3.0 us (zeros took the division's slow path).
// Products that only one of the 8-bit forms needs are formed in its branch: in front of it, int8 calls paid for E4M3's (8192 x 4096,
// back to back, 45.6 -> 42.7 us; before scaled2 43.9) and everybody for their registers (8192 x 2048 10.2 -> 9.9, 2048 x 11008 15.9 -> 15.2).
#include "sdq_codec.cuh"
#include "sdq_internal.h"
#include "sdq_layout.h"
#include "sdq_plain.h"
#include "sdq_ptx.cuh"

namespace sdq {

constexpr int QA_THREADS = 256;
constexpr int QA_WARPS = QA_THREADS / 32;
constexpr int QA_CHUNK = QA_WARPS * K2;                  // K per CTA: one 256-K unit per warp

// a lane's part of a unit: its token's elements 64 i + 16 l .. + 15 for NQ of the four Q-Vectors i
template <int NQ>
struct QaUnit {
  uint4 raw[NQ][2];
  uint32_t qmax[NQ];                                     // largest magnitude bits of the 16 elements
};
// `on`: the token exists and the unit lies inside the row (zeros otherwise)
template <int NQ>
__device__ __forceinline__ void qa_load(QaUnit<NQ>& u, const __nv_bfloat16* p, bool on) {
#pragma unroll
  for (int i = 0; i < NQ; ++i) {
    u.raw[i][0] = u.raw[i][1] = make_uint4(0, 0, 0, 0);
    if (on) {
      const uint4* q = reinterpret_cast<const uint4*>(p + i * 64);
      u.raw[i][0] = q[0];
      u.raw[i][1] = q[1];
    }
  }
}
// fills qmax and returns the largest magnitude bits of all the lane's elements.  +-Inf counts as the largest
// finite bf16: maxima are clamped, the elements only where a lane of the warp holds one
template <int NQ>
__device__ __forceinline__ uint32_t qa_maxima(QaUnit<NQ>& u) {
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < NQ; ++i) {
    const uint32_t r[8] = {u.raw[i][0].x, u.raw[i][0].y, u.raw[i][0].z, u.raw[i][0].w, u.raw[i][1].x, u.raw[i][1].y, u.raw[i][1].z, u.raw[i][1].w};
    uint32_t q = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) q = max_abs2(q, r[j]);
    q = max(q & 0xFFFFu, q >> 16);
    u.qmax[i] = min(q, 0x7F7Fu);
    m = max(m, q);
  }
  // (a branch of the warp: as predicated instructions in the encoding, the clamping cost 2 to 5 %)
  if (__any_sync(0xffffffffu, m > 0x7F7Fu)) {
#pragma unroll
    for (int i = 0; i < NQ; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint4& w = u.raw[i][h];
        w = make_uint4(finite2(w.x), finite2(w.y), finite2(w.z), finite2(w.w));
      }
  }
  return min(m, 0x7F7Fu);
}
// writes `w` (a token's four scales of one 128- or 256-K block) to the overlapping atoms that hold the token: lane l (0..3)
// of the token writes word l of atom m / 32 - l; `step` = bytes between atom numbers
__device__ __forceinline__ void qa_store_scales(uint8_t* atoms, uint32_t step, int64_t m, uint32_t l, uint32_t w) {
  const int64_t a = m / 32 - (int64_t)l;
  if (a >= 0) *reinterpret_cast<uint32_t*>(atoms + (size_t)a * step + (uint32_t)(m & 31) * 16 + l * 4) = w;
}

// encodes a unit: token m (existing: `live`), 256-K record k2 of the buffer, the token's largest magnitude `ramax`; with NQ < 4
// only its Q-Vectors from `first` on
template <bool UE, int NQ>                               // UE: two-level scaling with E4M3 Q-Vector scales
__device__ __forceinline__ void qa_encode(const QaUnit<NQ>& u, int first, float ramax, bool live, int64_t m, int k2, uint32_t l, const sdq_config_t& cfg,
                                          uint8_t* __restrict__ buf, const ActOffsets& off) {
  const int e = fp8_scale_exp(ramax);
  const float s8 = pow2_neg(e);
  const uint32_t s8x = (uint32_t)(127 - e) << 7;         // as bf16
  const bool i8 = cfg.out_fmt == SDQ_OUT_INT8;           // A_o in int8: fp32 token scale amax / 127
  const Int8Coder k8 = int8_coder(int8_scale(ramax));
  const bool b32 = cfg.in_block == 32;                   // one scale per 32 K: a Q-Vector is a lane pair
  uint8_t* xi = buf + off.xi + (size_t)k2 * off.xi_stride + (size_t)(m >> 3) * 1024 + (uint32_t)(m & 7) * 16;
  uint8_t* xo = buf + off.xo + (size_t)(2 * k2) * off.xo_stride + (size_t)(m >> 3) * 1024 + (uint32_t)(m & 7) * 16;
  uint32_t c[NQ];
#pragma unroll
  for (int i = 0; i < NQ; ++i) {
    const int iq = first + i;
    const uint32_t r[8] = {u.raw[i][0].x, u.raw[i][0].y, u.raw[i][0].z, u.raw[i][0].w, u.raw[i][1].x, u.raw[i][1].y, u.raw[i][1].z, u.raw[i][1].w};
    uint32_t bm = u.qmax[i];
    bm = max(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
    if (!b32) bm = max(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
    uint32_t q4[2] = {0, 0}, q8[4] = {0, 0, 0, 0};
    [[maybe_unused]] float v8[16];                       // in units of the token's 8-bit scale
    if constexpr (UE) {
#pragma unroll
      for (int j = 0; j < 8; ++j) scaled2(r[j], s8x, v8[2 * j], v8[2 * j + 1]);
    }
    if constexpr (!UE) {
      c[i] = e8m0_scale_code_bf16(bm, cfg.scale_rule == SDQ_SCALE_CEIL_NOSAT);
      const uint32_t s4x = (254u - c[i]) << 7;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float f[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) scaled2(r[4 * h + j], s4x, f[2 * j], f[2 * j + 1]);
        q4[h] = e2m1x8(f);
      }
    } else {
      c[i] = ue4m3_scale_code(bf16_bits_to_float(bm) * s8, bm != 0);
      if (c[i]) {
        // two-level scaling: the Q-Vector scale E4M3(c) * 2^e is not a power of two, the elements are divided by it
        const float inv = ue4m3_scale_inverse(c[i]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float f[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) f[j] = small_quotient(v8[8 * h + j], inv);
          q4[h] = e2m1x8(f);
        }
      }
    }
    if (!i8) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if constexpr (!UE) {                             // (here, since int8 has no use for them)
          scaled2(r[2 * j], s8x, v8[4 * j], v8[4 * j + 1]);
          scaled2(r[2 * j + 1], s8x, v8[4 * j + 2], v8[4 * j + 3]);
        }
        q8[j] = e4m3x4(v8[4 * j], v8[4 * j + 1], v8[4 * j + 2], v8[4 * j + 3]);
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        q8[j >> 1] |= (int8_code(__uint_as_float(r[j] << 16), k8) | (int8_code(__uint_as_float(r[j] & 0xFFFF0000u), k8) << 8)) << (16 * (j & 1));
    }
    if (live) {
      // 4-bit codes: bytes 32 i + 8 l of the token's 128; 8-bit codes: bytes 64 (i & 1) + 16 l of the 128-K record i / 2
      *reinterpret_cast<uint2*>(xi + (uint32_t)(2 * iq + (l >> 1)) * 128 + (l & 1) * 8) = make_uint2(q4[0], q4[1]);
      *reinterpret_cast<uint4*>(xo + (size_t)(iq >> 1) * off.xo_stride + (uint32_t)(4 * (iq & 1) + l) * 128) = make_uint4(q8[0], q8[1], q8[2], q8[3]);
    }
  }
  uint8_t* sf = buf + off.xi + (size_t)k2 * off.xi_stride + (size_t)off.Mpad * 128;
  if constexpr (NQ < 4) {
    // its bytes of the words that qa_store_scales writes whole
    const int64_t a = m / 32 - (int64_t)l;
    const uint32_t at = (uint32_t)(m & 31) * 16 + l * 4 + (b32 ? 2u * ((uint32_t)first & 1u) : (uint32_t)first);
    uint8_t* dst = sf + ((size_t)a * (b32 ? 2 : 1) + (b32 ? first >> 1 : 0)) * SF_ATOM_BYTES + at;
    uint32_t w = c[0];
    if constexpr (NQ == 2) w |= c[1] << (b32 ? 16 : 8);
    if (b32) {                                           // two scales per Q-Vector, one of each lane pair
      w <<= 8 * (l >> 1);
      w |= __shfl_xor_sync(0xffffffffu, w, 2);
    }
    if (live && a >= 0) {
      const int bytes = NQ * (b32 ? 2 : 1);
      if (bytes == 1) *dst = (uint8_t)w;
      else if (bytes == 2) *reinterpret_cast<uint16_t*>(dst) = (uint16_t)w;
      else *reinterpret_cast<uint32_t*>(dst) = w;
    }
  } else if (!b32) {
    if (live) qa_store_scales(sf, SF_ATOM_BYTES, m, l, c[0] | (c[1] << 8) | (c[2] << 16) | (c[3] << 24));
  } else {
#pragma unroll
    for (int kb = 0; kb < 2; ++kb) {                     // 128-K block: scales 2 kb and 2 kb + 1 of each lane pair
      uint32_t w = (c[2 * kb] << (8 * (l >> 1))) | (c[2 * kb + 1] << (16 + 8 * (l >> 1)));
      w |= __shfl_xor_sync(0xffffffffu, w, 2);
      if (live) qa_store_scales(sf + kb * SF_ATOM_BYTES, 2 * SF_ATOM_BYTES, m, l, w);
    }
  }
}
// the token's 8-bit scale: exponent (or the bit pattern of the fp32 scale), and its atoms of the outlier product
template <bool UE>
__device__ __forceinline__ void qa_token_scale(float ramax, int64_t m, uint32_t l, const sdq_config_t& cfg, uint8_t* __restrict__ buf, const ActOffsets& off) {
  const bool i8 = cfg.out_fmt == SDQ_OUT_INT8;
  const int e = fp8_scale_exp(ramax);
  if (l == 0) reinterpret_cast<int32_t*>(buf + off.sexp)[m] = i8 ? __float_as_int(int8_scale(ramax)) : e;
  // two-level scaling keeps a token's accumulator column in units of 2^e (the 4-bit scale codes leave that factor out):
  // the 8-bit product then takes the scale 1 here and the GEMM's epilogue multiplies 2^e back in
  qa_store_scales(buf + off.sfb_out, SF_ATOM_BYTES, m, l, (uint32_t)((UE || i8) ? 127 : e + 127) * 0x01010101u);
}

// partial[m][chunk] = max |x| of token m over its 2048-K chunk
__global__ void __launch_bounds__(QA_THREADS)
act_amax_kernel(const __nv_bfloat16* __restrict__ X, int64_t M, int64_t K, int64_t ldx, float* __restrict__ partial, int n_chunks)
{
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t = lane >> 2, l = lane & 3;
  const int64_t m = (int64_t)blockIdx.x * 8 + t;
  const int64_t k = (int64_t)blockIdx.y * QA_CHUNK + warp * K2;
  __shared__ float s_amax[QA_WARPS][8];
  QaUnit<4> u;
  qa_load(u, X + m * ldx + k + l * 16, m < M && k < K);
  float amax = bf16_bits_to_float(qa_maxima(u));
  amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
  amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
  if (l == 0) s_amax[warp][t] = amax;
  __syncthreads();
  if (tid < 8 && (int64_t)blockIdx.x * 8 + tid < M) {
    float a = 0.0f;
#pragma unroll
    for (int w = 0; w < QA_WARPS; ++w) a = fmaxf(a, s_amax[w][tid]);
    partial[((int64_t)blockIdx.x * 8 + tid) * n_chunks + blockIdx.y] = a;
  }
}

template <bool UE>
__global__ void __launch_bounds__(QA_THREADS)
quant_act_kernel(const __nv_bfloat16* __restrict__ X, int64_t M, int64_t K, int64_t ldx, sdq_config_t cfg, uint8_t* __restrict__ buf,
                 ActOffsets off, const float* __restrict__ partial, int n_chunks)
{
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t = lane >> 2, l = lane & 3;                 // token within the group of 8, quarter of the Q-Vector
  // a following sdq_linear may start its set-up and weight copies now; it waits for this grid before reading codes
  if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int64_t m = (int64_t)blockIdx.x * 8 + t;
  const bool live = m < M;
  const int64_t k = (int64_t)blockIdx.y * QA_CHUNK + warp * K2;

  // per-token 8-bit scale from the chunk maxima of the whole row
  float ramax = 0.0f;
  if (live)
    for (int c = l; c < n_chunks; c += 4) ramax = fmaxf(ramax, partial[m * n_chunks + c]);
  ramax = fmaxf(ramax, __shfl_xor_sync(0xffffffffu, ramax, 1));
  ramax = fmaxf(ramax, __shfl_xor_sync(0xffffffffu, ramax, 2));
  if (live && blockIdx.y == 0 && warp == 0) qa_token_scale<UE>(ramax, m, (uint32_t)l, cfg, buf, off);
  if (k >= K) return;
  QaUnit<4> u;
  qa_load(u, X + m * ldx + k + l * 16, live);
  qa_maxima(u);
  qa_encode<UE>(u, 0, ramax, live, m, (int)(k / K2), (uint32_t)l, cfg, buf, off);
}

// Single pass: the CTAs of a cluster share one group of 8 tokens and split its Q-Vectors, NQ per warp; every thread keeps
// its elements in registers (packed bf16) from the one read of X, the per-token maxima meet through distributed shared
// memory, and the codes are produced from the registers.  The two-launch path stays for rows longer than a cluster of
// eight CTAs holds (K > 16384).
template <bool UE, int NQ>
__global__ void __launch_bounds__(NQ == 4 ? QA_THREADS : 512, NQ == 4 ? 4 : 1)
quant_act_fused_kernel(const __nv_bfloat16* __restrict__ X, int64_t M, int64_t K, int64_t ldx, sdq_config_t cfg, uint8_t* __restrict__ buf,
                       ActOffsets off, uint32_t* __restrict__ flags, int early_next, int ahead)
{
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t = lane >> 2, l = lane & 3;                 // token within the group of 8, quarter of the Q-Vector
  const uint32_t cx = gridDim.x, rank = blockIdx.x;      // cluster = the gridDim.x CTAs of one token group
  const int warps = NQ == 4 ? QA_WARPS : (int)(blockDim.x >> 5);
  __shared__ float s_warp[NQ == 4 ? QA_WARPS : 16][8];
  __shared__ float s_all[8][8];                          // [cluster rank][token]: every CTA's maxima, pushed by their owners
  __shared__ uint64_t s_bar;                             // ... all of which have arrived
  if (tid == 0) {
    ptx::mbar_init(&s_bar, 1);
    ptx::fence_barrier_init();
    ptx::mbar_expect_tx(&s_bar, cx * 8u * 4u);
  }
  // (waited for before the first push: by then, behind the loads, every CTA's barrier has long been set up.  The fence has released the
  // barrier's set-up, nothing else was written: as a releasing arrival every warp stood in a memory barrier here, 9 % of the kernel)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  // launched with programmatic stream serialization: X may still be being written by the previous kernel.  The next launch of
  // the stream is let in behind that wait: a linear kernel reads packed weights before its own, and those may be what the
  // kernel in front of this one writes.  Before it only in calls that want the packed weights complete
  if (early_next && tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (!early_next && tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int64_t m = (int64_t)blockIdx.y * 8 + t;
  const bool live = m < M;
  const int q = ((int)rank * warps + warp) * NQ;         // this warp's first Q-Vector
  const bool on = q < (int)(K / 64);
  QaUnit<NQ> u;
  qa_load(u, X + m * ldx + (int64_t)q * 64 + l * 16, live && on);
  float amax = bf16_bits_to_float(qa_maxima(u));
  // The CTAs of a wave load together and encode together, so while this one encodes, the piece that the CTA taking its place will load
  // comes from DRAM into L2 (8192 x 11008 61.5 -> 58.3 us, 2048 x 4096, less than a wave, the same; half or one and a half waves ahead no better)
  if constexpr (NQ == 4) {
    const int64_t m2 = ((int64_t)blockIdx.y + ahead) * 8 + tid, k = (int64_t)rank * QA_CHUNK;
    if (ahead && tid < 8 && m2 < M) ptx::bulk_prefetch_l2(X + m2 * ldx + k, 2u * (uint32_t)(K - k < QA_CHUNK ? K - k : QA_CHUNK));
  }
  amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
  amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
  if (l == 0) s_warp[warp][t] = amax;
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  __syncthreads();
  if (tid < 8 * (int)cx) {
    // thread (peer, token): this CTA's maximum of the token goes into row `rank` of the peer's table; the store counts its bytes
    // on the peer's barrier, so that nothing but its own copies' arrival keeps a CTA waiting (a cluster barrier behind
    // plain stores cost a quarter of the stalls)
    const int tok = tid & 7;
    const uint32_t peer = (uint32_t)tid >> 3;
    float a = 0.0f;
#pragma unroll 8
    for (int w = 0; w < warps; ++w) a = fmaxf(a, s_warp[w][tok]);
    ptx::st_async_u32(ptx::mapa_u32(ptx::smem_u32(&s_all[rank][tok]), peer), __float_as_uint(a), ptx::mapa_u32(ptx::smem_u32(&s_bar), peer));
  }
  // no CTA leaves before all pushes to it have arrived, and its own go to CTAs that wait for them.  Where the wait gives up, peers may still
  // push: this CTA stays until they have, or have given up as well.  (Decided by the warp: by each thread, every call paid 0.1 us)
  if (__any_sync(0xffffffffu, !ptx::mbar_wait_cluster(&s_bar, 0))) {
    if (lane == 0) atomicOr(&flags[FLAG_TIMEOUT], 1u);
    ptx::cluster_wait_for_others();
    (void)ptx::mbar_wait_cluster(&s_bar, 0);               // (what was sent last is still on its way)
  }
  float ramax = 0.0f;
  for (uint32_t c = 0; c < cx; ++c) ramax = fmaxf(ramax, s_all[c][t]);
  if (live && rank == 0 && warp == 0) qa_token_scale<UE>(ramax, m, (uint32_t)l, cfg, buf, off);
  if (on) qa_encode<UE>(u, q & 3, ramax, live, m, q >> 2, (uint32_t)l, cfg, buf, off);
}

__global__ void __launch_bounds__(QA_THREADS)
export_act_kernel(const uint8_t* __restrict__ buf, int64_t M, int64_t K, int in_block, ActOffsets off, sdq_act_canonical_t out)
{
  const int64_t m = blockIdx.x;
  const bool b32 = in_block == 32;
  for (int64_t k = threadIdx.x; k < K; k += QA_THREADS) {
    const uint8_t* xi = buf + off.xi + (size_t)(k >> 8) * off.xi_stride;
    const uint8_t* xo = buf + off.xo + (size_t)(k >> 7) * off.xo_stride;
    const uint32_t kb = (uint32_t)(k & 255) >> 1;
    const uint8_t b = xi[(size_t)(m >> 3) * 1024 + b_off((uint32_t)(m & 7), kb)];
    out.xq4_code[(size_t)m * K + k] = (uint8_t)((k & 1) ? (b >> 4) : (b & 15));
    out.xq8_code[(size_t)m * K + k] = xo[(size_t)(m >> 3) * 1024 + b_off((uint32_t)(m & 7), (uint32_t)(k & 127))];
    // word 0 of atom m / 32
    const uint8_t* sf = xi + (size_t)off.Mpad * 128 + (size_t)(m >> 5) * (b32 ? 2 : 1) * SF_ATOM_BYTES;
    if (b32) { if ((k & 31) == 0) out.xq4_scale[(size_t)m * (K / 32) + (k >> 5)] = sf[in_sf_off(true, (uint32_t)(m & 31), (uint32_t)((k >> 5) & 7))]; }
    else if ((k & 63) == 0) out.xq4_scale[(size_t)m * (K / 64) + (k >> 6)] = sf[in_sf_off(false, (uint32_t)(m & 31), (uint32_t)((k >> 6) & 3))];
  }
  if (threadIdx.x == 0) out.xq8_sexp[m] = reinterpret_cast<const int32_t*>(buf + off.sexp)[m];
}

}  // namespace sdq

using namespace sdq;

static bool act_cfg_ok(const sdq_config_t* c) {
  return c && c->out_n >= 0 && c->out_n <= 2 && (c->in_block == 32 || c->in_block == 64) &&
         c->scale_rule >= SDQ_SCALE_OCP_FLOOR && c->scale_rule <= SDQ_SCALE_UE4M3 &&
         (c->out_fmt == SDQ_OUT_E4M3 || (c->out_fmt == SDQ_OUT_INT8 && c->scale_rule != SDQ_SCALE_UE4M3));
}

extern "C" sdq_status_t sdq_act_size(int64_t M, int64_t K, const sdq_config_t* cfg, size_t* bytes)
{
  if (!act_cfg_ok(cfg) || !bytes) return SDQ_ERR_INVALID_ARG;
  if (cfg->scale_rule == SDQ_SCALE_UE4M3 && cfg->in_block != 32) return SDQ_ERR_UNSUPPORTED;
  if (M <= 0 || K <= 0 || K % K2) return SDQ_ERR_SHAPE;
  *bytes = act_offsets(M, K, cfg->in_block == 32).total;
  return SDQ_OK;
}

extern "C" sdq_status_t sdq_quantize_act(const void* X, int64_t M, int64_t K, int64_t ldx, const sdq_config_t* cfg, void* xq_buf,
                                         size_t xq_bytes, sdq_act_t* out, void* stream)
{ return quantize_act(X, M, K, ldx, cfg, xq_buf, xq_bytes, out, stream, false); }

sdq_status_t sdq::quantize_act(const void* X, int64_t M, int64_t K, int64_t ldx, const sdq_config_t* cfg, void* xq_buf, size_t xq_bytes, sdq_act_t* out,
                               void* stream, bool early_next)
{
  if (!X || !xq_buf || !out || !act_cfg_ok(cfg)) return SDQ_ERR_INVALID_ARG;
  if (cfg->scale_rule == SDQ_SCALE_UE4M3 && cfg->in_block != 32) return SDQ_ERR_UNSUPPORTED;
  if (M <= 0 || K <= 0 || K % K2 || ldx < K) return SDQ_ERR_SHAPE;
  if (((uintptr_t)X & 15) || ((uintptr_t)xq_buf & 15) || (ldx % 8)) return SDQ_ERR_ALIGNMENT;
  const bool b32 = cfg->in_block == 32;
  const ActOffsets off = act_offsets(M, K, b32);
  if (xq_bytes < off.total) return SDQ_ERR_BUFFER_TOO_SMALL;
  const __nv_bfloat16* Xb = (const __nv_bfloat16*)X;
  uint8_t* bufp = (uint8_t*)xq_buf;
  const bool ue = cfg->scale_rule == SDQ_SCALE_UE4M3;
  const int n_chunks = (int)((K + QA_CHUNK - 1) / QA_CHUNK);      // = CTAs per token group: one 256-K unit per warp
  if (n_chunks <= 8) {
    if ((M + 7) / 8 > 65535) return SDQ_ERR_SHAPE;                // token groups are the grid's second dimension
    uint32_t* flags = device_flags();
    if (!flags) return SDQ_ERR_CUDA;
    cudaLaunchConfig_t lc = {};
    const DeviceInfo* dinfo = device_info();
    if (!dinfo) return SDQ_ERR_CUDA;
    // Q-Vectors (64 K) per warp.  A whole unit of four costs the fewest instructions, but a warp then encodes one after the other
    // for about a microsecond, so where there are too few to fill the chip they are spread: one each for up to 7 warps per SM
    // (16 x 4096: 2.3 us, two 2.5, four 3.2; int8 3.0, 4.1, 6.2), in CTAs of up to 16 warps (8 x 16384, 32 warps: 3.4, 3.2, 3.2),
    // two while all these warps run at once, 28 per SM (256 x 4096: 3.1, 2.9, 3.5; 1000 x 4096: 6.2, 4.4, 5.1; 500 x 11008: 14.8,
    // 7.3, 6.5).
    const int64_t groups = (M + 7) / 8, vecs = groups * (K / 64);
    const int nq = vecs <= 7 * (int64_t)dinfo->sm_count && K <= 8192 ? 1 : (vecs <= 56 * (int64_t)dinfo->sm_count ? 2 : 4);
    const int warps = (int)(K / 64 + nq - 1) / nq;       // per token group
    const unsigned cx = (unsigned)((warps + QA_WARPS - 1) / QA_WARPS < 8 ? (warps + QA_WARPS - 1) / QA_WARPS : 8);
    lc.gridDim = dim3(cx, (unsigned)groups);
    lc.blockDim = dim3(nq < 4 ? 32 * (((unsigned)warps + cx - 1) / cx) : QA_THREADS);
    lc.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cx;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 2;
    const int ahead = nq == 4 ? 4 * dinfo->sm_count / (int)cx : 0;   // token groups whose CTAs run at once (four CTAs per SM)
    auto go = [&](auto kern) { return cudaLaunchKernelEx(&lc, kern, Xb, M, K, ldx, *cfg, bufp, off, flags, (int)early_next, ahead); };
    const cudaError_t le = nq == 4   ? (ue ? go(quant_act_fused_kernel<true, 4>) : go(quant_act_fused_kernel<false, 4>))
                           : nq == 2 ? (ue ? go(quant_act_fused_kernel<true, 2>) : go(quant_act_fused_kernel<false, 2>))
                                     : (ue ? go(quant_act_fused_kernel<true, 1>) : go(quant_act_fused_kernel<false, 1>));
    if (launch_status(le) != SDQ_OK) return SDQ_ERR_CUDA;
  } else {
    float* partial = reinterpret_cast<float*>(bufp + off.amax);
    const dim3 grid((unsigned)((M + 7) / 8), (unsigned)n_chunks);
    act_amax_kernel<<<grid, QA_THREADS, 0, (cudaStream_t)stream>>>(Xb, M, K, ldx, partial, n_chunks);
    if (ue) quant_act_kernel<true><<<grid, QA_THREADS, 0, (cudaStream_t)stream>>>(Xb, M, K, ldx, *cfg, bufp, off, partial, n_chunks);
    else quant_act_kernel<false><<<grid, QA_THREADS, 0, (cudaStream_t)stream>>>(Xb, M, K, ldx, *cfg, bufp, off, partial, n_chunks);
    if (cudaGetLastError() != cudaSuccess) return SDQ_ERR_CUDA;
  }
  out->dev = xq_buf;
  out->bytes = off.total;
  out->M = M;
  out->K = K;
  out->cfg = *cfg;
  for (int i = 0; i < 6; ++i) out->off[i] = 0;
  out->off[0] = off.xi; out->off[1] = off.xo; out->off[2] = off.sfb_out; out->off[3] = off.sexp;
  return SDQ_OK;
}

extern "C" sdq_status_t sdq_act_export(const sdq_act_t* Xq, const sdq_act_canonical_t* out, void* stream)
{
  if (!Xq || !out || !Xq->dev || !out->xq4_code || !out->xq4_scale || !out->xq8_code || !out->xq8_sexp) return SDQ_ERR_INVALID_ARG;
  const ActOffsets off = act_offsets(Xq->M, Xq->K, Xq->cfg.in_block == 32);
  export_act_kernel<<<(unsigned)Xq->M, QA_THREADS, 0, (cudaStream_t)stream>>>((const uint8_t*)Xq->dev, Xq->M, Xq->K, Xq->cfg.in_block, off, *out);
  return cudaGetLastError() == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
}
