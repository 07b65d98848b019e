// Grouped decomposed GEMM for few tokens: several independent linear layers in ONE persistent launch
//   Y_i = A_i,in W_i,in^T + A_i,out W_i,out^T   (Section 5.1: O = O_i + O_o, per layer i)
//
// With a handful of tokens a layer is a stream of its packed weights through the tensor core, and one launch per
// layer costs more than the stream itself (set-up, the dependency on the previous grid, the split-K reduction).  Here
// the work items (layer, 128-row tile) of all layers of the call are dealt out round-robin over one CTA per SM; a CTA
// runs its items back to back through its shared-memory rings, so the weights of the next item are already landing
// while the current one is multiplied and stored.  Items left over after the whole rounds -- or all, when there are fewer than
// SMs -- have their K range split over the CTAs of a cluster, which add their parts through distributed shared memory.
//
// The outlier part is streamed in the form the method states it -- an 8-bit code and a position per S-Vector (the WC
// section, 1.5 bits per weight) -- not as the 2:4 FP8 container of the many-token kernels (5 bits per weight): sixteen
// warps in groups of four rebuild the containers of each 256-K unit (one weight row per thread) and write them with
// tcgen05.st into tensor memory, from where the outlier MMAs take their A operand and their metadata, while the tensor
// core works on earlier units.  Shared memory carries every streamed byte once in (bulk copy) and once out (operand
// read); an earlier version that rebuilt the containers in shared memory moved 86 KB per unit through it, two thirds of
// its bandwidth at the rate aimed for, and had room for two container pairs only, whose build -> multiply -> release
// cycle set the pace.  Streamed bytes: 2.625 + 1.5 = 4.125 bits per weight against 4.0 algorithmic.
//
// The stages are organised in units of 256 K of one item, in three rings that fill and drain by themselves: inlier slots (the
// WI record with the tokens' 4-bit codes and scale atom), compact outlier records (two of 128 K), and the tokens' 8-bit codes;
// tensor memory holds one container set per position of the last two.  An inlier slot is free again when the inlier MMAs of
// its unit have completed, a compact record as soon as the builders have read it, codes and container when the outlier MMAs
// have.  What a CTA streams is bytes in flight over a position's round trip (copy 1.3 us, build 0.9, multiply, notice); with one
// ring for everything, released as a whole, that was 2.8 us for eight units, 0.37 us a unit however few CTAs shared the
// DRAM.  With three rings: 74 row tiles of 64 units 27.5 -> 24.4 us, of 16 units 9.6 -> 7.9; q / k / v of 16 tokens 10.2 ->
// 9.5, gate / up 16.4 -> 15.0, 32 layers of 4096 x 4096 53.9 -> 50.5 (46.4 with the matrix of an item looked for from the last
// one on instead of from the first).  Left-over items shared by clusters: 74 row tiles of 64 units 24.4 -> 18.0, gate / up
// 15.0 -> 14.2; one layer 11008 -> 4096 of one token 12.7 (single-layer kernel) -> 10.0.  An mbarrier test costs 15..50 cycles
// when the phase has completed, a tcgen05 instruction ~40 to issue, but a hand-over between roles (complete -> noticed)
// several hundred, so every role keeps its trips few and its waits parallel: where a role waits for several barriers,
// different lanes wait for them at the same time.
//
// Warps: 0, 10 and 24 bulk-copy producers (inlier slots, six lanes / compact records, two lanes / 8-bit codes and the items'
// outlier scale atoms, four lanes), 1 and 23 MMA issuers (inlier / outlier
// product, each into its own accumulator; warp-uniform loops, one elected lane issues; they also copy the inlier metadata
// and the scales to TMEM), 2..5 epilogue (adds the two accumulators; accumulator pairs alternate per item, so the next
// item's MMAs never wait for the stores), 6..9, 11..14, 15..18 and 19..22 container builders (four groups).
// Every wait is bounded; a timeout sets the sticky flag.
//
// Variants.  Outlier operands in int8 (SDQ_OUT_INT8): the same containers and token codes read as integers by a sparse
// kind::i8 MMA into an int32 accumulator; the epilogue converts the exact sums and applies the fp32 row and token scales.
// Activation-resident (template XRES, sdq_linear_group_x): all layers read one bf16 X of up to 16 tokens, which every CTA
// quantizes into its own shared memory (22 warps; the codes, scales and layouts of sdq_quantize_act) while its producers
// already stream weights; the ring slots then hold the weight records only.
//
// What bounds it (measured): with every SM at work the DRAM (0.43 us a unit against 0.385 at its peak), else the ring's round
// trip; the SM's instruction issue is half used, more than half of it by the builders' byte arithmetic.
#include <cuda_bf16.h>

#include "sdq_codec.cuh"
#include "sdq_internal.h"
#include "sdq_layout.h"
#include "sdq_linear.h"
#include "sdq_ptx.cuh"

namespace sdq {

// 25 warps, or 24 when the tokens' codes are resident (no producer for them); 25 take at most 72 registers per thread, since
// seven of them share a register file of 16384
__host__ __device__ constexpr int group_threads(bool xres) { return xres ? 768 : 800; }
constexpr int GRP_UNITS = 8;                     // outlier ring positions (container sets tensor memory holds)
constexpr int GRP_MAX_IN = 12;                   // inlier ring positions: as many as fit, an even number
constexpr int GRP_BUILDERS = 4;                  // builder groups (divides GRP_UNITS: a group then sees every phase of its positions' barriers)
constexpr uint32_t GRP_TM_ACC = 0;               // per item parity 64 columns: O_i at +0, O_o at +32 (32 columns each)
constexpr uint32_t GRP_TM_I = 128;               // 2 x 12: E_in 4 | SFA_in 4 | SFB_in 4
constexpr uint32_t GRP_TM_SO = 152;              // 2 x 8: SFA_out 4 | SFB_out 4 (per item parity)
constexpr uint32_t GRP_TM_C = 168;               // per ring position 40: A_out of the unit's two 128-K stages 2 x 16 | E_out 2 x 4
constexpr uint32_t GRP_TM_C_COLS = 40;
constexpr uint32_t GRP_TMEM_COLS = 512;
constexpr int GRP_BAR_BYTES = (2 * GRP_MAX_IN + 5 * GRP_UNITS + 4 + 2) * 8 + 8;
// activation-resident variant (16 tokens): per 256-K unit the tokens' 4-bit codes, their scale atom and the 8-bit codes of the
// unit's two 128-K stages, in the operand layouts of the quantizer's buffer; then one atom of token scales for the outlier
// product; then the quantizing warps' per-token maxima and the tokens' fp32 scales (int8 outliers)
constexpr uint32_t GRP_XU = 16 * 128 + SF_ATOM_BYTES + 2 * 16 * 128;   // 6656
constexpr int GRP_XQ_WARPS = 22;                                       // every warp but the two producers quantizes
constexpr int GRP_X_TAIL = SF_ATOM_BYTES + GRP_XQ_WARPS * 8 * 4 + 16 * 4 + 64;
__host__ __device__ inline int group_xres_bytes(int T2) { return T2 * (int)GRP_XU + GRP_X_TAIL; }

// inlier slot: | WI record | 4-bit codes of the tokens | their scale atom |
__host__ __device__ inline int group_is_bytes(int n_tile) { return WI_BYTES + n_tile * 128 + SF_ATOM_BYTES; }
// beside the ring: alternating per item, the outlier row / token scale atoms (SFA_out | SFB_out)
constexpr int GRP_SIDE_BYTES = 2 * 2 * SF_ATOM_BYTES;

// A CTA's work is a sequence of segments: whole items dealt round-robin over the CTAs, and at the end, where the items left
// over are fewer than the CTAs, its part of the K range of one of them.  2^p.cluster_log2 CTAs take 2^p.tail_log2 left-over
// items (one each without clusters), 2^(cluster_log2 - tail_log2) CTAs per item.
struct GroupSeg { int item, mat, kb, ke; };                // item, its matrix, its 256-K units [kb, ke)
// segment i, i rising by one from 0 with s.mat = 0 before the first (items only grow, so the matrix is looked for from the last one on)
template <bool SPLIT>
__host__ __device__ __forceinline__ bool group_seg_of(const GroupParams& p, int b, int ctas, int i, GroupSeg& s) {   // CTA b of `ctas`
  const bool whole = !SPLIT || i < p.rounds;
  const int w_log2 = SPLIT ? p.cluster_log2 - p.tail_log2 : 0, r = SPLIT ? b & ((1 << p.cluster_log2) - 1) : 0;
  s.item = whole ? b + i * ctas : p.rounds * ctas + ((b >> p.cluster_log2) << p.tail_log2) + (r >> w_log2);
  if ((SPLIT && i > p.rounds) || s.item >= p.total_items) return false;
  while (s.mat + 1 < p.n && s.item >= p.m[s.mat + 1].item0) ++s.mat;
  const int T2 = p.m[s.mat].T2, part = r & ((1 << w_log2) - 1);
  s.kb = whole ? 0 : (part * T2) >> w_log2;
  s.ke = whole ? T2 : ((part + 1) * T2) >> w_log2;
  return true;
}
template <bool SPLIT>
__device__ __forceinline__ bool group_seg(const GroupParams& p, int i, GroupSeg& s) { return group_seg_of<SPLIT>(p, (int)blockIdx.x, (int)gridDim.x, i, s); }

template <bool F32_OUT, bool XRES, bool SPLIT>
__global__ void __launch_bounds__(group_threads(XRES), 1)
sdq_linear_group_kernel(const __grid_constant__ GroupParams p)
{
  extern __shared__ uint8_t smem_raw[];
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t* sm = smem_raw + ((128 - (ptx::smem_u32(smem_raw) & 127)) & 127);
  constexpr uint32_t NU = GRP_UNITS;
  const uint32_t NI = (uint32_t)p.nslot;                                     // inlier ring positions
  // (activation-resident variant: the slots hold the weight records only)
  const uint32_t xb = (uint32_t)p.n_tile * 128u, isb = XRES ? (uint32_t)WI_BYTES : (uint32_t)group_is_bytes(p.n_tile);
  constexpr uint32_t wcb = 2u * (WC_CODE_BYTES + WC_POS_BYTES);              // the two compact records of a unit
  uint8_t* wc_ring = sm + NI * isb;
  uint8_t* x8_ring = wc_ring + (p.out_n ? NU * wcb : 0u);                    // 8-bit codes of the tokens, 2 x 128 K per position
  uint8_t* xres = x8_ring + (p.out_n && !XRES ? NU * 2u * xb : 0u);          // XRES: the quantized activations of all K
  const uint32_t xres_main = XRES ? (uint32_t)p.m[0].T2 * GRP_XU : 0u;
  uint8_t* x_sfb = xres + xres_main;                                         // XRES: token-scale atom of the outlier product
  float* x_part = reinterpret_cast<float*>(x_sfb + SF_ATOM_BYTES);           // XRES: [quantizing warp][token of its group] maxima
  float* x_sx = x_part + GRP_XQ_WARPS * 8;                                   // XRES: the tokens' fp32 scales (int8 outliers)
  uint8_t* sfbuf = xres + (XRES ? (uint32_t)group_xres_bytes(p.m[0].T2) : 0u);   // 2 x (SFA_out | SFB_out) of the item, alternating
  uint64_t* full_is = reinterpret_cast<uint64_t*>(sfbuf + (p.out_n ? GRP_SIDE_BYTES : 0));  // inlier slot of ring position v has landed
  uint64_t* done_i = full_is + GRP_MAX_IN;                                   // the inlier MMAs of the unit at inlier position v have completed
  uint64_t* full_wc = done_i + GRP_MAX_IN;                                   // compact records of position v have landed
  uint64_t* free_wc = full_wc + GRP_UNITS;                                   // ... have been read by the builders
  uint64_t* full_x8 = free_wc + GRP_UNITS;                                   // 8-bit codes of position v have landed
  uint64_t* built = full_x8 + GRP_UNITS;                                     // the containers of position v are in tensor memory
  uint64_t* done_o = built + GRP_UNITS;                                      // the outlier MMAs of the unit at position v have completed
  uint64_t* acc_full = done_o + GRP_UNITS;                                   // [2]
  uint64_t* acc_empty = acc_full + 2;                                        // [2]
  uint64_t* sf_full = acc_empty + 2;                                         // [2] outlier scale atoms of the item have landed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sf_full + 2);
  volatile uint32_t* timed_out = tmem_slot + 1;                              // a container builder's wait gave up

  if (tid == 0) ptx::griddep_launch_dependents();
  if (tid == 0) {
    *timed_out = 0u;
    const uint32_t issuers = p.out_n ? 2u : 1u;   // MMA-issuing warps: both commit to `acc_full`
    for (uint32_t v = 0; v < NI; ++v) { ptx::mbar_init(&full_is[v], 1); ptx::mbar_init(&done_i[v], 1); }
    for (uint32_t v = 0; v < NU; ++v) {
      ptx::mbar_init(&full_wc[v], 1); ptx::mbar_init(&free_wc[v], 4); ptx::mbar_init(&full_x8[v], 1); ptx::mbar_init(&built[v], 4); ptx::mbar_init(&done_o[v], 1);
    }
    for (int a = 0; a < 2; ++a) { ptx::mbar_init(&acc_full[a], issuers); ptx::mbar_init(&acc_empty[a], 4); ptx::mbar_init(&sf_full[a], 1); }
    ptx::fence_barrier_init();
  }
  if (warp == 1) ptx::tmem_alloc(tmem_slot, GRP_TMEM_COLS);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (XRES && warp != 0 && warp != 10) {
    // ---------------- activation-resident variant: every warp but the producers quantizes the shared X (up to 16 tokens x K)
    // into this CTA's shared memory, in the operand layouts and with the arithmetic of sdq_quantize_act (Section 5, Stage 3:
    // A_i as E2M1 with one scale per 64 K, A_o as E4M3 or int8 per token), while the producers already stream the first
    // weights.  4 lanes per token and Q-Vector as in the quantizer; a warp takes TM tokens (the power of two that holds them
    // all; two groups of 8 above 8 tokens, half the warps each) and 8 / TM Q-Vectors at a time.
    ptx::griddep_wait();                         // X comes from an earlier kernel
    const uint32_t qw = warp - (warp > 10 ? 2u : 1u);      // 0..21
    const uint32_t TM = p.x_M > 4 ? 8u : (p.x_M > 2 ? 4u : (uint32_t)p.x_M), groups = p.x_M > 8 ? 2u : 1u;
    const uint32_t tg = qw % groups, wi = qw / groups, nw = GRP_XQ_WARPS / groups, nq = 8u / TM;
    const uint32_t t = (lane >> 2) % TM, l = lane & 3, qs = (lane >> 2) / TM;
    const uint32_t mtok = tg * 8 + t;
    const bool live = (int)mtok < p.x_M;
    const __nv_bfloat16* xrow = reinterpret_cast<const __nv_bfloat16*>(p.x_bf16) + (int64_t)mtok * p.x_ld;
    const int NB = p.m[0].T2 * 4;                // Q-Vectors of 64 per token
    // one read of X: a lane keeps its (up to six) 16-element pieces in registers across the maxima's barrier
    constexpr int XT = 6;                        // trips per warp: K <= 4096 -> 64 / 11
    const int b0 = (int)(wi * nq + qs), bs = (int)(nw * nq);   // this lane's Q-Vectors: b0, b0 + bs, ...
    uint4 raw[XT][2];
    uint32_t m2 = 0;
#pragma unroll
    for (int i = 0; i < XT; ++i) {
      const int b = b0 + i * bs;
      raw[i][0] = raw[i][1] = make_uint4(0, 0, 0, 0);
      if (live && b < NB) {
        const uint4* src = reinterpret_cast<const uint4*>(xrow + (int64_t)b * 64 + l * 16);
        raw[i][0] = __ldg(src);
        raw[i][1] = __ldg(src + 1);
      }
    }
    // largest magnitude bits of piece i; > 0x7F7F: it holds an infinity (counts as the largest finite bf16)
    auto largest = [&](int i) {
      const uint32_t r[8] = {raw[i][0].x, raw[i][0].y, raw[i][0].z, raw[i][0].w, raw[i][1].x, raw[i][1].y, raw[i][1].z, raw[i][1].w};
      uint32_t q = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) q = max_abs2(q, r[j]);
      return max(q & 0xFFFFu, q >> 16);
    };
#pragma unroll
    for (int i = 0; i < XT; ++i) m2 = max(m2, min(largest(i), 0x7F7Fu));
    float amax = __uint_as_float(m2 << 16);
    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
    for (uint32_t d = 4 * TM; d < 32; d *= 2) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
    if (l == 0 && qs == 0) x_part[qw * 8 + t] = amax;
    ptx::named_bar_sync(8, GRP_XQ_WARPS * 32);
    float ramax = 0.0f;
    for (uint32_t q2 = 0; q2 < nw; ++q2) ramax = fmaxf(ramax, x_part[(groups * q2 + tg) * 8 + t]);
    const int e = fp8_scale_exp(ramax);
    const float s8 = pow2_neg(e), sx = int8_scale(ramax);
    const Int8Coder k8 = int8_coder(sx);
    const bool i8 = p.out_i8 != 0;
    if (wi == 0 && l == 0 && qs == 0) {
      x_sx[mtok] = sx;
      *reinterpret_cast<uint32_t*>(x_sfb + sf_off(mtok, 0)) = (uint32_t)((i8 || !live) ? 127 : e + 127) * 0x01010101u;
    }
#pragma unroll
    for (int i = 0; i < XT; ++i) {
      const int b = b0 + i * bs;
      if (b - (int)qs >= NB) break;               // uniform over the warp
      const uint32_t r[8] = {raw[i][0].x, raw[i][0].y, raw[i][0].z, raw[i][0].w, raw[i][1].x, raw[i][1].y, raw[i][1].z, raw[i][1].w};
      float v[16];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        v[2 * j] = __uint_as_float(r[j] << 16);
        v[2 * j + 1] = __uint_as_float(r[j] & 0xFFFF0000u);
      }
      const uint32_t qmax = largest(i);
      if (qmax > 0x7F7Fu) {
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = sat(v[j]);
      }
      uint32_t bm = min(qmax, 0x7F7Fu);
      bm = max(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
      bm = max(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
      const uint32_t c = e8m0_scale_code_bf16(bm, p.scale_rule == SDQ_SCALE_CEIL_NOSAT);
      const float s4 = pow2_inv_e8m0(c);
      uint32_t q4[2] = {0, 0}, q8[4] = {0, 0, 0, 0};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float f[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = v[8 * h + j] * s4;
        q4[h] = e2m1x8(f);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        q8[j >> 1] |= (i8 ? (int8_code(v[2 * j], k8) | (int8_code(v[2 * j + 1], k8) << 8)) : e4m3x2(v[2 * j] * s8, v[2 * j + 1] * s8)) << (16 * (j & 1));
      }
      if (!live || b >= NB) continue;             // (what the other columns of the product hold is not stored)
      const uint32_t k = (uint32_t)b * 64 + l * 16;          // first element of this lane
      uint8_t* xu = xres + (size_t)(k >> 8) * GRP_XU;
      *reinterpret_cast<uint2*>(xu + b_off(mtok, (k & 255) >> 1)) = make_uint2(q4[0], q4[1]);
      *reinterpret_cast<uint4*>(xu + 16 * 128 + SF_ATOM_BYTES + ((k >> 7) & 1) * 16 * 128 + b_off(mtok, k & 127)) = make_uint4(q8[0], q8[1], q8[2], q8[3]);
      if (l == 0) xu[16 * 128 + in_sf_off(false, mtok, (uint32_t)(b & 3))] = (uint8_t)c;
    }
    ptx::fence_proxy_async();                    // generic-proxy writes -> visible to the tensor core's operand reads
    ptx::named_bar_sync(8, GRP_XQ_WARPS * 32);
  }

  if (warp == 0 || warp == 10 || warp == 24) {
    // ---------------- producers: warp 0 the inlier slots (lane 2 c + l issues copy c of three), warp 10 the compact records,
    // warp 24 the 8-bit codes (copy c of two, one per 128 K).  Lane l of a copy takes the units u = l, l + 2, ... of this CTA's
    // sequence (the rings have an even number of positions, so a lane's positions keep its parity) -- issuing a bulk copy
    // costs its thread ~100 ns, so one instruction issues a copy for each of the lanes instead of one thread all in a row.
    // (Activation-resident variant: warp 0's c = 0 is the one copy of a slot, its c = 1 the row-scale atom of each item.)
    const uint32_t l = lane & 1, c = lane >> 1;
    const bool inl = warp == 0, wc = warp == 10;
    const uint32_t copies = inl ? (XRES ? (p.out_n && !p.out_i8 ? 2u : 1u) : 3u) : (wc ? 1u : 2u);
    if (c < copies && (inl || p.out_n)) {
      bool ok = true;
      GroupSeg sg;                               // this lane's position: segment, unit counted from the segment's start
      int iseq = 0, k = (int)l, k2 = 0, rt = 0;  // ... as work item: 256-K unit, row tile
      bool have = false;
      sg.mat = 0;
      const uint32_t N = inl ? NI : NU;
      uint64_t* freed = inl ? done_i : (wc ? free_wc : done_o);
      uint32_t v = l, wrapped = 0, ph = 0;       // ring position, whether the ring has wrapped, parity of `freed` to wait for
      uint32_t ahead = 0;                        // units whose weights were fetched ahead of the wait below
      // advances to the segment that holds unit k; false at the end of the sequence
      auto seek = [&]() {
        for (;;) {
          if (!have) {
            if (!group_seg<SPLIT>(p, iseq, sg)) return false;
            rt = sg.item - p.m[sg.mat].item0;
            have = true;
          }
          k2 = sg.kb + k;
          if (k2 < sg.ke) return true;
          k = k2 - sg.ke; ++iseq; have = false;
        }
      };
      if (!XRES) {
        // activations come from an earlier kernel.  Packed weights are waited for too, but in calls that start from bf16 activations
        // and are documented to want them complete: there the first lap's inlier records and all compact ones are fetched before the
        // wait (gate / up int8, 5 tokens: 18.0 us per pass waiting for them, 17.3)
        if (p.w_early && inl && c == 0) {
          for (uint32_t u = l; u < NI && seek(); u += 2, k += 2, ++ahead) {
            const GroupMat& m = p.m[sg.mat];
            ptx::mbar_expect_tx(&full_is[u], WI_BYTES + xb + SF_ATOM_BYTES);
            ptx::bulk_g2s(sm + (size_t)u * isb, m.w + m.wi + ((size_t)rt * m.T2 + k2) * WI_BYTES, WI_BYTES, &full_is[u]);
          }
          k = (int)l; iseq = 0; have = false; sg.mat = 0;
        }
        if (!(p.w_early && wc)) ptx::griddep_wait();
      }
      while (seek()) {
        const GroupMat& m = p.m[sg.mat];
        if (wrapped && !(ok = ptx::mbar_wait(&freed[v], ph ^ 1))) break;
        if (inl) {
          uint8_t* st = sm + (size_t)v * isb;
          const uint8_t* wi = m.w + m.wi + ((size_t)rt * m.T2 + k2) * WI_BYTES;
          if (XRES) {
            if (c == 0) {
              ptx::mbar_expect_tx(&full_is[v], WI_BYTES);
              ptx::bulk_g2s(st, wi, WI_BYTES, &full_is[v]);
            } else if (k2 == sg.kb) {            // (see warp 24; the tokens' atom is resident)
              const uint32_t sb = iseq & 1;
              if (iseq >= 2 && !(ok = ptx::mbar_wait(&acc_full[sb], ((iseq >> 1) - 1) & 1))) break;
              ptx::mbar_expect_tx(&sf_full[sb], SF_ATOM_BYTES);
              ptx::bulk_g2s(sfbuf + sb * 2 * SF_ATOM_BYTES, m.w + m.sfa_out + (size_t)rt * SF_ATOM_BYTES, SF_ATOM_BYTES, &sf_full[sb]);
            }
          } else if (ahead) {
            --ahead;
          } else {
            const uint8_t* xi = m.x + m.xi + (size_t)k2 * XI_BYTES;
            if (c == 0) ptx::mbar_expect_tx(&full_is[v], WI_BYTES + xb + SF_ATOM_BYTES);
            const uint32_t off = c == 0 ? 0u : (c == 1 ? (uint32_t)WI_BYTES : (uint32_t)WI_BYTES + xb);
            ptx::bulk_g2s(st + off, c == 0 ? wi : (c == 1 ? xi : xi + B4_BYTES), c == 0 ? (uint32_t)WI_BYTES : (c == 1 ? xb : (uint32_t)SF_ATOM_BYTES), &full_is[v]);
          }
        } else if (wc) {
          ptx::mbar_expect_tx(&full_wc[v], wcb);
          ptx::bulk_g2s(wc_ring + (size_t)v * wcb, m.w + m.wc + ((size_t)rt * m.T2 + k2) * wcb, wcb, &full_wc[v]);
        } else {
          const uint8_t* xo = m.x + m.xo + (size_t)(2 * k2 + (int)c) * XO_BYTES;
          if (c == 0) ptx::mbar_expect_tx(&full_x8[v], 2 * xb);
          ptx::bulk_g2s(x8_ring + (size_t)v * 2 * xb + c * xb, xo, xb, &full_x8[v]);
          if (k2 == sg.kb && !p.out_i8) {        // (int8 outliers take fp32 scales in the epilogue: no scale atoms)
            // the item's outlier scale atoms (lane c = 0: of the weight rows, c = 1: of the tokens): a buffer and a barrier
            // of their own per item parity.  The buffer is free once every MMA of the item two back has completed (`acc_full`
            // of that item: it cannot complete again before these atoms land, since the next item on that accumulator needs
            // them) -- the rings alone do not say so when an item has fewer units than half a ring.
            const uint32_t sb = iseq & 1;
            if (iseq >= 2 && !(ok = ptx::mbar_wait(&acc_full[sb], ((iseq >> 1) - 1) & 1))) break;
            if (c == 0) ptx::mbar_expect_tx(&sf_full[sb], 2u * SF_ATOM_BYTES);
            ptx::bulk_g2s(sfbuf + sb * 2 * SF_ATOM_BYTES + c * SF_ATOM_BYTES, c == 0 ? m.w + m.sfa_out + (size_t)rt * SF_ATOM_BYTES : m.x + m.sfb_out,
                          SF_ATOM_BYTES, &sf_full[sb]);
          }
        }
        k += 2;
        v += 2;
        if (v >= N) { v -= N; wrapped = 1; ph ^= 1; }
      }
      if (!ok) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
    }
  } else if (warp == 1 || warp == 23) {
    // ---------------- MMA issuers: warp 1 the inlier product O_i, warp 23 the outlier product O_o, each into its own
    // accumulator (the epilogue adds them: O = O_i + O_o) -- a tcgen05 instruction costs its issuing thread ~45 cycles, and
    // all of a 256-K unit's in one thread were the longest serial piece of the kernel.  Warp-uniform loops, one elected
    // lane issues (descriptors and TMEM addresses are uniform-register operands).  tcgen05.cp and tcgen05.mma of one
    // thread execute in issue order, so the inlier metadata and the scales need no barrier of their own; their TMEM buffers
    // alternate.  The outlier product takes its A operand and metadata from tensor memory, where the builders put them.
    // Each warp's commits release its own ring's positions.
    const bool outw = warp == 23;
    if (!outw || p.out_n) {
      bool ok = true;
      const uint32_t smb = ptx::smem_u32(sm);
      const uint32_t id4[2] = {ptx::idesc_block_scaled(128, (uint32_t)p.n_tile, 1, true, 0, 0), ptx::idesc_block_scaled(128, (uint32_t)p.n_tile, 1, true, 2, 2)};
      const uint32_t id8 = p.out_i8 ? ptx::idesc_i8(128, (uint32_t)p.n_tile, true) : ptx::idesc_block_scaled(128, (uint32_t)p.n_tile, 0, true, 0, 0);
      const uint32_t N = outw ? NU : NI;
      uint32_t v = 0, ph = 0, itc = 0;             // ring position and its lap parity, item count
      GroupSeg sg;
      sg.mat = 0;
      for (; ok && group_seg<SPLIT>(p, (int)itc, sg); ++itc) {
        const int kb = sg.kb, ke = sg.ke;
        const uint32_t ab = itc & 1, acc_col = tmem + GRP_TM_ACC + 64u * ab + (outw ? 32u : 0u), so = tmem + GRP_TM_SO + 8u * ab;
        if (itc >= 2) {    // the epilogue has read this accumulator pair's previous item
          ok = __all_sync(0xffffffffu, ptx::mbar_wait(&acc_empty[ab], ((itc >> 1) - 1) & 1));
          if (!ok) break;
        }
        for (int k2 = kb; k2 < ke && ok;) {
          // Up to four units of the item per trip: lane i tests unit k2 + i (for the outlier product: lane i its containers,
          // lane 8 + i the tokens' 8-bit codes), lane 4 the item's scale
          // atoms; the units ready in a row from k2 on are issued together.  A trip costs several hundred cycles beside the
          // instructions it issues (test, vote, fence, election, reconvergence), so taking what is ready in one trip keeps
          // the issuer ahead whenever it has fallen behind.  With nothing ready it waits for unit k2 and votes again.
          const int nb = ke - k2 < 4 ? ke - k2 : 4;
          const uint32_t i = lane & 3;
          uint32_t vi = v + i, phi = ph;
          if (vi >= N) { vi -= N; phi ^= 1; }
          const bool sf_lane = outw && k2 == kb && lane == 4 && !p.out_i8, x_lane = outw && !XRES && (lane >> 2) == 2;
          uint64_t* bar = sf_lane ? &sf_full[ab] : (x_lane ? &full_x8[vi] : (outw ? &built[vi] : &full_is[vi]));
          const uint32_t par = sf_lane ? ((itc >> 1) & 1) : phi;
          const bool mine = ((lane < 4 || x_lane) && (int)i < nb) || sf_lane;
          uint32_t ready = __ballot_sync(0xffffffffu, mine ? ptx::mbar_test(bar, par) : (lane == 4));
          if (outw && !XRES) ready &= (ready >> 8) | ~15u;
          int n = __ffs((int)~ready) - 1;          // units ready in a row (lane 4 votes yes when it has nothing to test)
          if (n > nb) n = nb;
          if (!(ready & 16u)) n = 0;
          if (n == 0) {
            ok = __all_sync(0xffffffffu, (lane == 0 || sf_lane || (x_lane && i == 0)) ? ptx::mbar_wait(bar, par) : true);
            continue;
          }
          ptx::tc_fence_after();
          if (ptx::elect_one()) {
            uint32_t vv = v;
            for (int i = 0; i < n; ++i) {
              const int kk = k2 + i;
              const uint32_t sb = smb + vv * isb;
              // the tokens' operands of unit kk: in the slot behind the weight records, or resident
              const uint32_t xu = ptx::smem_u32(xres) + (uint32_t)kk * GRP_XU;
              const uint32_t b4 = XRES ? xu : sb + WI_BYTES, sf4 = XRES ? xu + 16 * 128 : sb + WI_BYTES + xb;
              if (!outw) {
                const uint32_t mb = tmem + GRP_TM_I + 12u * (uint32_t)(kk & 1);
                ptx::tc_cp_128x128b(mb, ptx::smem_desc(sb + A_IN_BYTES, 0, 128));
                ptx::tc_cp_32x128b_warpx4(mb + 4, ptx::smem_desc(sb + A_IN_BYTES + E_IN_BYTES, 0, 128));
                ptx::tc_cp_32x128b_warpx4(mb + 8, ptx::smem_desc(sf4, 0, 128));
                ptx::mma_sp_mxf4(acc_col, ptx::smem_desc(sb, 128, 256), ptx::smem_desc(b4, 128, 1024), id4[0], mb, mb + 4, mb + 8,
                                 kk != kb ? 1u : 0u);
                ptx::mma_sp_mxf4(acc_col, ptx::smem_desc(sb + 4096, 128, 256), ptx::smem_desc(b4 + 512, 128, 1024), id4[1], mb + 2,
                                 mb + 4, mb + 8, 1u);
              } else {
                if (kk == kb && !p.out_i8) {
                  const uint32_t sf = ptx::smem_u32(sfbuf) + ab * 2 * SF_ATOM_BYTES;
                  ptx::tc_cp_32x128b_warpx4(so, ptx::smem_desc(sf, 0, 128));
                  ptx::tc_cp_32x128b_warpx4(so + 4, ptx::smem_desc(XRES ? ptx::smem_u32(x_sfb) : sf + SF_ATOM_BYTES, 0, 128));
                }
#pragma unroll
                for (uint32_t h = 0; h < 2; ++h) {
                  const uint32_t ca = tmem + GRP_TM_C + GRP_TM_C_COLS * vv + 16u * h, eb = tmem + GRP_TM_C + GRP_TM_C_COLS * vv + 32u + 4u * h;
                  const uint32_t xa = XRES ? xu + 16 * 128 + SF_ATOM_BYTES + h * 16 * 128 : ptx::smem_u32(x8_ring) + vv * 2 * xb + h * xb;
                  if (p.out_i8) {     // the same containers and token codes as integers, int32 accumulator
                    ptx::mma_sp_i8_ta(acc_col, ca, ptx::smem_desc(xa, 128, 1024), id8, eb, (kk != kb || h) ? 1u : 0u);
                    ptx::mma_sp_i8_ta(acc_col, ca + 8, ptx::smem_desc(xa + 512, 128, 1024), id8, eb + 2, 1u);
                  } else {
                    ptx::mma_sp_mxf8_ta(acc_col, ca, ptx::smem_desc(xa, 128, 1024), id8, eb, so, so + 4, (kk != kb || h) ? 1u : 0u);
                    ptx::mma_sp_mxf8_ta(acc_col, ca + 8, ptx::smem_desc(xa + 512, 128, 1024), id8, eb + 2, so, so + 4, 1u);
                  }
                }
              }
              ptx::tc_commit(outw ? &done_o[vv] : &done_i[vv]);
              if (kk == ke - 1) ptx::tc_commit(&acc_full[ab]);
              if (++vv == N) vv = 0;
            }
          }
          __syncwarp();
          k2 += n;
          v += (uint32_t)n;
          if (v >= N) { v -= N; ph ^= 1; }
        }
      }
      if (!ok && lane == 0) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
    }
  } else if (warp >= 2 && warp <= 5) {
    // ---------------- epilogue: warp w owns TMEM lanes 32 (w % 4) .. + 31 (weight rows), columns = tokens
    const uint32_t qd = warp & 3;
    bool ok = true;
    uint32_t itc = 0;
    ptx::griddep_wait();                   // Y may still be in use by the previous kernel
    GroupSeg sg;
    sg.mat = 0;
    for (; ok && group_seg<SPLIT>(p, (int)itc, sg); ++itc) {
      const GroupMat& m = p.m[sg.mat];
      const int64_t n0 = (int64_t)(sg.item - m.item0) * TILE_ROWS;
      const bool split = SPLIT && sg.ke - sg.kb < m.T2;      // a part of a left-over item: the last segment
      const uint32_t ab = itc & 1;
      // one thread polls the barrier and releases the other 127 through a hardware barrier: many threads polling an mbarrier
      // slow every other barrier operation of the CTA down
      if (warp == 2 && lane == 0 && !ptx::mbar_wait(&acc_full[ab], (itc >> 1) & 1)) *timed_out = 1u;
      ptx::named_bar_sync(3, 128);
      if (*timed_out) { ok = false; break; }
      ptx::tc_fence_after();
      // int8 outliers: O_o = s_w[row] s_x[token] (exact int32 sum of code products); this thread's row scale
      const float sw = p.out_i8 ? __ldg(reinterpret_cast<const float*>(m.w + m.wsc) + n0 + qd * 32 + lane) : 0.0f;
      const float* sxp = reinterpret_cast<const float*>(m.x + m.xsc);
      uint32_t val[32];
      {
        // O = O_i + O_o: the two partial products of the item, added in fp32
        uint32_t a[16], b[16];
        const uint32_t tb = tmem + ((qd * 32u) << 16) + GRP_TM_ACC + 64u * ab;
#pragma unroll
        for (uint32_t c = 0; c < 32; c += 16) {
          if (c < (uint32_t)p.n_tile) {
            ptx::tmem_ld_32x32b_x16(tb + c, a);
            if (p.out_n) ptx::tmem_ld_32x32b_x16(tb + 32 + c, b);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) val[c + i] = p.out_n ? __float_as_uint(__uint_as_float(a[i]) + __uint_as_float(b[i])) : a[i];
            if (split && p.out_i8) {     // the parts' sums are added as integers, then scaled
              int* pb = reinterpret_cast<int*>(sm + 32 * TILE_ROWS * 4);
#pragma unroll
              for (int i = 0; i < 16; ++i) { val[c + i] = a[i]; pb[(c + i) * TILE_ROWS + qd * 32 + lane] = (int)b[i]; }
            } else if (p.out_i8) {      // b holds exact int32 sums: scale them, tokens that exist only
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float o = (int)(c + i) < m.M ? (float)(int)b[i] * (sw * (XRES ? x_sx[c + i] : __ldg(sxp + c + i))) : 0.0f;
                val[c + i] = __float_as_uint(__uint_as_float(a[i]) + o);
              }
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) val[c + i] = 0u;
          }
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&acc_empty[ab]);
      if (split) {       // to shared memory, where the rings are idle by now
        float* pa = reinterpret_cast<float*>(sm);
#pragma unroll
        for (int t = 0; t < 32; ++t)
          if (t < m.M) pa[t * TILE_ROWS + qd * 32 + lane] = __uint_as_float(val[t]);
        continue;
      }
#pragma unroll
      for (int t = 0; t < 32; ++t) {
        if (t < m.M) {
          const int64_t idx = (int64_t)t * m.ldy + n0 + qd * 32 + lane;
          if (F32_OUT) reinterpret_cast<float*>(m.Y)[idx] = __uint_as_float(val[t]);
          else reinterpret_cast<__nv_bfloat16*>(m.Y)[idx] = __float2bfloat16_rn(__uint_as_float(val[t]));
        }
      }
    }
    if (!ok && lane == 0) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
  } else if (p.out_n && warp >= 6 && warp <= 22) {
    // ---------------- outlier container builders: four groups of four warps (6..9, 11..14, 15..18, 19..22); group g
    // rebuilds the containers of the units u = g, g + 4, ... -- straight into tensor memory, where the outlier MMAs read their
    // A operand and metadata: shared memory is written once (by the bulk copies) and never again.  A warp can reach the 32
    // TMEM lanes 32 (warp % 4) .., so its thread `lane` rebuilds weight row 32 (warp % 4) + lane, both 128-K stages of the
    // unit, each from 16 codes + 16 positions: per S-Vector of 8 the code goes to the 2:4 slot of its group of 4 (two
    // ascending slot indices per 4: (p, 3) with the value first, or (0, 3) with the value second when p = 3; a group without
    // outlier gets (0, 1) and zeros), the form the packer writes for the many-token kernels.  A row's 64 stored bytes per
    // stage are 16 columns of its lane, its 16 metadata bytes 4 columns.  Several groups, because a trip is mostly latency
    // (measured ~1800 cycles, a tenth of it arithmetic): they overlap in time.  Container set v is free when the outlier MMAs of
    // the unit that had it before have completed; the compact record at position v is given back once its codes and positions
    // are in registers.
    const uint32_t bw = warp - (warp >= 11 ? 7u : 6u);       // 0..15
    const uint32_t grp = bw >> 2;
    const uint32_t r = (warp & 3) * 32 + lane;
    const bool poller = (bw & 3u) == 0;
    bool ok = true;
    uint32_t v = 0, ph = 0, lap = 0;             // position of the unit in the ring, lap parity, whether the ring has wrapped
    const uint32_t tlane = tmem + (((warp & 3) * 32u) << 16) + GRP_TM_C;
    GroupSeg sg;
    sg.mat = 0;
    for (int iseq = 0; ok && group_seg<SPLIT>(p, iseq, sg); ++iseq) {
      for (int k2 = sg.kb; k2 < sg.ke; ++k2) {
        if ((v & (GRP_BUILDERS - 1)) == grp) {
          // Only ONE thread of the group waits on the mbarrier and then releases the others through a hardware barrier: with
          // every warp waiting on the same mbarrier some of them noticed its completion more than a microsecond late.
          // (lane 0 waits for the records, lane 1 for the container set)
          if (poller && (lane == 0 || (lane == 1 && lap)) && !ptx::mbar_wait(lane ? &done_o[v] : &full_wc[v], lane ? ph ^ 1 : ph)) *timed_out = 1u;
          ptx::named_bar_sync(4 + grp, 128);   // (barrier 3 belongs to the epilogue)
          if (*timed_out) { ok = false; break; }
          ptx::tc_fence_after();               // the container set is rewritten: after the MMAs that read it
          const uint8_t* st = wc_ring + (size_t)v * wcb;
          uint4 codes[2];
          uint2 pos[2];
#pragma unroll
          for (uint32_t h = 0; h < 2; ++h) {
            codes[h] = *reinterpret_cast<const uint4*>(st + h * (uint32_t)wc_bytes(1) + r * 16);
            pos[h] = *reinterpret_cast<const uint2*>(st + h * (uint32_t)wc_bytes(1) + WC_CODE_BYTES + r * 8);
          }
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&free_wc[v]);
          const uint32_t tc = tlane + GRP_TM_C_COLS * v;
#pragma unroll
          for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t cw[4] = {codes[h].x, codes[h].y, codes[h].z, codes[h].w}, pw[2] = {pos[h].x, pos[h].y};
            // position ps (0..7) of the outlier in its S-Vector: it sits in the group of 4 number ps >> 2 at p = ps & 3.  Stored
            // bytes of the S-Vector (two per group of 4): the code moves to byte (p == 3) + 2 (ps >> 2); metadata byte = the two
            // groups' slot-index nibbles, (p, 3) or (0, 3) for p = 3 where the outlier is, (0, 1) elsewhere.  Both come from
            // 8-entry byte tables held in two registers each, and one byte-permute looks up four S-Vectors at a time: the four
            // position nibbles of a 16-bit piece of the position word are its selector.
            uint32_t stored[16], meta[4], shw[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint32_t sel = pw[i >> 1] >> (16 * (i & 1));
              meta[i] = __byte_perm(0x4C4E4D4Cu, 0xC4E4D4C4u, sel);
              shw[i] = __byte_perm(0x08000000u, 0x18101010u, sel);
            }
#pragma unroll
            for (int g = 0; g < 16; ++g)
              stored[g] = __funnelshift_l(0u, __byte_perm(cw[g >> 2], 0u, 0x4440u + (uint32_t)(g & 3)), shw[g >> 2] >> (8 * (g & 3)));   // (shift count mod 32: the byte's 0 / 8 / 16 / 24)
            // columns 0..7 of the stage: the row's stored bytes of K-block 0 (the first MMA's A), 8..15: of K-block 1
            ptx::tmem_st_32x32b_x16(tc + 16u * h, stored);
            ptx::tmem_st_32x32b_x4(tc + 32u + 4u * h, meta);
          }
          ptx::tmem_st_wait();
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&built[v]);      // one arrival per warp
        }
        if (++v == NU) { v = 0; ph ^= 1; lap = 1; }
      }
    }
    if (!ok && lane == 0) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) ptx::tmem_dealloc(tmem, GRP_TMEM_COLS);
  if constexpr (SPLIT) {
    // ---------------- left-over items: every CTA adds its share of the item's rows over the parts, in order
    ptx::cluster_sync();                           // the parts are in shared memory
    GroupSeg sg;
    sg.mat = 0;
    const uint32_t w_log2 = (uint32_t)(p.cluster_log2 - p.tail_log2), tail_w = 1u << w_log2;   // CTAs per left-over item
    if (group_seg<SPLIT>(p, p.rounds, sg)) {
      const GroupMat& m = p.m[sg.mat];
      const uint32_t rank = ptx::cluster_ctarank(), part = rank & (tail_w - 1u), r0 = rank - part;
      const uint32_t q_per = 32u >> w_log2, q_begin = part * q_per;      // quads of rows
      const uint32_t local = ptx::smem_u32(sm);
      const int64_t n0 = (int64_t)(sg.item - m.item0) * TILE_ROWS;
      for (uint32_t idx = tid; idx < q_per * (uint32_t)m.M; idx += blockDim.x) {
        const uint32_t t = idx >> (5 - w_log2), row = (q_begin + (idx & (q_per - 1u))) << 2, off = (t * TILE_ROWS + row) * 4;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        int4 b = make_int4(0, 0, 0, 0);
        for (uint32_t i = 0; i < tail_w; ++i) {
          const uint32_t peer = ptx::mapa_u32(local, r0 + i) + off;
          const float4 v = ptx::ld_cluster_f32x4(peer);
          a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
          if (p.out_i8) {
            const float4 w = ptx::ld_cluster_f32x4(peer + 32 * TILE_ROWS * 4);
            b.x += __float_as_int(w.x); b.y += __float_as_int(w.y); b.z += __float_as_int(w.z); b.w += __float_as_int(w.w);
          }
        }
        if (p.out_i8) {
          const float4 sw = __ldg(reinterpret_cast<const float4*>(m.w + m.wsc) + (n0 + row) / 4);
          const float sx = XRES ? x_sx[t] : __ldg(reinterpret_cast<const float*>(m.x + m.xsc) + t);
          a.x += (float)b.x * (sw.x * sx); a.y += (float)b.y * (sw.y * sx); a.z += (float)b.z * (sw.z * sx); a.w += (float)b.w * (sw.w * sx);
        }
        const int64_t at = (int64_t)t * m.ldy + n0 + row;
        if (F32_OUT) {
          *reinterpret_cast<float4*>(reinterpret_cast<float*>(m.Y) + at) = a;
        } else {
          const __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
          *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(m.Y) + at) =
              make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        }
      }
    }
    ptx::cluster_sync();                           // nobody leaves while its parts may still be read
  }
}

// inlier ring positions for `n_tile` tokens per tile (an even number, as many as fit beside the outlier rings)
static int group_units(int n_tile, int out_n, int xres_bytes) {
  const int is = xres_bytes ? WI_BYTES : group_is_bytes(n_tile), os = out_n ? 2 * wc_bytes(1) + (xres_bytes ? 0 : 2 * n_tile * 128) : 0;
  const int n = (232448 - 128 - (out_n ? GRP_SIDE_BYTES : 0) - GRP_BAR_BYTES - xres_bytes - GRP_UNITS * os) / is & ~1;
  return n > GRP_MAX_IN ? GRP_MAX_IN : n;
}

// shared-memory budget of the activation-resident variant: do at least six inlier slots fit beside X of K / 256 = T2 units?
bool group_xres_fits(int T2, int out_n) { return group_units(16, out_n, group_xres_bytes(T2)) >= 6; }

// How the items are dealt out: clusters of 1, 2 or 4 CTAs, whole rounds of items, left-over items per cluster.  Times in us,
// fitted to measurements (74 to 1024 items of 4 to 64 units): 3.5 for the launch, 0.28 a unit or 0.42 with every SM
// pulling from DRAM, 2.3 for the clusters and adding the parts.
struct GroupPlan { int cluster, ctas, rounds, tail_items; double us; };
static GroupPlan group_plan(int64_t items, int T2, int T2_min, int sm_count, const int* max_clusters)
{
  GroupPlan best;
  best.us = -1.0;
  for (int c = 1; c <= 4; c *= 2) {
    const int64_t C = c == 1 ? sm_count : (c == 2 ? sm_count / 2 : max_clusters[2]);   // clusters that run at once
    if (C <= 0) continue;
    GroupPlan q;
    q.cluster = c;
    q.rounds = (int)(items / (C * c));
    const int64_t left = items - q.rounds * C * c;
    q.tail_items = c;
    while (q.tail_items > 1 && left <= C * (q.tail_items / 2) && c / (q.tail_items / 2) <= T2_min) q.tail_items /= 2;
    const int w = c / q.tail_items;
    if (c > 1 && w == 1) continue;                      // nothing is split: clusters only cost
    q.ctas = (int)(q.rounds ? C * c : (left + q.tail_items - 1) / q.tail_items * c);
    const double unit = 0.42 * q.ctas / sm_count > 0.28 ? 0.42 * q.ctas / sm_count : 0.28;
    const int64_t tail_ctas = left * w;
    const double tail_unit = 0.42 * tail_ctas / sm_count > 0.28 ? 0.42 * tail_ctas / sm_count : 0.28;
    q.us = 3.5 + q.rounds * T2 * unit + (left ? (double)((T2 + w - 1) / w) * tail_unit : 0.0) + (w > 1 ? 2.3 : 0.0);
    if (best.us < 0 || q.us < best.us) best = q;
  }
  return best;
}
double group_kernel_us(int64_t items, int T2, int sm_count, const int* max_clusters) { return group_plan(items, T2, T2, sm_count, max_clusters).us; }

// how p's items are dealt out, into p
static GroupPlan group_deal(GroupParams& p, int sm_count, const int* max_clusters)
{
  int T2_min = p.m[0].T2;
  int64_t units = 0;
  for (int i = 0; i < p.n; ++i) {
    T2_min = p.m[i].T2 < T2_min ? p.m[i].T2 : T2_min;
    units += (int64_t)((i + 1 < p.n ? p.m[i + 1].item0 : p.total_items) - p.m[i].item0) * p.m[i].T2;
  }
  const GroupPlan plan = group_plan(p.total_items, (int)((units + p.total_items - 1) / p.total_items), T2_min, sm_count, max_clusters);
  auto log2 = [](int v) { return v == 4 ? 2 : v - 1; };
  p.cluster_log2 = log2(plan.cluster); p.tail_log2 = log2(plan.tail_items); p.rounds = plan.rounds;
  return plan;
}

void group_describe(GroupParams p, int sm_count, const int* max_clusters, sdq_diag_plan_t* out, sdq_diag_task_t* segs, int64_t cap)
{
  const GroupPlan plan = group_deal(p, sm_count, max_clusters);
  out->cluster = plan.cluster; out->ctas = plan.ctas; out->rounds = plan.rounds; out->tail_items = plan.tail_items;
  out->ksplit = plan.cluster / plan.tail_items;
  int64_t n = 0;
  for (int b = 0; b < plan.ctas; ++b) {
    GroupSeg s;
    s.mat = 0;
    for (int i = 0; plan.cluster > 1 ? group_seg_of<true>(p, b, plan.ctas, i, s) : group_seg_of<false>(p, b, plan.ctas, i, s); ++i, ++n)
      if (segs && n < cap) segs[n] = {s.mat, s.item - p.m[s.mat].item0, 1, s.kb, s.ke};
  }
  out->tasks = (int32_t)n;
}

cudaError_t launch_linear_group(GroupParams p, bool f32_out, DeviceInfo* d, cudaStream_t stream)
{
  const GroupPlan plan = group_deal(p, d->sm_count, pair_max_clusters(d));
  const bool xres = p.x_bf16 != nullptr;
  const int xbytes = xres ? group_xres_bytes(p.m[0].T2) : 0;
  const int is = xres ? WI_BYTES : group_is_bytes(p.n_tile), os = p.out_n ? 2 * wc_bytes(1) + (xres ? 0 : 2 * p.n_tile * 128) : 0;
  p.nslot = group_units(p.n_tile, p.out_n, xbytes);
  const int smem = p.nslot * is + GRP_UNITS * os + xbytes + (p.out_n ? GRP_SIDE_BYTES : 0) + GRP_BAR_BYTES + 128;
  if (!d->group_attr) {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    bool ok = true;
    auto set = [&](auto kern) { ok = ok && cudaFuncSetAttribute(kern, a, 232448) == cudaSuccess; };
    set(sdq_linear_group_kernel<false, false, false>); set(sdq_linear_group_kernel<true, false, false>);
    set(sdq_linear_group_kernel<false, true, false>); set(sdq_linear_group_kernel<true, true, false>);
    set(sdq_linear_group_kernel<false, false, true>); set(sdq_linear_group_kernel<true, false, true>);
    set(sdq_linear_group_kernel<false, true, true>); set(sdq_linear_group_kernel<true, true, true>);
    if (!ok)
      return cudaErrorUnknown;
    d->group_attr = 1;
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)plan.ctas);
  lc.blockDim = dim3((unsigned)group_threads(xres));
  lc.dynamicSmemBytes = (size_t)smem;
  lc.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)plan.cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = plan.cluster > 1 ? 2 : 1;
  auto go = [&](auto kern) { return cudaLaunchKernelEx(&lc, kern, p); };
  if (plan.cluster > 1) {      // (without left-over items to share the kernel carries no cluster code: 0.6 us a launch)
    if (xres) return f32_out ? go(sdq_linear_group_kernel<true, true, true>) : go(sdq_linear_group_kernel<false, true, true>);
    return f32_out ? go(sdq_linear_group_kernel<true, false, true>) : go(sdq_linear_group_kernel<false, false, true>);
  }
  if (xres) return f32_out ? go(sdq_linear_group_kernel<true, true, false>) : go(sdq_linear_group_kernel<false, true, false>);
  return f32_out ? go(sdq_linear_group_kernel<true, false, false>) : go(sdq_linear_group_kernel<false, false, false>);
}

}  // namespace sdq
