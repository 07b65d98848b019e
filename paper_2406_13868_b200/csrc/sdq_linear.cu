// Fused decomposed GEMM for few tokens (up to 128)  Y = A_i W_i^T + A_o W_o^T   (Section 5.1: O = O_i + O_o), and the
// C-ABI entry points of the linear layer (more tokens: sdq_linear_pair.cu; groups of layers: sdq_linear_group.cu).
//
// The sparse operand of tcgen05.mma.sp is A, so the kernel computes Y^T = W X^T: the 128 weight rows of a
// tile sit on the 128 TMEM lanes, tokens on the accumulator columns.  A tile first runs its inlier K loop
//   2 x tcgen05.mma.sp kind::mxf4 per 256 K     (pair-wise 4:8 E2M1 inliers x E2M1 activations, E8M0 per 64 K)
// then its outlier K loop
//   2 x tcgen05.mma.sp kind::mxf8f6f4 per 128 K (1:8 / 2:8 E4M3 outliers embedded in 2:4 x E4M3 activations;
//                                                the power-of-two row / token scales ride in as E8M0 factors)
// both into ONE fp32 TMEM accumulator (dense / n:8 inliers: 4 x dense tcgen05.mma kind::mxf4 of 64 K per 256 K instead;
// one scale per 32 K: kind::mxf4nvf4 .block16).
// Warp roles: warps 0, 6, 7 = bulk-copy (TMA) producers for weights, activations and scale atoms (issuing a
// bulk copy costs one thread ~50 ns, so the copies of a stage are spread over three threads), warp 1 = TMEM
// owner + MMA issuer (which also moves metadata and scale atoms to TMEM, tcgen05.cp), warps 2..5 = epilogue (tcgen05.ld,
// convert, shared-memory transpose, 16-byte row stores).
// The K range of a row tile is split over several CTAs: either a thread-block cluster whose members
// keep their fp32 partial tiles in shared memory and each add one slice of rows over all members in rank order
// (no global scratch), or, with a caller-provided workspace, partial tiles in global memory that the last CTA to
// arrive adds in split order.  Both orders are fixed.  Launches carry programmatic stream serialization: the
// kernel lets its successor be scheduled at once and itself waits for its predecessor only before it reads
// activations or writes Y.  Every wait is bounded; a timeout sets a sticky flag.
#include <cuda_bf16.h>

#include "sdq_internal.h"
#include "sdq_layout.h"
#include "sdq_linear.h"
#include "sdq_plain.h"
#include "sdq_ptx.cuh"

namespace sdq {

constexpr int LIN_THREADS = 256;   // warps: 0 weight producer, 1 MMA issuer, 2..5 epilogue, 6 activation producer, 7 scale-atom producer
constexpr int MAX_SLOTS = 16;
constexpr int SL_A = 0;                        // WI record (A_in | E_in | SFA_in) or WO record (A_out | E_out)
constexpr int RING_BYTES = 225280;             // largest ring: nslot slots of slot_bytes each
constexpr int SM_TAIL = 4096 + 640 + 128;      // epilogue transpose buffer (16 tokens x 128 features bf16) + barriers + slack
constexpr int LIN_SMEM_MAX = RING_BYTES + SM_TAIL;

// TMEM columns: accumulator at 0 (n_tile columns, tokens), then metadata / scales.
// (84 columns at `meta_col`):
//   +0  2 buffers x 32: E_in 4 | SFA_in 4 or 8 | SFB_in 4 or 8     +64 2 buffers x 4: E_out     +72 SFA_out 4     +76 SFB_out 4
//   (one scale per 64 K: SFA_in 4, SFB_in 4; per 32 K: one scale word per 128-K block, so twice as many)
constexpr uint32_t TM_D = 0;
constexpr uint32_t TM_META_COLS = 84;

// slot = | A record 10752 | B n_tile*128 | scale atoms 1024 |  (inlier: SFB_in, one atom or two with one scale per 32 K; first
// outlier stage: SFA_out | SFB_out)
// (one scale per 32 K: the weight record is 512 B longer; dense inliers: it holds twice the codes and no pattern metadata)
__host__ __device__ inline int slot_bytes_for(int n_tile, bool b32 = false, bool dense = false) {
  return wi_bytes(b32, dense) + n_tile * 128 + 2 * SF_ATOM_BYTES;
}

// 2^ex as a float (ex limited to the normal range), for the exact rescaling of two-level-scaled accumulators
__device__ __forceinline__ float pow2i(int ex) { return __int_as_float((min(max(ex, -126), 127) + 127) << 23); }

struct TileCoord {
  int rt, split;
  int i0, i1, o0, o1;   // inlier stages [i0, i1) of T2, outlier stages [o0, o1) of T1
};
__device__ __forceinline__ TileCoord tile_coord(int ksplit, int tile, int T1, int T2) {
  TileCoord c;
  c.rt = tile / ksplit;
  c.split = tile - c.rt * ksplit;
  c.i0 = c.split * T2 / ksplit;           // 32-bit: split < 32, T1 <= K/128
  c.i1 = (c.split + 1) * T2 / ksplit;
  c.o0 = c.split * T1 / ksplit;
  c.o1 = (c.split + 1) * T1 / ksplit;
  return c;
}

template <bool F32_OUT>
__global__ void __maxnreg__(96)   // two CTAs share an SM only below ~100 registers per thread
sdq_linear_kernel(const LinearParams p)
{
  extern __shared__ uint8_t smem_raw[];
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t* sm = smem_raw + ((128 - (ptx::smem_u32(smem_raw) & 127)) & 127);
  const int ksplit = p.ksplit, cluster_ks = p.cluster_ks;
  const bool release = p.release != 0;
  // the transpose buffer and then the barriers follow the ring
  const uint32_t SM_STG = (uint32_t)p.ring_bytes, SM_BARS = SM_STG + 4096;
  const uint32_t TM_I = (uint32_t)p.meta_col, TM_EO = TM_I + 64, TM_SFA_OUT = TM_I + 72, TM_SFB_OUT = TM_I + 76;
  const uint32_t tmem_cols = (uint32_t)p.tmem_cols;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + SM_BARS);
  uint64_t* empty = full + MAX_SLOTS;
  uint64_t* acc_full = empty + MAX_SLOTS;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
  uint32_t* last_flag = tmem_slot + 1;

  const int n_tile = p.n_tile;
  const int T1 = p.out_n ? (int)(p.K / K1) : 0, T2 = (int)(p.K / K2);
  const uint32_t nslot = (uint32_t)p.nslot, slot_bytes = (uint32_t)p.slot_bytes;
  const bool b32 = p.b32 != 0;                             // one scale per 32 K
  const bool dense = p.dense != 0;                         // dense inliers (always with one scale per 32 K)
  const uint32_t wib = (uint32_t)wi_bytes(b32, dense), na = b32 ? 2u : 1u;
  const uint32_t sl_b = wib;                               // B4 / B8 follow the (longest) weight record
  const uint32_t sl_sf = sl_b + (uint32_t)n_tile * 128u;

  // the coordinates of the first tile are worked out by every thread while the barriers and TMEM are being set up
  // (a lone thread needs ~0.5 us for the integer divisions, which would otherwise delay the first copies)
  const TileCoord first_tc = tile_coord(ksplit, (int)blockIdx.x, T1, T2);
  if (tid == 0) ptx::griddep_launch_dependents();   // the next launch may be scheduled as soon as every CTA got here
  if (tid == 0) {
    for (uint32_t s = 0; s < nslot; ++s) {
      ptx::mbar_init(&full[s], 3);
      ptx::mbar_init(&empty[s], 1);
    }
    ptx::mbar_init(acc_full, 1);
    ptx::mbar_init(acc_empty, 4);
    ptx::fence_barrier_init();
  }
  if (warp == 1) ptx::tmem_alloc(tmem_slot, tmem_cols);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 || warp == 6 || warp == 7) {
    if (lane == 0) {
      // ---------------- producers: role 0 = weight records, role 1 = activation codes, role 2 = scale atoms.
      // Each arrives once per stage on full[s] with the bytes it is about to copy.
      const int role = warp == 0 ? 0 : (int)warp - 5;
      if (role != 0) ptx::griddep_wait();    // activations and their scales come from an earlier kernel; weights do not
      bool ok = true;
      uint32_t s = 0, wrapped = 0, ph = 0;   // ring slot, whether the ring has wrapped, phase parity of `empty`
      for (int tile = blockIdx.x; tile < p.total_tiles && ok; tile += gridDim.x) {
        const TileCoord tc = (tile == (int)blockIdx.x) ? first_tc : tile_coord(ksplit, tile, T1, T2);
        const uint32_t tok_bytes = (uint32_t)n_tile * 128u;                  // (n_tile <= 128 <= Mpad)
        const uint8_t* wi = p.w + p.poff.wi + ((size_t)tc.rt * T2 + tc.i0) * wib;
        const uint8_t* wo = p.w + p.poff.wo + ((size_t)tc.rt * T1 + tc.o0) * WO_BYTES;
        const uint8_t* xi = p.x + p.aoff.xi + (size_t)tc.i0 * p.aoff.xi_stride;
        const uint8_t* xs = xi + (size_t)p.aoff.Mpad * 128u;                 // scale atom 0: the 128 tokens there are room for
        const uint8_t* xo = p.x + p.aoff.xo + (size_t)tc.o0 * p.aoff.xo_stride;
        const int ni = tc.i1 - tc.i0, no = tc.o1 - tc.o0;
        for (int k = 0; k < ni + no; ++k) {
          if (wrapped && release && !(ok = ptx::mbar_wait(&empty[s], ph ^ 1))) break;
          uint8_t* st = sm + (size_t)s * slot_bytes;
          const bool first_o = (k == ni);
          if (role == 0) {
            if (k < ni) {
              ptx::mbar_expect_tx(&full[s], wib);
              ptx::bulk_g2s(st + SL_A, wi, wib, &full[s]);
              wi += wib;
            } else {
              ptx::mbar_expect_tx(&full[s], WO_BYTES + (first_o ? SF_ATOM_BYTES : 0u));
              ptx::bulk_g2s(st + SL_A, wo, WO_BYTES, &full[s]);
              if (first_o) ptx::bulk_g2s(st + sl_sf, p.w + p.poff.sfa_out + (size_t)tc.rt * SF_ATOM_BYTES, SF_ATOM_BYTES, &full[s]);
              wo += WO_BYTES;
            }
          } else if (role == 1) {
            ptx::mbar_expect_tx(&full[s], tok_bytes);
            if (k < ni) {
              ptx::bulk_g2s(st + sl_b, xi, tok_bytes, &full[s]);
              xi += p.aoff.xi_stride;
            } else {
              ptx::bulk_g2s(st + sl_b, xo, tok_bytes, &full[s]);
              xo += p.aoff.xo_stride;
            }
          } else {
            if (k < ni) {
              ptx::mbar_expect_tx(&full[s], na * SF_ATOM_BYTES);
              ptx::bulk_g2s(st + sl_sf, xs, na * SF_ATOM_BYTES, &full[s]);
              xs += p.aoff.xi_stride;
            } else if (first_o) {
              ptx::mbar_expect_tx(&full[s], SF_ATOM_BYTES);
              ptx::bulk_g2s(st + sl_sf + SF_ATOM_BYTES, p.x + p.aoff.sfb_out, SF_ATOM_BYTES, &full[s]);
            } else {
              ptx::mbar_arrive(&full[s]);
            }
          }
          if (++s == nslot) { s = 0; wrapped = 1; ph ^= 1; }
        }
      }
      if (!ok) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer
      bool ok = true;
      const uint32_t smb = ptx::smem_u32(sm);
      uint32_t s = 0, ph = 0, tcount = 0;
      bool ready = false;
      // (two-level scaling: the .block16 kind reads its scale codes as unsigned E4M3 when bit 23 is clear)
      const uint32_t id4[2] = {ptx::idesc_block_scaled(128, (uint32_t)n_tile, 1, true, 0, 0) ^ (p.tw ? (1u << 23) : 0u),
                               ptx::idesc_block_scaled(128, (uint32_t)n_tile, 1, true, 2, 2)};
      const uint32_t id8 = ptx::idesc_block_scaled(128, (uint32_t)n_tile, 0, true, 0, 0);
      const uint32_t idd[2] = {ptx::idesc_block_scaled(128, (uint32_t)n_tile, 1, false, 0, 0),      // dense inliers
                               ptx::idesc_block_scaled(128, (uint32_t)n_tile, 1, false, 2, 2)};
      // descriptors of slot 0; slot s adds s * slot_bytes / 16 to the start-address field
      const uint64_t d_a = ptx::smem_desc(smb + SL_A, 128, 256), d_b = ptx::smem_desc(smb + sl_b, 128, 1024);
      const uint64_t d_e_in = ptx::smem_desc(smb + SL_A + A_IN_BYTES, 0, 128);
      const uint64_t d_sfa_in = ptx::smem_desc(smb + SL_A + (uint32_t)(a_in_bytes(dense) + e_in_bytes(dense)), 0, 128);
      const uint64_t d_e_out = ptx::smem_desc(smb + SL_A + A_OUT_BYTES, 0, 128);
      const uint64_t d_sf0 = ptx::smem_desc(smb + sl_sf, 0, 128), d_sf1 = ptx::smem_desc(smb + sl_sf + SF_ATOM_BYTES, 0, 128);
      const uint32_t slot16 = slot_bytes >> 4;
      for (int tile = blockIdx.x; tile < p.total_tiles && ok; tile += gridDim.x, ++tcount) {
        const TileCoord tc = (tcount == 0) ? first_tc : tile_coord(ksplit, tile, T1, T2);
        const int ni = tc.i1 - tc.i0, no = tc.o1 - tc.o0;
        if (tcount > 0) {   // the epilogue must have drained the accumulator of the previous tile
          ok = ptx::mbar_wait(acc_empty, (tcount - 1) & 1);
          if (!ok) break;
          ptx::tc_fence_after();
        }
        uint32_t acc = 0;   // the first MMA of the tile overwrites the accumulator
        for (int k = 0; k < ni + no; ++k) {
          if (!ready) ok = ptx::mbar_wait(&full[s], ph);
          if (!ok) break;
          ptx::tc_fence_after();
          const uint32_t sn = (s + 1 == nslot) ? 0 : s + 1;
          // poll the next slot now: the answer is back by the time this stage's instructions are issued
          ready = ptx::mbar_test(&full[sn], sn ? ph : ph ^ 1);
          const uint64_t so = (uint64_t)(s * slot16);
          if (k < ni) {
            // inlier stage: 256 logical K = 2 sparse MXFP4 MMAs; metadata and scale atoms go to TMEM first
            const uint32_t mb = tmem + TM_I + 32u * (uint32_t)(k & 1);
            if (!dense) ptx::tc_cp_128x128b(mb + 0, d_e_in + so);
            ptx::tc_cp_32x128b_warpx4(mb + 4, d_sfa_in + so);
            if (!b32) {
              ptx::tc_cp_32x128b_warpx4(mb + 8, d_sf0 + so);
              ptx::mma_sp_mxf4(tmem + TM_D, d_a + so, d_b + so, id4[0], mb, mb + 4, mb + 8, acc);
              ptx::mma_sp_mxf4(tmem + TM_D, d_a + so + (4096 >> 4), d_b + so + (512 >> 4), id4[1], mb + 2, mb + 4, mb + 8, 1u);
            } else {
              // one scale per 32 K: scale word of K-block kb for the weights at mb + 4 + 4 kb, for the tokens at mb + 12 + 4 kb
              ptx::tc_cp_32x128b_warpx4(mb + 8, d_sfa_in + so + (SF_ATOM_BYTES >> 4));
              ptx::tc_cp_32x128b_warpx4(mb + 12, d_sf0 + so);
              ptx::tc_cp_32x128b_warpx4(mb + 16, d_sf1 + so);
              if (!dense) {
                ptx::mma_sp_nvf4(tmem + TM_D, d_a + so, d_b + so, id4[0], mb, mb + 4, mb + 12, acc);
                ptx::mma_sp_nvf4(tmem + TM_D, d_a + so + (4096 >> 4), d_b + so + (512 >> 4), id4[0], mb + 2, mb + 8, mb + 16, 1u);
              } else {
                // dense inliers: four MMAs of 64 K; MMA j reads K-block j of the weights (4096 B apart), bytes 32 j .. 32 j + 31
                // of every token (two 16-byte chunks, 256 B apart per j) and scales 2 (j & 1), 2 (j & 1) + 1 of the scale
                // word of 128-K block j / 2
#pragma unroll
                for (uint32_t j = 0; j < 4; ++j)
                  ptx::mma_mxf4(tmem + TM_D, d_a + so + ((4096 * j) >> 4), d_b + so + ((256 * j) >> 4), idd[j & 1], mb + 4 + 4 * (j >> 1),
                                mb + 12 + 4 * (j >> 1), j ? 1u : acc);
              }
            }
          } else {
            // outlier stage: 128 logical K = 2 sparse FP8 MMAs; the row / token scales (E8M0) arrive with the first one
            const uint32_t eb = tmem + TM_EO + 4u * (uint32_t)(k & 1);
            ptx::tc_cp_128x128b(eb, d_e_out + so);
            if (k == ni) {
              ptx::tc_cp_32x128b_warpx4(tmem + TM_SFA_OUT, d_sf0 + so);
              ptx::tc_cp_32x128b_warpx4(tmem + TM_SFB_OUT, d_sf1 + so);
            }
            ptx::mma_sp_mxf8(tmem + TM_D, d_a + so, d_b + so, id8, eb, tmem + TM_SFA_OUT, tmem + TM_SFB_OUT, acc);
            ptx::mma_sp_mxf8(tmem + TM_D, d_a + so + (4096 >> 4), d_b + so + (512 >> 4), id8, eb + 2, tmem + TM_SFA_OUT,
                             tmem + TM_SFB_OUT, 1u);
          }
          acc = 1;
          if (release) ptx::tc_commit(&empty[s]);   // ring slots are reused only when a CTA runs more stages than slots
          s = sn;
          if (sn == 0) ph ^= 1;
        }
        ptx::tc_commit(acc_full);
      }
      if (!ok) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
    }
  } else {
    // ---------------- epilogue: warp w owns TMEM lanes 32*(w%4) .. +31 (weight rows), columns = tokens
    const uint32_t q = warp & 3;
    const uint32_t et = (warp - 2) * 32 + lane;     // 0..127 among the epilogue threads
    uint32_t tcount = 0;
    bool ok = true;
    ptx::griddep_wait();                            // Y and the workspace may still be in use by the previous kernel
    for (int tile = blockIdx.x; tile < p.total_tiles && ok; tile += gridDim.x, ++tcount) {
      const TileCoord tc = (tcount == 0) ? first_tc : tile_coord(ksplit, tile, T1, T2);
      const int n_valid = (int)p.M;
      ok = ptx::mbar_wait(acc_full, tcount & 1);
      ptx::tc_fence_after();
      if (!ok) break;
      const int64_t n0 = (int64_t)tc.rt * TILE_ROWS;
      const int twr = p.tw ? __ldg(p.tw + n0 + q * 32 + lane) : 0;     // two-level scaling: this thread's row factor
      auto rescale = [&](uint32_t (&v)[16], int c0) {                  // columns c0 .. c0 + 15 of the tile, by 2^(tw + tx)
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (c0 + j < n_valid) v[j] = __float_as_uint(__uint_as_float(v[j]) * pow2i(twr + __ldg(p.tx + c0 + j)));
      };
      // split-K: this CTA's fp32 partial tile [token][128 rows] in the workspace
      float* part = nullptr;
      if (cluster_ks > 1) part = reinterpret_cast<float*>(sm);   // the ring is idle once the accumulator is complete
      else if (ksplit > 1)
        part = p.ws_partial + ((size_t)tc.rt * ksplit + tc.split) * (size_t)n_tile * TILE_ROWS;
      if (part) {
        // split K: all n_tile token columns of the partial tile go out (the reduction reads only the valid ones); the
        // TMEM load of the next 16 columns is in flight while the current 16 are stored
        uint32_t va[16], vb[16];
        const uint32_t tbase = tmem + ((q * 32u) << 16) + TM_D;
        float* dst = part + q * 32 + lane;
        ptx::tmem_ld_32x32b_x16(tbase, va);
#pragma unroll 1
        for (int c0 = 0; c0 < n_tile; c0 += 32) {
          ptx::tmem_ld_wait();
          if (c0 + 16 < n_tile) ptx::tmem_ld_32x32b_x16(tbase + (uint32_t)(c0 + 16), vb);
#pragma unroll
          for (int j = 0; j < 16; ++j) dst[(size_t)(c0 + j) * TILE_ROWS] = __uint_as_float(va[j]);
          if (c0 + 16 < n_tile) {
            ptx::tmem_ld_wait();
            if (c0 + 32 < n_tile) ptx::tmem_ld_32x32b_x16(tbase + (uint32_t)(c0 + 32), va);
#pragma unroll
            for (int j = 0; j < 16; ++j) dst[(size_t)(c0 + 16 + j) * TILE_ROWS] = __uint_as_float(vb[j]);
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(acc_empty);   // accumulator fully read
      }
#pragma unroll 1
      for (int c0 = 0; c0 < (part ? 0 : n_tile); c0 += 16) {
        uint32_t v[16];
        if (c0 < n_valid) {
          ptx::tmem_ld_32x32b_x16(tmem + ((q * 32u) << 16) + TM_D + (uint32_t)c0, v);
          ptx::tmem_ld_wait();
        }
        if (c0 + 16 >= n_tile) {      // accumulator fully read: hand TMEM back before the stores
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(acc_empty);
        }
        if (c0 >= n_valid) continue;  // uniform over the four epilogue warps
        if (p.tw) rescale(v, c0);
        if (F32_OUT) {
          float* Y = reinterpret_cast<float*>(p.Y);
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j < n_valid) Y[(int64_t)(c0 + j) * p.ldy + n0 + q * 32 + lane] = __uint_as_float(v[j]);
        } else {
          // transpose through shared memory: [16 tokens][128 features] bf16, then 16-byte stores of full 256 B rows
          __nv_bfloat16* stg = reinterpret_cast<__nv_bfloat16*>(sm + SM_STG);
#pragma unroll
          for (int j = 0; j < 16; ++j) stg[j * 128 + q * 32 + lane] = __float2bfloat16_rn(__uint_as_float(v[j]));
          ptx::named_bar_sync(1, 128);
          __nv_bfloat16* Y = reinterpret_cast<__nv_bfloat16*>(p.Y);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const uint32_t idx = i * 128 + et, tok = idx >> 4, seg = idx & 15;
            if (c0 + (int)tok < n_valid) {
              const uint4 w = *reinterpret_cast<const uint4*>(stg + tok * 128 + seg * 8);
              *reinterpret_cast<uint4*>(Y + (int64_t)(c0 + tok) * p.ldy + n0 + seg * 8) = w;
            }
          }
          ptx::named_bar_sync(1, 128);   // the buffer is rewritten by the next chunk
        }
      }
      if (part && cluster_ks <= 1) {
        // the last CTA of this (row tile, token tile) to finish adds the partial tiles in split order
        __threadfence();
        ptx::named_bar_sync(1, 128);
        uint32_t* counter = p.ws_counter + tc.rt;
        if (et == 0) {
          const uint32_t old = atomicAdd(counter, 1u);
          *last_flag = (old == (uint32_t)ksplit - 1) ? 1u : 0u;
        }
        ptx::named_bar_sync(1, 128);
        if (*last_flag) {
          __threadfence();
          const float* base = p.ws_partial + (size_t)tc.rt * ksplit * (size_t)n_tile * TILE_ROWS;
          // 8 tokens at a time: the loads of one split are independent, only the adds follow split order
          for (int t0 = 0; t0 < n_valid; t0 += 8) {
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
            for (int sp = 0; sp < ksplit; ++sp) {
              const float* src = base + ((size_t)sp * n_tile + t0) * TILE_ROWS + et;
              float v[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) v[j] = (t0 + j < n_valid) ? __ldcg(src + (size_t)j * TILE_ROWS) : 0.0f;
#pragma unroll
              for (int j = 0; j < 8; ++j) acc[j] += v[j];
            }
            if (p.tw) {
              const int twe = __ldg(p.tw + n0 + et);
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (t0 + j < n_valid) acc[j] *= pow2i(twe + __ldg(p.tx + t0 + j));
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (t0 + j < n_valid) {
                if (F32_OUT) reinterpret_cast<float*>(p.Y)[(int64_t)(t0 + j) * p.ldy + n0 + et] = acc[j];
                else reinterpret_cast<__nv_bfloat16*>(p.Y)[(int64_t)(t0 + j) * p.ldy + n0 + et] = __float2bfloat16_rn(acc[j]);
              }
          }
          if (et == 0) *counter = 0u;     // ready for the next call
        }
        ptx::named_bar_sync(1, 128);       // last_flag is rewritten by the next tile
      }
    }
    if (!ok && lane == 0) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
  }
  if (cluster_ks > 1) {
    // ---------------- cluster split-K: one tile per CTA; CTA r adds its share of the tile's rows over all members
    ptx::cluster_sync();                         // every member's partial tile is in its shared memory
    if (warp >= 2 && warp <= 5) {
      const uint32_t et = (warp - 2) * 32 + lane;
      const uint32_t ks = (uint32_t)cluster_ks, rank = ptx::cluster_ctarank();
      const int n_valid = (int)p.M;
      const int64_t n0 = (int64_t)first_tc.rt * TILE_ROWS;
      const uint32_t local = ptx::smem_u32(sm);
      // four rows x one token per item: one 16-byte load per member, added in rank order.  The 32 quads of rows are
      // dealt out evenly over the members (ks need not divide 32: 3 members take 10, 11 and 11 quads)
      uint32_t peer[8];
#pragma unroll
      for (uint32_t sp = 0; sp < 8; ++sp) peer[sp] = ptx::mapa_u32(local, sp < ks ? sp : 0u);
      const uint32_t q_begin = rank * 32u / ks, q_per = (rank + 1) * 32u / ks - q_begin;
      const uint32_t n_items = q_per * (uint32_t)n_valid;
      auto item_row = [&](uint32_t idx, uint32_t& tok) { tok = idx / q_per; return (q_begin + (idx - tok * q_per)) << 2; };
      auto out4 = [&](uint32_t idx, float4 acc) {
        uint32_t tok;
        const uint32_t row = item_row(idx, tok);
        if (p.tw) {
          const int4 t4 = __ldg(reinterpret_cast<const int4*>(p.tw + n0 + row));
          const int txe = __ldg(p.tx + tok);
          acc.x *= pow2i(t4.x + txe); acc.y *= pow2i(t4.y + txe); acc.z *= pow2i(t4.z + txe); acc.w *= pow2i(t4.w + txe);
        }
        if (F32_OUT) {
          *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.Y) + (int64_t)tok * p.ldy + n0 + row) = acc;
        } else {
          const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
          uint2 w;
          w.x = *reinterpret_cast<const uint32_t*>(&lo);
          w.y = *reinterpret_cast<const uint32_t*>(&hi);
          *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.Y) + (int64_t)tok * p.ldy + n0 + row) = w;
        }
      };
      auto item_off = [&](uint32_t idx) { uint32_t tok; const uint32_t row = item_row(idx, tok); return (tok * TILE_ROWS + row) * 4; };
      // two items per round: up to 16 loads of 16 bytes in flight per thread
      for (uint32_t idx = et; idx < n_items; idx += 256) {
        const uint32_t idx2 = idx + 128;
        const bool two = idx2 < n_items;
        const uint32_t off = item_off(idx), off2 = item_off(two ? idx2 : idx);
        float4 v[8], w[8];
#pragma unroll
        for (uint32_t sp = 0; sp < 8; ++sp) {
          v[sp] = sp < ks ? ptx::ld_cluster_f32x4(peer[sp] + off) : make_float4(0.f, 0.f, 0.f, 0.f);
          w[sp] = (sp < ks && two) ? ptx::ld_cluster_f32x4(peer[sp] + off2) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), acc2 = acc;
#pragma unroll
        for (uint32_t sp = 0; sp < 8; ++sp) {   // rank order; absent members add +0
          acc.x += v[sp].x; acc.y += v[sp].y; acc.z += v[sp].z; acc.w += v[sp].w;
          acc2.x += w[sp].x; acc2.y += w[sp].y; acc2.z += w[sp].z; acc2.w += w[sp].w;
        }
        out4(idx, acc);
        if (two) out4(idx2, acc2);
      }
    }
    ptx::cluster_sync();                         // nobody leaves while its shared memory may still be read
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) ptx::tmem_dealloc(tmem, tmem_cols);
}

}  // namespace sdq

using namespace sdq;

// SM count of the current device (0 on failure)
static int sm_count_current() {
  const DeviceInfo* d = device_info();
  return d ? d->sm_count : 0;
}

// number of K splits for a call: only for M <= 128 (one token tile), as many as keep one CTA per SM,
// never more than the inlier stages so that every split owns at least one
static int choose_ksplit(int64_t M, int64_t N, int64_t K, int sm_count) {
  if (M > 128 || sm_count <= 0) return 1;
  const int RT = (int)(N / TILE_ROWS), T2 = (int)(K / K2);
  // few tokens: short K chains and two small CTAs per SM hide the per-CTA latencies best
  int ks = (M <= 32 ? 2 * sm_count : sm_count) / RT;
  if (ks > T2) ks = T2;
  if (ks > 32) ks = 32;
  return ks < 1 ? 1 : ks;
}
static int n_tile_for(int64_t M) { return (M > 64 ? 128 : (M > 32 ? 64 : (M > 16 ? 32 : 16))); }

// Estimated time of a call of up to 128 tokens on this file's kernel, in us, without a workspace: a fixed part that grows
// with the token tile, and the stored bytes at the rate the split grid streams them (measured on 1024 x 4096 to 16384 x 4096
// and 4096 x 11008 at 1 to 128 tokens: within 10 %)
static double few_token_us(int64_t M, int64_t N, int64_t K, const sdq_config_t& cfg) {
  const double mb = (double)(N / TILE_ROWS) * ((double)(K / K2) * wi_bytes(cfg.in_block == 32, is_dense_layout(cfg)) + (cfg.out_n ? (double)(K / K1) * WO_BYTES : 0.0)) * 1e-6;
  return 5.4 + 0.028 * n_tile_for(M) + (M > 64 ? 0.22 : 0.15) * mb;
}

extern "C" sdq_status_t sdq_workspace_size(int64_t M, int64_t N, int64_t K, const sdq_config_t* cfg, size_t* bytes)
{
  if (!cfg || !bytes) return SDQ_ERR_INVALID_ARG;
  if (M <= 0 || N <= 0 || K <= 0 || N % TILE_ROWS || K % K2) return SDQ_ERR_SHAPE;
  const int ks = choose_ksplit(M, N, K, sm_count_current());
  const size_t RT = (size_t)(N / TILE_ROWS);
  // counters first (one per row tile, 256 B aligned), then ks fp32 partial tiles per row tile
  *bytes = ks > 1 ? ((RT * 4 + 255) & ~(size_t)255) + RT * (size_t)ks * (size_t)n_tile_for(M) * TILE_ROWS * 4 : 0;
  return SDQ_OK;
}

// The grouped kernel carries the primary format: up to 32 tokens, pair-wise 4:8 inliers, one E8M0 scale per 64 K, at most one
// outlier per S-Vector, and K >= 1024, the range it is tested and measured in.  (Its per-item barriers ask for no minimum: an item's
// scale atoms are not overwritten before `acc_full` of it, nor its accumulators before `acc_empty`, so that the last, shared item of a
// CTA may be a single unit.)
static bool group_format(const sdq_config_t& c, int64_t K) {
  return c.in_gran == SDQ_GRAN_PAIR && c.in_block == 64 && c.scale_rule != SDQ_SCALE_UE4M3 && c.out_n <= 1 && K >= 4 * K2;
}
static bool group_kernel_takes(int64_t M, const sdq_packed_t& w) { return M <= 32 && group_format(w.cfg, w.K); }
// launch parameters of `n` layers with the format of `w`, up to `max_m` tokens; then one group_add per layer, in order
static void group_begin(GroupParams& g, int n, int64_t max_m, const sdq_packed_t& w) {
  g.n = n;
  g.n_tile = max_m <= 16 ? 16 : 32;
  g.out_n = w.cfg.out_n;
  g.out_i8 = g.out_n > 0 && w.cfg.out_fmt == SDQ_OUT_INT8;
  g.x_bf16 = nullptr; g.x_ld = 0; g.x_M = 0; g.scale_rule = w.cfg.scale_rule;
  g.w_early = 0;
  g.total_items = 0;
  g.flags = device_flags();
}
// x == nullptr: the layers share g.x_bf16
static void group_add(GroupParams& g, int i, const sdq_act_t* x, const sdq_packed_t& w, void* Y, int64_t ldy, int64_t M) {
  const PackedOffsets po = tiled_offsets(w);
  GroupMat& m = g.m[i];
  m.w = (const uint8_t*)w.dev; m.Y = Y; m.ldy = ldy;
  m.wi = po.wi; m.wc = po.wc; m.sfa_out = po.sfa_out; m.wsc = po.osexp;
  m.x = nullptr; m.xi = m.xo = m.sfb_out = m.xsc = 0;
  if (x) {
    const ActOffsets ao = act_offsets(x->M, x->K, false);
    m.x = (const uint8_t*)x->dev;
    m.xi = ao.xi; m.xo = ao.xo; m.sfb_out = ao.sfb_out; m.xsc = ao.sexp;
  }
  m.M = (int)M; m.T2 = (int)(w.K / K2);
  m.item0 = g.total_items;
  g.total_items += (int)(w.N / TILE_ROWS);
}

// How a single call is run: CTA pairs above 128 tokens.  Up to 128, unless a workspace asks for its split, the kernel with the least
// estimated time: this file's, the pairs, or the grouped kernel on one layer (one token: 4096 x 4096 7.7 -> 7.4 us,
// 4096 -> 11008 12.1 -> 8.7, 11008 -> 4096 12.7 -> 10.0; 100 tokens, 4096 -> 11008: 17.0 -> 15.1 on pairs).
struct LinearRoute { int kernel, ksplit, cluster_ks; };            // SDQ_DIAG_*; the split of K of this file's kernel (cluster_ks = 1: over the workspace)
static LinearRoute linear_route(int64_t M, int64_t N, int64_t K, const sdq_config_t& cfg, bool ws, int sm_count, const int* max_clusters) {
  LinearRoute r = {SDQ_DIAG_PAIRS, 1, 1};
  if (M > 128) return r;
  if (ws) {
    r.ksplit = choose_ksplit(M, N, K, sm_count);
    if (r.ksplit > 1) { r.kernel = SDQ_DIAG_FEW; return r; }
  }
  const bool dense = is_dense_layout(cfg);
  const int tiles = (int)(N / TILE_ROWS), T2 = (int)(K / K2);
  const double few = few_token_us(M, N, K, cfg), two = pair_kernel_us(M, N, K, cfg.out_n, cfg.in_block == 32, dense, sm_count, max_clusters);
  if (M <= 32 && group_format(cfg, K)) {
    const double one = group_kernel_us(tiles, T2, sm_count, max_clusters);
    if (one < few && one < two) { r.kernel = SDQ_DIAG_GROUP; return r; }
  }
  if (two < few) return r;
  r.kernel = SDQ_DIAG_FEW;
  // cluster split-K: a cluster of up to 8 CTAs per row tile, one tile per CTA
  // as many members (1..8) as the budget and the inlier stages allow.  Clusters are placed inside one GPC, whose SM count
  // varies: sizes 3, 5, 6, 7 pack worse than powers of two, and a grid that needs every slot then runs a second wave
  // (96 clusters of 3 took 21 us, 96 of 2 take 14), so odd sizes only get 88 % of the budget
  auto split_for = [&](int cta_budget) {
    for (int k = 8; k > 1; --k) {
      const bool pow2 = (k & (k - 1)) == 0;
      if (k <= T2 && (int64_t)k * tiles <= (pow2 ? cta_budget : cta_budget * 22 / 25)) return k;
    }
    return 1;
  };
  // CTAs the grid may have: up to 64 tokens the CTAs are small enough for two per SM; from 65 to 128 tokens two
  // per SM leave only three ring slots, which pays only when one per SM would leave many SMs idle
  int ks = split_for(M <= 64 ? 2 * sm_count : sm_count);
  if (M > 64 && ks * tiles * 5 <= sm_count * 3) ks = split_for(2 * sm_count);
  // more row tiles than SMs: one CTA per SM walking whole-K tiles streams a tile in ~19 us however few tiles its
  // last round holds (149 tiles took 38 us, 148 took 16), while two half-K CTAs per SM keep more bytes in flight;
  // split in two and let the grid run in waves of two CTAs per SM (K >= 2048: below that the halves are too short)
  if (ks == 1 && tiles > sm_count && T2 >= 8) ks = 2;
  r.ksplit = r.cluster_ks = ks;
  return r;
}

static sdq_status_t launch_linear(const sdq_act_t* Xq, const sdq_packed_t* P, void* Y, int64_t ldy, void* ws, size_t ws_bytes,
                                  void* stream, bool f32)
{
  if (!Xq || !P || !Y || !Xq->dev || !P->dev) return SDQ_ERR_INVALID_ARG;
  if (Xq->K != P->K || Xq->M <= 0 || P->N <= 0 || P->N % TILE_ROWS || P->K % K2 || ldy < P->N) return SDQ_ERR_SHAPE;
  if (Xq->cfg.in_block != P->cfg.in_block || Xq->cfg.scale_rule != P->cfg.scale_rule) return SDQ_ERR_SHAPE;
  if (!is_tensor_core_reading(P->cfg)) return SDQ_ERR_UNSUPPORTED;
  if (P->cfg.out_n > 0 && Xq->cfg.out_fmt != P->cfg.out_fmt) return SDQ_ERR_SHAPE;
  if (P->cfg.out_n > 0 && P->cfg.out_fmt == SDQ_OUT_INT8) return SDQ_ERR_UNSUPPORTED;   // int8 outliers: the grouped few-token kernel only
  if (is_compact(*P)) return SDQ_ERR_UNSUPPORTED;                                       // no 2:4 containers in the buffer: likewise
  if (P->cfg.scale_rule == SDQ_SCALE_UE4M3 && !(P->cfg.in_gran == SDQ_GRAN_PAIR && P->cfg.in_block == 32)) return SDQ_ERR_UNSUPPORTED;
  if (((uintptr_t)Y & 15) || (ldy % 8) || ((uintptr_t)ws & 15)) return SDQ_ERR_ALIGNMENT;
  DeviceInfo* dinfo = device_info();
  if (!dinfo) return SDQ_ERR_CUDA;
  if (!dinfo->linear_attr) {     // function attributes belong to the device's context: once per device
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (cudaFuncSetAttribute(sdq_linear_kernel<true>, a, LIN_SMEM_MAX) != cudaSuccess ||
        cudaFuncSetAttribute(sdq_linear_kernel<false>, a, LIN_SMEM_MAX) != cudaSuccess)
      return SDQ_ERR_CUDA;
    dinfo->linear_attr = 1;
  }
  const int sm_count = dinfo->sm_count;
  LinearParams p;
  p.w = (const uint8_t*)P->dev;
  p.x = (const uint8_t*)Xq->dev;
  p.b32 = P->cfg.in_block == 32 ? 1 : 0;
  const bool ue = P->cfg.scale_rule == SDQ_SCALE_UE4M3;
  p.dense = is_dense_layout(P->cfg) ? 1 : 0;   // the n:8, 3:4 and element-wise 2:4 patterns are stored and run like the dense one
  p.poff = tiled_offsets(P->N, P->K, P->cfg);
  p.aoff = act_offsets(Xq->M, Xq->K, p.b32 != 0);
  p.tw = ue ? reinterpret_cast<const int32_t*>(p.w + p.poff.wtexp) : nullptr;
  p.tx = reinterpret_cast<const int32_t*>(p.x + p.aoff.sexp);
  p.M = Xq->M; p.N = P->N; p.K = P->K;
  p.out_n = P->cfg.out_n;
  const int64_t M = Xq->M;
  p.ws_counter = nullptr;
  p.ws_partial = nullptr;
  p.Y = Y; p.ldy = ldy;
  p.flags = device_flags();
  if (!p.flags) return SDQ_ERR_CUDA;
  const LinearRoute route = linear_route(M, P->N, P->K, P->cfg, ws != nullptr, sm_count, pair_max_clusters(dinfo));
  if (route.kernel == SDQ_DIAG_GROUP) {
    GroupParams g;
    group_begin(g, 1, M, *P);
    if (!g.flags) return SDQ_ERR_CUDA;
    group_add(g, 0, Xq, *P, Y, ldy, M);
    return launch_status(launch_linear_group(g, f32, dinfo, (cudaStream_t)stream));
  }
  if (route.kernel == SDQ_DIAG_PAIRS) return launch_status(launch_linear_pair(p, f32, dinfo, (cudaStream_t)stream));
  p.n_tile = n_tile_for(M);
  p.slot_bytes = slot_bytes_for(p.n_tile, p.b32 != 0, p.dense != 0);
  const int tiles = (int)(P->N / TILE_ROWS);
  p.ksplit = route.ksplit;
  p.cluster_ks = route.cluster_ks;
  if (p.ksplit > 1 && p.cluster_ks == 1) {
    size_t need = 0;
    sdq_workspace_size(M, P->N, P->K, &P->cfg, &need);
    if (ws_bytes < need) return SDQ_ERR_BUFFER_TOO_SMALL;
    p.ws_counter = (uint32_t*)ws;
    p.ws_partial = (float*)((uint8_t*)ws + (((size_t)tiles * 4 + 255) & ~(size_t)255));
  }
  p.total_tiles = tiles * p.ksplit;
  // ring geometry: a CTA that runs a single tile with no more stages than fit never reuses a slot, needs only as
  // much shared memory as its stages take (so that small CTAs share an SM) and skips the slot-release traffic
  const int T1 = p.out_n ? (int)(P->K / K1) : 0, T2 = (int)(P->K / K2);
  const int stages_per_tile = (T2 + p.ksplit - 1) / p.ksplit + (T1 + p.ksplit - 1) / p.ksplit;
  int max_slots = RING_BYTES / p.slot_bytes;
  if (p.cluster_ks > 1 && p.total_tiles > sm_count) {
    // cluster split K with more CTAs than SMs (few tokens, one tile per CTA): the grid is one wave only if two CTAs
    // share an SM, so a ring gets half of an SM's shared memory (228 KB, 1 KB of it reserved per CTA)
    const int half = (233472 / 2 - 1024 - SM_TAIL) / p.slot_bytes;
    if (half < max_slots) max_slots = half;
  }
  if (max_slots > MAX_SLOTS) max_slots = MAX_SLOTS;
  int grid_x;
  if (p.total_tiles <= 2 * sm_count && stages_per_tile <= max_slots && p.n_tile <= 32) {
    grid_x = p.total_tiles;
    p.nslot = stages_per_tile;
    p.release = 0;
  } else if (p.cluster_ks > 1) {
    grid_x = p.total_tiles;          // one tile per CTA (the cluster reduction relies on it); total_tiles <= SM count
    p.nslot = max_slots;
    p.release = 1;
  } else {
    grid_x = p.total_tiles < sm_count ? p.total_tiles : sm_count;
    p.nslot = max_slots;
    p.release = 1;
  }
  p.ring_bytes = p.nslot * p.slot_bytes;
  p.meta_col = p.n_tile < 32 ? 32 : p.n_tile;
  int cols = p.meta_col + (int)TM_META_COLS;
  p.tmem_cols = cols <= 128 ? 128 : (cols <= 256 ? 256 : 512);
  const int smem = p.ring_bytes + SM_TAIL;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)grid_x);
  lc.blockDim = dim3(LIN_THREADS);
  lc.dynamicSmemBytes = (size_t)smem;
  lc.stream = (cudaStream_t)stream;
  // the kernel may be scheduled while the previous one in the stream drains: set-up and weight copies overlap its tail
  cudaLaunchAttribute attr[2];
  int na = 0;
  attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[na].val.programmaticStreamSerializationAllowed = 1;
  ++na;
  if (p.cluster_ks > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = (unsigned)p.cluster_ks;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  lc.attrs = attr;
  lc.numAttrs = na;
  const cudaError_t le = f32 ? cudaLaunchKernelEx(&lc, sdq_linear_kernel<true>, p) : cudaLaunchKernelEx(&lc, sdq_linear_kernel<false>, p);
  return launch_status(le);
}

extern "C" sdq_status_t sdq_linear(const sdq_act_t* Xq, const sdq_packed_t* P, void* Y, int64_t ldy, void* stream)
{ return launch_linear(Xq, P, Y, ldy, nullptr, 0, stream, false); }

extern "C" sdq_status_t sdq_linear_f32(const sdq_act_t* Xq, const sdq_packed_t* P, float* Y, int64_t ldy, void* stream)
{ return launch_linear(Xq, P, (void*)Y, ldy, nullptr, 0, stream, true); }

extern "C" sdq_status_t sdq_workspace_init(void* ws, size_t ws_bytes, void* stream)
{
  if (!ws) return SDQ_ERR_INVALID_ARG;
  if ((uintptr_t)ws & 15) return SDQ_ERR_ALIGNMENT;
  return cudaMemsetAsync(ws, 0, ws_bytes, (cudaStream_t)stream) == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
}

extern "C" sdq_status_t sdq_linear_ws(const sdq_act_t* Xq, const sdq_packed_t* P, void* Y, int64_t ldy, void* ws, size_t ws_bytes,
                                      void* stream)
{ return launch_linear(Xq, P, Y, ldy, ws, ws_bytes, stream, false); }

extern "C" sdq_status_t sdq_linear_f32_ws(const sdq_act_t* Xq, const sdq_packed_t* P, float* Y, int64_t ldy, void* ws, size_t ws_bytes,
                                          void* stream)
{ return launch_linear(Xq, P, (void*)Y, ldy, ws, ws_bytes, stream, true); }

// ---------------------------------------------------------------------------------------------------------
// Several independent layers in one call (see include/sdq.h).  Few tokens everywhere and enough row tiles to occupy
// the GPU: one persistent launch of the grouped kernel; otherwise the layers are enqueued one after the other.
static sdq_status_t launch_group(int n, const sdq_act_t* const* Xq, const sdq_packed_t* const* P, void* const* Y, const int64_t* ldy,
                                 void* stream, bool f32)
{
  if (n <= 0 || !Xq || !P || !Y || !ldy) return SDQ_ERR_INVALID_ARG;
  DeviceInfo* dinfo = device_info();
  if (!dinfo) return SDQ_ERR_CUDA;
  bool fused = n <= GROUP_MAX;
  int64_t items = 0, max_m = 0;
  for (int i = 0; i < n; ++i) {
    const sdq_act_t* x = Xq[i];
    const sdq_packed_t* w = P[i];
    if (!x || !w || !Y[i] || !x->dev || !w->dev) return SDQ_ERR_INVALID_ARG;
    if (x->K != w->K || x->M <= 0 || w->N <= 0 || w->N % TILE_ROWS || w->K % K2 || ldy[i] < w->N) return SDQ_ERR_SHAPE;
    if (x->cfg.in_block != w->cfg.in_block || x->cfg.scale_rule != w->cfg.scale_rule) return SDQ_ERR_SHAPE;
    if (!is_tensor_core_reading(w->cfg)) return SDQ_ERR_UNSUPPORTED;
    if (w->cfg.out_n > 0 && x->cfg.out_fmt != w->cfg.out_fmt) return SDQ_ERR_SHAPE;
    if (((uintptr_t)Y[i] & 15) || (ldy[i] % 8)) return SDQ_ERR_ALIGNMENT;
    fused = fused && group_kernel_takes(x->M, *w) && w->cfg.out_n == P[0]->cfg.out_n && w->cfg.out_fmt == P[0]->cfg.out_fmt;
    items += w->N / TILE_ROWS;
    if (x->M > max_m) max_m = x->M;
  }
  fused = fused && items * 2 >= dinfo->sm_count && items < (1 << 30);
  if (!fused) {
    for (int i = 0; i < n; ++i) {
      const sdq_status_t st = launch_linear(Xq[i], P[i], Y[i], ldy[i], nullptr, 0, stream, f32);
      if (st != SDQ_OK) return st;
    }
    return SDQ_OK;
  }
  GroupParams g;
  group_begin(g, n, max_m, *P[0]);
  if (!g.flags) return SDQ_ERR_CUDA;
  for (int i = 0; i < n; ++i) group_add(g, i, Xq[i], *P[i], Y[i], ldy[i], Xq[i]->M);
  const cudaError_t e = launch_linear_group(g, f32, dinfo, (cudaStream_t)stream);
  return launch_status(e);
}

// The same from one bf16 X that all layers read (see include/sdq.h): with scratch, the quantizer's launch and then the grouped
// kernel's, whose first weights are on their way while the quantizer runs; without, the quantizer inside the kernel, once per
// CTA.  gate and up of 11008 x 4096, 1 / 5 / 16 tokens: 15.3 / 15.5 / 15.7 us against 15.5 / 17.2 / 20.5, int8 outliers 16.0 / 16.2 /
// 16.6 against 16.3 / 19.8 / 25.8; three of 8192 x 1024: 8.0 / 8.1 / 8.9 against 8.9 / 9.1 / 9.8.
static sdq_status_t launch_group_x(int n, const void* X, int64_t M, int64_t K, int64_t ldx, const sdq_packed_t* const* P, void* const* Y,
                                   const int64_t* ldy, void* ws, size_t ws_bytes, void* stream, bool f32)
{
  if (n <= 0 || !X || !P || !Y || !ldy) return SDQ_ERR_INVALID_ARG;
  if (M <= 0 || K <= 0 || K % K2 || ldx < K) return SDQ_ERR_SHAPE;
  if (((uintptr_t)X & 15) || (ldx % 8)) return SDQ_ERR_ALIGNMENT;
  DeviceInfo* dinfo = device_info();
  if (!dinfo) return SDQ_ERR_CUDA;
  int64_t items = 0;
  for (int i = 0; i < n; ++i) {
    const sdq_packed_t* w = P[i];
    if (!w || !Y[i] || !w->dev) return SDQ_ERR_INVALID_ARG;
    if (w->K != K || w->N <= 0 || w->N % TILE_ROWS || ldy[i] < w->N) return SDQ_ERR_SHAPE;
    if (!is_tensor_core_reading(w->cfg)) return SDQ_ERR_UNSUPPORTED;
    if (((uintptr_t)Y[i] & 15) || (ldy[i] % 8)) return SDQ_ERR_ALIGNMENT;
    const sdq_config_t& c = w->cfg, &c0 = P[0]->cfg;
    if (!group_format(c, w->K) || c.out_n != c0.out_n || c.out_fmt != c0.out_fmt || c.scale_rule != c0.scale_rule) return SDQ_ERR_UNSUPPORTED;
    items += w->N / TILE_ROWS;
  }
  // (the same range with and without scratch: the in-kernel quantizer keeps a token's K <= 4096 elements in the registers of its 11 x 4 lanes)
  if (n > GROUP_MAX || M > 16 || K < 4 * K2 || K > 16 * K2 || !group_xres_fits((int)(K / K2), P[0]->cfg.out_n) || items * 2 < dinfo->sm_count || items >= (1 << 30))
    return SDQ_ERR_UNSUPPORTED;
  GroupParams g;
  group_begin(g, n, M, *P[0]);
  if (!g.flags) return SDQ_ERR_CUDA;
  sdq_act_t xq;
  if (ws) {
    const sdq_status_t st = quantize_act(X, M, K, ldx, &P[0]->cfg, ws, ws_bytes, &xq, stream, true);
    if (st != SDQ_OK) return st;
    g.w_early = 1;
  } else {
    g.x_bf16 = X; g.x_ld = ldx; g.x_M = (int)M;
  }
  for (int i = 0; i < n; ++i) group_add(g, i, ws ? &xq : nullptr, *P[i], Y[i], ldy[i], M);
  const cudaError_t e = launch_linear_group(g, f32, dinfo, (cudaStream_t)stream);
  return launch_status(e);
}

extern "C" sdq_status_t sdq_linear_group_x(int n, const void* X_bf16, int64_t M, int64_t K, int64_t ldx, const sdq_packed_t* const* P,
                                           void* const* Y, const int64_t* ldy, void* stream)
{ return launch_group_x(n, X_bf16, M, K, ldx, P, Y, ldy, nullptr, 0, stream, false); }

extern "C" sdq_status_t sdq_linear_group_x_f32(int n, const void* X_bf16, int64_t M, int64_t K, int64_t ldx, const sdq_packed_t* const* P,
                                               float* const* Y, const int64_t* ldy, void* stream)
{ return launch_group_x(n, X_bf16, M, K, ldx, P, (void* const*)Y, ldy, nullptr, 0, stream, true); }

extern "C" sdq_status_t sdq_linear_group_x_ws(int n, const void* X_bf16, int64_t M, int64_t K, int64_t ldx, const sdq_packed_t* const* P,
                                              void* const* Y, const int64_t* ldy, void* ws, size_t ws_bytes, void* stream)
{ return launch_group_x(n, X_bf16, M, K, ldx, P, Y, ldy, ws, ws_bytes, stream, false); }

extern "C" sdq_status_t sdq_linear_group_x_f32_ws(int n, const void* X_bf16, int64_t M, int64_t K, int64_t ldx, const sdq_packed_t* const* P,
                                                  float* const* Y, const int64_t* ldy, void* ws, size_t ws_bytes, void* stream)
{ return launch_group_x(n, X_bf16, M, K, ldx, P, (void* const*)Y, ldy, ws, ws_bytes, stream, true); }

extern "C" sdq_status_t sdq_linear_group(int n, const sdq_act_t* const* Xq, const sdq_packed_t* const* P, void* const* Y,
                                         const int64_t* ldy, void* stream)
{ return launch_group(n, Xq, P, Y, ldy, stream, false); }

extern "C" sdq_status_t sdq_linear_group_f32(int n, const sdq_act_t* const* Xq, const sdq_packed_t* const* P, float* const* Y,
                                             const int64_t* ldy, void* stream)
{ return launch_group(n, Xq, P, (void* const*)Y, ldy, stream, true); }

// ---------------------------------------------------------------------------------------------------------
// What a call would run, for tests (see include/sdq_diag.h): the functions above decide, nothing is launched.
static bool diag_machine(int& sm_count, const int*& max_clusters) {
  static const int none[5] = {0, 0, 0, 0, 0};
  if (sm_count > 0) { if (!max_clusters) max_clusters = none; return true; }
  DeviceInfo* d = device_info();
  if (!d) return false;
  sm_count = d->sm_count; max_clusters = pair_max_clusters(d);
  return true;
}

static LinearParams pair_params(int64_t M, int64_t N, int64_t K, const sdq_config_t& cfg) {
  LinearParams p = {};
  p.M = M; p.N = N; p.K = K; p.out_n = cfg.out_n; p.b32 = cfg.in_block == 32; p.dense = is_dense_layout(cfg);
  return p;
}

extern "C" sdq_status_t sdq_diag_linear_plan(int64_t M, int64_t N, int64_t K, const sdq_config_t* cfg, int workspace, int sm_count,
                                             const int* max_clusters, sdq_diag_plan_t* out, sdq_diag_task_t* tasks, int64_t cap)
{
  if (!cfg || !out) return SDQ_ERR_INVALID_ARG;
  if (M <= 0 || N <= 0 || K <= 0 || N % TILE_ROWS || K % K2) return SDQ_ERR_SHAPE;
  if (!is_tensor_core_reading(*cfg)) return SDQ_ERR_UNSUPPORTED;
  if (!diag_machine(sm_count, max_clusters)) return SDQ_ERR_CUDA;
  *out = sdq_diag_plan_t{};
  const LinearRoute r = linear_route(M, N, K, *cfg, workspace != 0, sm_count, max_clusters);
  out->kernel = r.kernel;
  if (r.kernel == SDQ_DIAG_FEW) { out->ksplit = r.ksplit; out->cluster = r.cluster_ks; out->token_tile = n_tile_for(M); }
  if (r.kernel == SDQ_DIAG_PAIRS) pair_describe(pair_params(M, N, K, *cfg), sm_count, max_clusters, out, tasks, cap);
  if (r.kernel == SDQ_DIAG_GROUP) return sdq_diag_group_plan(1, M, &N, &K, sm_count, max_clusters, out, tasks, cap);
  return SDQ_OK;
}

extern "C" sdq_status_t sdq_diag_linear_rings(int64_t M, int64_t N, int64_t K, const sdq_config_t* cfg, int sm_count, const int* max_clusters,
                                              sdq_diag_rings_t* out)
{
  sdq_diag_plan_t plan;
  if (!out) return SDQ_ERR_INVALID_ARG;
  const sdq_status_t st = sdq_diag_linear_plan(M, N, K, cfg, 0, sm_count, max_clusters, &plan, nullptr, 0);
  if (st != SDQ_OK) return st;
  *out = sdq_diag_rings_t{};
  if (plan.kernel != SDQ_DIAG_PAIRS) return SDQ_OK;
  if (!diag_machine(sm_count, max_clusters)) return SDQ_ERR_CUDA;
  pair_describe_rings(pair_params(M, N, K, *cfg), sm_count, max_clusters, out);
  return SDQ_OK;
}

extern "C" sdq_status_t sdq_diag_group_plan(int n, int64_t M, const int64_t* N, const int64_t* K, int sm_count, const int* max_clusters,
                                            sdq_diag_plan_t* out, sdq_diag_task_t* segs, int64_t cap)
{
  if (n <= 0 || n > GROUP_MAX || !N || !K || !out) return SDQ_ERR_INVALID_ARG;
  if (!diag_machine(sm_count, max_clusters)) return SDQ_ERR_CUDA;
  GroupParams g = {};
  g.n = n;
  for (int i = 0; i < n; ++i) {
    if (N[i] <= 0 || N[i] % TILE_ROWS || K[i] < 4 * K2 || K[i] % K2) return SDQ_ERR_SHAPE;
    g.m[i].T2 = (int)(K[i] / K2);
    g.m[i].item0 = g.total_items;
    g.total_items += (int)(N[i] / TILE_ROWS);
  }
  *out = sdq_diag_plan_t{};
  out->kernel = SDQ_DIAG_GROUP;
  out->token_tile = M <= 16 ? 16 : 32;
  group_describe(g, sm_count, max_clusters, out, segs, cap);
  return SDQ_OK;
}

// ---------------------------------------------------------------------------------------------------------
// Allocation-free variant of sdq_linear_ws (see include/sdq.h).  The split-K scratch lives in this library's
// own device image instead of a caller buffer.
namespace sdq {
static __device__ __align__(256) unsigned char g_static_ws[SDQ_STATIC_WS_BYTES];
}

// Device address of the built-in scratch for the current device.  `g_static_ws` in host code is only a handle
// for the symbol, not an address a kernel could use, so the address is asked from the runtime, once per
// device and with that device current.
static void* static_ws_address() {
  static void* cache[64] = {nullptr};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  if (!cache[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress((void**)&ptr, sdq::g_static_ws) != cudaSuccess) return nullptr;
    cache[dev] = ptr;
  }
  return cache[dev];
}

extern "C" sdq_status_t sdq_linear_noalloc(const sdq_act_t* Xq, const sdq_packed_t* P, void* Y, int64_t ldy, void* stream)
{
  if (!Xq || !P) return SDQ_ERR_INVALID_ARG;
  size_t need = 0;
  const sdq_status_t st = sdq_workspace_size(Xq->M, P->N, P->K, &P->cfg, &need);
  if (st != SDQ_OK) return st;
  if (need == 0) return launch_linear(Xq, P, Y, ldy, nullptr, 0, stream, false);   // this shape uses no scratch
  if (need > (size_t)SDQ_STATIC_WS_BYTES) return SDQ_ERR_BUFFER_TOO_SMALL;
  void* ws = static_ws_address();
  if (!ws) return SDQ_ERR_CUDA;
  // the array keeps whatever the previous call left: the arrival counters must start at zero
  const size_t counter_bytes = ((size_t)(P->N / TILE_ROWS) * 4 + 255) & ~(size_t)255;
  if (cudaMemsetAsync(ws, 0, counter_bytes, (cudaStream_t)stream) != cudaSuccess) return SDQ_ERR_CUDA;
  return launch_linear(Xq, P, Y, ldy, ws, need, stream, false);
}
