// Fused decomposed GEMM for many tokens, CTA-pair form  Y = A_i W_i^T + A_o W_o^T   (Section 5.1: O = O_i + O_o)
//
// The two CTAs of a cluster work as one tensor-core unit (tcgen05 cta_group::2).  A task is one token tile of T tokens and
// one or two row units of 256 weight rows: CTA r stages weight rows 128 r .. 128 r + 127 of each unit and the codes of
// tokens r T/2 .. only, and the pair-wide MMA takes half of its B operand from each CTA's shared memory.  All inlier stages
// (256 K) run first, then all outlier stages (128 K), into one fp32 accumulator per unit.
//
// What bounds the layer is the bytes a task pulls from L2 into shared memory: with every SM pulling, an SM receives ~90 of
// the ~117 B/ns that the copy-only kernel reaches, since the ring (all the shared memory there is) over the loaded L2 latency
// is what can be in flight.  Per 256 K an SM stages 31 KB of weights per unit and 384 B per token of its half:
//   one unit  x 256 tokens   80 KB for 6 MMAs of 80 ns    (167 B per ns of tensor time)
//   two units x 224 tokens  105 KB for 12 MMAs of 76 ns   (116)
// so two units share every staged activation byte, which T = 224 tokens leave room for in tensor memory: 2 x 224
// accumulator columns, two alternating sets of metadata and scales (24 each) and the outlier scales (16) are 512.  Token
// tiles are cut at any multiple of 32, so that they are equally wide and nothing is multiplied for padding.
// Under a sustained load the GPU's power limit holds the clock at 1.3 to 1.45 GHz (1.97 otherwise); two-unit tasks then run
// their four MMAs of a stage in 640 cycles (the pipe needs ~600), one-unit tasks their two in 427 (300).
//
// Sustained (0.3 s of calls), one unit x 256 tokens before -> now: 2048 x 4096 -> 11008 80.2 -> 77.5 us, 8192 x 11008 -> 4096
// 278 -> 259 us, with E4M3 scales 4096 x 16384 -> 4096 265 -> 232 us, dense inliers 1500 x 11008 -> 4096 90 -> 78 us; K over
// several pairs 130 x 16384 -> 4096 27 -> 21 us, 400 x 16384 -> 1024 35 -> 17 us.  A chain of calls at burst clocks: 500 x 4096 -> 4096 21.1 ->
// 13.9 us (K over pairs 14.9, wide tiles of it too 14.3, the set-up below 13.9).
//
// Few tasks (narrow matrices, few tokens): a task is one chain of stages at ~0.16 us each however few tokens it has, so its K
// range is split over 2 to 4 pairs of a larger cluster; their fp32 partial tiles meet in shared memory and every CTA adds
// one slice of rows over the splits, in order (no global scratch, reproducible).
//
// Per CTA: warps 0 / 2 / 3 bulk-copy producers (weight records / activation codes / scale atoms; two lanes each), warps
// 4..19 epilogue in four groups (TMEM -> registers as packed bf16, TMEM handed back, transposed stores under the next
// task's K loop).  Even CTA (leader): warp 1 copies metadata and scales of both CTAs to TMEM (pair-wide tcgen05.cp) and
// issues the pair-wide MMAs; its tcgen05.commit signals "slots consumed" / "accumulator complete" to the barriers of both
// CTAs.  Odd CTA: two lanes of warp 1 forward "my part of the slot has landed" to the leader's barriers.  Every wait is
// bounded.
//
// Facts behind the form of the loops (measured on B200): a remote mbarrier arrive with .release.cluster costs ~0.8 us under
// load (the default semantics suffice: the data was written by the bulk-copy engine and is read by the tensor core, both
// outside the forwarding thread's view of memory); descriptors and TMEM addresses of tcgen05 instructions are
// uniform-register operands, so the issue loop is warp-uniform with one elected lane; a trip of a single-thread loop costs
// 0.3 us, hence two lanes per producer and runs of landed slots in the issuer; a pair-wide commit costs the pipe ~80 ns.
#include <cuda_bf16.h>
#include <mutex>
#include <type_traits>

#include "sdq_internal.h"
#include "sdq_layout.h"
#include "sdq_linear.h"
#include "sdq_ptx.cuh"

namespace sdq {

constexpr int PAIR_THREADS = 640;            // 20 warps
constexpr int PAIR_MAX_SLOTS = 12;
constexpr int PAIR_STG = 4096;               // transpose buffer: 4 groups x 4 tokens x 128 features bf16
constexpr int PAIR_BARS = 14;                // full barriers, and as many for the releases: two geometries of a ring have 14 slots at most
constexpr int PAIR_TAIL = PAIR_STG + (2 * PAIR_BARS + 4) * 8 + 16 + 128;   // + barriers + alignment slack

// Geometry of a launch.  TWO: tasks of two units (and one), FULL: of one unit with token tiles of up to 256, both with the
// ring's and tensor memory's geometry known at compile time (the issue loop pays for every runtime parameter: 474 against
// 427 cycles per stage of two 256-token MMAs); FLEX: one unit, narrower tiles or K split, geometry from the launch parameters.
enum { PAIR_TWO = 0, PAIR_FULL = 1, PAIR_FLEX = 2 };

template <bool B32, bool DENSE>
struct PairGeom {
  static constexpr bool S32 = B32 || DENSE;                       // one scale per 32 K
  static constexpr uint32_t WIB = DENSE ? 17408u : (B32 ? 11264u : 10752u);   // inlier weight record (>= the outlier record + one atom)
  static constexpr uint32_t NA = S32 ? 2u : 1u;                   // scale atoms per 128 rows / tokens and inlier stage
  // TMEM columns of one set of metadata / scales: E 2 x 4 | SFA 2 x 4 NA | SFB 8 NA; two sets alternate; then SFA_out 2 x 4 | SFB_out 8
  static constexpr uint32_t SFA = 8u, SFB = 8u + 8u * NA, SET = 8u + 16u * NA, COLS = 2u * SET + 16u;
};
__host__ __device__ constexpr int pair_tmax(int form, bool s32) { return form == PAIR_TWO ? (s32 ? 192 : 224) : 256; }
// slot = | weight record of each unit | codes of T / 2 tokens | scale atoms of the tokens, [128 tokens][K-block] |
// (first outlier stage: the units' row-scale atoms directly behind their outlier records, the token-scale atoms like SFB)
__host__ __device__ constexpr uint32_t pair_slot_bytes(uint32_t wib, bool s32, int units, int T) {
  return (uint32_t)units * wib + (uint32_t)T * 64u + (s32 ? 4u : 2u) * SF_ATOM_BYTES;
}
__host__ __device__ constexpr int pair_slots(uint32_t slot) {      // released two at a time: an even number
  const int n = (int)((232448u - PAIR_TAIL) / slot) / 2 * 2;
  return n < PAIR_MAX_SLOTS ? n : PAIR_MAX_SLOTS;
}

// Dense inliers: an inlier weight record has 17 KB, an outlier record 10, so slots that hold the former leave a third of the ring
// unused in the outlier stages, two thirds of the task, while the bytes in flight are what bounds it.  With one task per pair (DUAL) the
// outlier stages use the ring in another geometry: | outlier record, row-scale atom | x units | codes | two token-scale atoms |, six
// slots instead of four (two units x 192 tokens), eight instead of six (one unit x 256).  The first stage in such a slot waits for the
// inlier slots that had its bytes.  1500 x 11008 -> 4096, 1:8 + 6:8: 71.5 -> 61.9 us, 1500 x 4096 -> 4096 29.7 -> 26.3, 300 x 8704 -> 10880 53.7
// -> 46.3 (chains of calls, burst clocks).  With several tasks per pair the ring would have to turn back for each: 8192 x 2560 -> 2560 57 ->
// 63, long K the same (the clock is lower there and the tensor pipe the bound).  A turn costs about 1.2 us, the slots give what the task's
// length makes of them.  Two-unit tasks, of four slots that were too few, from K = 2048 on: 360 x 2048 -> 14592 19.8 -> 18.4, 329 x 2304 -> 11392 18.0
// -> 17.4; below, 1500 tokens, 1024 14.15 -> 14.02, 1280 15.2 -> 15.6.  One-unit tasks, of six that nearly did, from K = 6144 on: 692 x 6144 ->
// 4864 24.9 -> 23.9, 512 x 7168 -> 6528 30.9 -> 28.8, 498 x 7936 -> 6912 35.9 -> 35.0; below, 387 x 2048 -> 8192 12.7 -> 13.8, 423 x 3584 -> 6272
// 17.1 -> 18.2, 243 x 4864 -> 9728 22.5 -> 23.0, 604 x 5376 -> 4864 21.4 -> 21.7.
__host__ __device__ constexpr uint32_t pair_out_slot_bytes(int units, int T) {
  return (uint32_t)units * (WO_BYTES + SF_ATOM_BYTES) + (uint32_t)T * 64u + 2u * SF_ATOM_BYTES;
}
__host__ __device__ constexpr uint32_t pair_ring_bytes(uint32_t slot, int nslot, bool dual, int units, int T) {
  const uint32_t i = slot * (uint32_t)nslot, o = dual ? pair_out_slot_bytes(units, T) * (uint32_t)pair_slots(pair_out_slot_bytes(units, T)) : 0u;
  return i > o ? i : o;
}

struct PairTask { int u0, nu, mt; };
template <int FORM>
__host__ __device__ __forceinline__ PairTask pair_task(const LinearParams& p, int task) {
  PairTask t;
  if (FORM != PAIR_TWO) {
    t.mt = task / p.pt_units; t.u0 = task - t.mt * p.pt_units; t.nu = 1;
    return t;
  }
  const int rp = p.pt_units >> 1;                                 // unit pairs per token tile
  if (task < p.pt_doubles) {
    t.mt = task / rp; t.u0 = 2 * (task - t.mt * rp); t.nu = 2;
    return t;
  }
  const int s = task - p.pt_doubles;
  t.nu = 1;
  if (s < p.pt_split) {
    const int d = p.pt_doubles + (s >> 1);
    t.mt = d / rp; t.u0 = 2 * (d - t.mt * rp) + (s & 1);
  } else {
    t.mt = s - p.pt_split; t.u0 = p.pt_units - 1;                 // the odd unit of every token tile
  }
  return t;
}
// first 32-token group of token tile `mt`
__host__ __device__ __forceinline__ int pair_group0(const LinearParams& p, int mt) { return (int)((int64_t)mt * p.pt_groups / p.pt_mtiles); }

template <bool F32_OUT, bool B32, bool DENSE, int FORM, bool DUAL>
__global__ void __maxnreg__(96)
sdq_linear_pair_kernel(const __grid_constant__ LinearParams p)
{
  using G = PairGeom<B32, DENSE>;
  constexpr bool S32 = G::S32, TWO_LEVEL = B32 && !DENSE && !F32_OUT;   // (bf16 outputs of two-level scaling)
  constexpr uint32_t NA = G::NA;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t* sm = smem_raw + ((128 - (ptx::smem_u32(smem_raw) & 127)) & 127);
  constexpr uint32_t SL_B = FORM == PAIR_TWO ? 2u * G::WIB : G::WIB, FIXED_T = (uint32_t)pair_tmax(FORM, S32);
  constexpr uint32_t FIXED_SLOT = pair_slot_bytes(G::WIB, S32, FORM == PAIR_TWO ? 2 : 1, (int)FIXED_T);
  const uint32_t TMAX = FORM == PAIR_FLEX ? (uint32_t)p.n_tile : FIXED_T, SLOT = FORM == PAIR_FLEX ? (uint32_t)p.slot_bytes : FIXED_SLOT;
  const uint32_t NSLOT = FORM == PAIR_FLEX ? (uint32_t)p.nslot : (uint32_t)pair_slots(FIXED_SLOT), SL_SF = SL_B + TMAX * 64u;
  const bool acc2 = FORM == PAIR_FLEX && p.pt_acc2;
  // the ring of the outlier stages: the same one, or (DUAL) the second geometry
  static_assert(!DUAL || (DENSE && FORM != PAIR_FLEX));
  static_assert(PAIR_MAX_SLOTS <= PAIR_BARS && PAIR_BARS <= 29);   // (lanes 29 to 31 of the warp that sets the barriers up have others)
  constexpr int UNITS = FORM == PAIR_TWO ? 2 : 1;
  constexpr uint32_t O_UNIT = DUAL ? WO_BYTES + SF_ATOM_BYTES : G::WIB;     // from one unit's record to the next
  constexpr uint32_t O_FIXED = pair_out_slot_bytes(UNITS, (int)FIXED_T);
  static_assert(!DUAL || pair_slots(FIXED_SLOT) + pair_slots(O_FIXED) <= PAIR_BARS);
  const uint32_t O_SLOT = DUAL ? O_FIXED : SLOT, O_NSLOT = DUAL ? (uint32_t)pair_slots(O_FIXED) : NSLOT;
  const uint32_t O_B = DUAL ? UNITS * O_UNIT : SL_B, O_SF = O_B + TMAX * 64u;
  uint8_t* stg_base = sm + (FORM == PAIR_FLEX ? NSLOT * SLOT : pair_ring_bytes(FIXED_SLOT, pair_slots(FIXED_SLOT), DUAL, UNITS, (int)FIXED_T));
  uint64_t* full = reinterpret_cast<uint64_t*>(stg_base + PAIR_STG);   // the producers' parts of slot s have landed (leader: + the peer's)
  uint64_t* empty = full + PAIR_BARS;                              // [s / 2]: the MMAs that read slots s and s ^ 1 have completed
  uint64_t* acc_full = empty + PAIR_BARS;                          // [2]
  uint64_t* acc_empty = acc_full + 2;                              // [2] leader: all epilogue warps of the pair have drained the accumulator
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile uint32_t* timed_out = tmem_slot + 1;                    // an epilogue group's wait gave up

  uint64_t *full_o = DUAL ? full + NSLOT : full, *empty_o = DUAL ? empty + NSLOT / 2 : empty;   // of the outlier stages' ring
  const uint32_t crank = ptx::cluster_ctarank(), rank = crank & 1u, lead = crank & ~1u;   // rank 0 = leader of the pair
  const int ks = FORM == PAIR_FLEX ? p.pt_ks : 1, split = (int)(crank >> 1);   // pairs that share the K range of a task
  const int pair = (int)blockIdx.x / (2 * ks), n_pairs = (int)gridDim.x / (2 * ks);
  const uint16_t both = (uint16_t)(3u << lead);
  const int RT = (int)(p.N / TILE_ROWS);
  const int T1 = p.out_n ? (int)(p.K / K1) : 0, T2 = (int)(p.K / K2);
  const int i0 = ks == 1 ? 0 : split * T2 / ks, o0 = ks == 1 ? 0 : split * T1 / ks;       // first inlier / outlier stage of this pair
  const int NI = ks == 1 ? T2 : (split + 1) * T2 / ks - i0, S = NI + (ks == 1 ? T1 : (split + 1) * T1 / ks - o0);
  const int my_tasks = p.pt_tasks > pair ? (p.pt_tasks - pair + n_pairs - 1) / n_pairs : 0;
  const int total = my_tasks * S;                                  // stages of this CTA, numbered through its tasks

  // Set-up.  The producers need nothing but this CTA's barriers for the ring's first lap, so they start on those while tensor memory
  // is being allocated and the other CTAs of the cluster are waited for (by everybody else, before anything remote).  The fence behind
  // the barriers releases them; only warp 1's allocation has to be released besides.  Everybody behind one barrier -> so, chains of calls at
  // burst clocks: 40 x 4096 -> 4096 9.48 -> 9.15 us, 500 14.3 -> 13.9, 1000 17.06 -> 16.80, 100 x 4096 -> 11008 14.47 -> 14.24; with a quantizer in front of each
  // 11.3 -> 11.1, 18.2 -> 18.0, 21.8 -> 21.3, but 16.56 -> 16.65: 60 to 230 tokens against 43 units lose half a percent
  const bool producer = warp == 0 || warp == 2 || warp == 3;
  if (warp == 0) {
    if (lane == 0) ptx::griddep_launch_dependents();   // (first of all: behind the barriers' set-up a pass of 100 tokens took 17.82 instead of 17.72 us)
    if (lane < NSLOT + (DUAL ? O_NSLOT : 0u)) {
      ptx::mbar_init(&full[lane], rank == 0 ? 3 : 2);
      if (!(lane & 1)) ptx::mbar_init(&empty[lane >> 1], 1);
    } else if (lane >= 30) {
      ptx::mbar_init(&acc_full[lane - 30], 1);
      ptx::mbar_init(&acc_empty[lane - 30], 32);
    } else if (lane == 29) {
      *timed_out = 0u;
    }
    ptx::fence_barrier_init();
  }
  __syncwarp();
  uint32_t tmem = 0;
  if (producer) {
    if (warp == 0) ptx::named_bar_arrive(6, PAIR_THREADS - 64);
    ptx::named_bar_sync(5, 96);
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  } else {
    if (warp == 1) ptx::tmem_alloc_pair(tmem_slot, 512);
    ptx::tc_fence_before();
    ptx::named_bar_sync(6, PAIR_THREADS - 64);
    if (warp == 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    else asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // both CTAs' barriers and tensor memory exist before anything remote
    ptx::tc_fence_after();
    tmem = *tmem_slot;
  }
  const uint32_t meta = tmem + (FORM == PAIR_TWO || acc2 ? 2u * TMAX : TMAX);   // metadata and scales follow the accumulator columns

  if (producer) {
    if (lane < 2) {
      // ---------------- producers (both CTAs): role 0 = own weight records, 1 = own activation codes, 2 = scale atoms.
      // Ring slots are released in pairs, so lanes 0 and 1 of the warp run the loop in lockstep, lane l filling the slots of
      // parity l: two stages per trip.  A trip has to stay short -- with the addresses worked out from scratch and the release
      // tested at its head it took 0.3 us, and no stage could take less than half of that: what belongs to a task is worked out
      // once, and the next release is tested while this trip's copies go out.
      // The expected bytes of codes and atoms are announced by role 1, so role 2 has nothing to do for an outlier stage but
      // the first.
      bool ok = true;
      auto produce = [&](auto on_task, auto on_stage) {
        if constexpr (DUAL) {
          // n stages in N slots of SZ bytes; both lanes wait for every pair of slots, also where an odd number leaves the second one empty
          auto stages = [&](int k0, int n, uint32_t N, uint32_t SZ, uint64_t* fl, uint64_t* em, auto first_lap) {
            uint32_t s = lane;
            bool ready = false;
            for (uint32_t g = 0; (int)(2 * g) < n && ok; ++g) {
              if (g < N / 2) ok = first_lap(s >> 1);
              else if (!ready) ok = ptx::mbar_wait(&em[s >> 1], ((g / (N / 2)) & 1u) ^ 1u);
              if (!ok) break;
              if ((int)(2 * g + lane) < n) on_stage(k0 + (int)(2 * g + lane), sm + (size_t)s * SZ, &fl[s]);
              s += 2;
              if (s >= N) s -= N;
              ready = g + 1 >= N / 2 && ptx::mbar_test(&em[s >> 1], (((g + 1) / (N / 2)) & 1u) ^ 1u);
            }
            ok = __all_sync(3u, ok);       // (together again behind an odd number: lanes that run apart take twice as long a trip, 62 -> 72 us)
          };
          on_task(pair_task<FORM>(p, pair));
          stages(0, NI, NSLOT, SLOT, full, empty, [](uint32_t) { return true; });
          if (ok)
            stages(NI, S - NI, O_NSLOT, O_SLOT, full_o, empty_o, [&](uint32_t e) {
              // the pairs of inlier slots with bytes of this pair, of `used` uses in all: the last use of each
              const uint32_t used = (uint32_t)(NI + 1) / 2, y1 = min((2 * (e + 1) * O_SLOT - 1) / (2 * SLOT), NSLOT / 2 - 1);
              bool free = true;
              for (uint32_t y = e * O_SLOT / SLOT; y <= y1 && free; ++y)
                if (used > y) free = ptx::mbar_wait(&empty[y], ((used - 1 - y) / (NSLOT / 2)) & 1u);
              return free;
            });
          return;
        }
        uint32_t s = lane, wrapped = 0, ph = 0;
        int tseq = 0, k = (int)lane, cur = -1;                               // this lane's stage: task number in the CTA's sequence, stage in the task
        while (k >= S) { k -= S; ++tseq; }
        bool ready = false;
        for (int i = (int)lane; i < total; i += 2) {
          if (tseq != cur) { cur = tseq; on_task(pair_task<FORM>(p, pair + tseq * n_pairs)); }
          if (wrapped && !ready && !(ok = ptx::mbar_wait(&empty[s >> 1], ph ^ 1))) break;
          on_stage(k, sm + (size_t)s * SLOT, &full[s]);
          s += 2;
          if (s >= NSLOT) { s -= NSLOT; wrapped = 1; ph ^= 1; }
          ready = wrapped && ptx::mbar_test(&empty[s >> 1], ph ^ 1);
          k += 2;
          while (k >= S) { k -= S; ++tseq; }
        }
      };
      if (warp == 0) {
        // weight records of the one or two units
        const uint8_t *wi0 = nullptr, *wi1 = nullptr, *wo0 = nullptr, *wo1 = nullptr, *sf0 = nullptr, *sf1 = nullptr;
        uint32_t nu = 1, early = NSLOT / 4;     // pairs of slots filled before the previous kernel has ended
        produce([&](const PairTask& t) {
          nu = (uint32_t)t.nu;
          // (an odd number of row tiles: the last unit's second half repeats the last tile and is not stored)
          const int rt0 = min(2 * t.u0 + (int)rank, RT - 1), rt1 = min(2 * t.u0 + 2 + (int)rank, RT - 1);
          wi0 = p.w + p.poff.wi + ((size_t)rt0 * T2 + i0) * G::WIB;
          wo0 = p.w + p.poff.wo + ((size_t)rt0 * T1 + o0) * WO_BYTES;
          sf0 = p.w + p.poff.sfa_out + (size_t)rt0 * SF_ATOM_BYTES;
          if (FORM == PAIR_TWO) {
            wi1 = p.w + p.poff.wi + ((size_t)rt1 * T2 + i0) * G::WIB;
            wo1 = p.w + p.poff.wo + ((size_t)rt1 * T1 + o0) * WO_BYTES;
            sf1 = p.w + p.poff.sfa_out + (size_t)rt1 * SF_ATOM_BYTES;
          }
        }, [&](int k, uint8_t* st, uint64_t* bar) {
          // half a lap of weights is under way when the activations come; the other half would only stand in the way of what the previous
          // kernel, as a rule the quantizer, still has to load.  No weights / half a lap / a lap / no limit, behind a quantizer: 150 x 4096 -> 16384
          // 19.01, 18.96, 19.07, 19.15 us, 300 x 4096 -> 11008 23.8, 23.6, 24.0, 23.4, 1000 x 11008 -> 4096 53.4, 52.8, 53.3, 52.7; behind a product: 60 x
          // 4096 -> 11008 13.47, 13.48, 13.56, 13.56, 260 19.38, 19.15, 19.09, 19.05, 1000 x 4096 -> 4096 16.90, 16.80, 16.80, 16.67
          if (early-- == 0) ptx::griddep_wait();
          const bool two = FORM == PAIR_TWO && nu == 2;
          if (k < NI) {
            const uint32_t off = (uint32_t)k * G::WIB;
            ptx::mbar_expect_tx(bar, (two ? 2u : 1u) * G::WIB);
            ptx::bulk_g2s(st, wi0 + off, G::WIB, bar);
            if (two) ptx::bulk_g2s(st + G::WIB, wi1 + off, G::WIB, bar);
          } else {
            const uint32_t off = (uint32_t)(k - NI) * WO_BYTES;
            const bool first_o = k == NI;
            ptx::mbar_expect_tx(bar, (two ? 2u : 1u) * (WO_BYTES + (first_o ? SF_ATOM_BYTES : 0u)));
            ptx::bulk_g2s(st, wo0 + off, WO_BYTES, bar);
            if (two) ptx::bulk_g2s(st + O_UNIT, wo1 + off, WO_BYTES, bar);
            if (first_o) {
              ptx::bulk_g2s(st + WO_BYTES, sf0, SF_ATOM_BYTES, bar);
              if (two) ptx::bulk_g2s(st + O_UNIT + WO_BYTES, sf1, SF_ATOM_BYTES, bar);
            }
          }
        });
      } else {
        // own activation codes (role 1) and the scale atoms of both token halves (role 2)
        const bool codes = warp == 2;
        const uint8_t *xi = nullptr, *xo = nullptr, *sf = nullptr;
        uint32_t own = 0, have = 1;
        ptx::griddep_wait();                   // activations come from an earlier kernel; weights do not
        produce([&](const PairTask& t) {
          const int g0 = pair_group0(p, t.mt), T = 32 * (pair_group0(p, t.mt + 1) - g0);   // the tile's first scale atom, its tokens
          const int64_t t0 = (int64_t)g0 * 32 + rank * (T / 2);
          own = (uint32_t)max((int64_t)0, min((int64_t)(T / 2), p.aoff.Mpad - t0)) * 128u; // this CTA's code bytes that exist
          have = T > 128 && g0 + 4 < p.aoff.atoms ? 2u : 1u;
          xi = p.x + p.aoff.xi + (size_t)i0 * p.aoff.xi_stride + (codes ? (size_t)t0 * 128u : (size_t)p.aoff.Mpad * 128u + (size_t)g0 * (NA * SF_ATOM_BYTES));
          xo = p.x + p.aoff.xo + (size_t)o0 * p.aoff.xo_stride + (size_t)t0 * 128u;
          sf = p.x + p.aoff.sfb_out + (size_t)g0 * SF_ATOM_BYTES;
        }, [&](int k, uint8_t* st, uint64_t* bar) {
          const bool inl = k < NI, first_o = k == NI;
          if (codes) {
            const uint32_t bytes = own + (inl ? have * NA * SF_ATOM_BYTES : (first_o ? have * SF_ATOM_BYTES : 0u));
            if (bytes) ptx::mbar_expect_tx(bar, bytes); else ptx::mbar_arrive(bar);
            if (own) ptx::bulk_g2s(st + (inl ? SL_B : O_B), inl ? xi + (size_t)k * p.aoff.xi_stride : xo + (size_t)(k - NI) * p.aoff.xo_stride, own, bar);
          } else if (inl || first_o) {
            const uint8_t* src = inl ? xi + (size_t)k * p.aoff.xi_stride : sf;
            const uint32_t nb = inl ? NA * SF_ATOM_BYTES : SF_ATOM_BYTES;
            uint8_t* dst = st + (inl ? SL_SF : O_SF);
            ptx::bulk_g2s(dst, src, nb, bar);
            if (have == 2) ptx::bulk_g2s(dst + nb, src + 4 * nb, nb, bar);
          }
        });
      }
      if (!ok) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else if (warp == 1 && rank == 1) {
    if (lane < 2) {
      // ---------------- odd CTA: forward "my part of the slot has landed" to the leader's barrier (lane l: slots of parity l)
      bool ok = true;
      uint32_t s = lane, ph = 0;
      auto forward = [&](int n, uint64_t* fl, uint32_t N) {
        for (int i = (int)lane; i < n; i += 2) {
          if (!(ok = ptx::mbar_wait(&fl[s], ph))) break;
          ptx::mbar_arrive_remote(&fl[s], lead);
          s += 2;
          if (s >= N) { s -= N; ph ^= 1; }
        }
      };
      forward(DUAL ? NI : total, full, NSLOT);
      if (DUAL) ok = __all_sync(3u, ok);
      if (DUAL && ok) { s = lane; ph = 0; forward(S - NI, full_o, O_NSLOT); }
      if (!ok) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader): per slot the copies of metadata and scales to TMEM (both CTAs), then the
    // pair-wide MMAs of its one or two units; tcgen05.cp and tcgen05.mma of one thread execute in issue order, so nothing
    // waits in between and two alternating TMEM sets serve all slots.
    // The whole warp runs the loop and one elected lane issues.  One trip of the loop (barrier test, vote, election) costs
    // more than the tensor pipe needs for two MMAs, so a trip takes every slot that has landed: lane i tests slot s + i, one
    // ballot gives the run of ready slots, and their instructions go out back to back.  (Testing the slots behind a run
    // while the run is being issued hides that latency, but the answers are stale: 690 against 640 cycles per stage.)
    // A pair-wide commit costs the pipe a bubble of ~80 ns, hence one release per two slots.
    bool ok = true;
    const uint32_t smb = ptx::smem_u32(sm);
    uint32_t s = 0, ph = 0, par = 0;                                // ring slot, its lap parity, parity of the TMEM set
    const uint64_t d_a = ptx::smem_desc(smb, 128, 256), d_b = ptx::smem_desc(smb + SL_B, 128, 1024), d_bo = ptx::smem_desc(smb + O_B, 128, 1024);
    const uint64_t d_cp = ptx::smem_desc(smb, 0, 128), d_sf = ptx::smem_desc(smb + SL_SF, 0, 128), d_sfo = ptx::smem_desc(smb + O_SF, 0, 128);   // copies to TMEM
    constexpr uint32_t wib16 = G::WIB >> 4, atom16 = SF_ATOM_BYTES >> 4;
    const uint32_t slot16 = SLOT >> 4, o_slot16 = O_SLOT >> 4;
    constexpr uint32_t o_unit16 = O_UNIT >> 4;
    const uint32_t sfo = meta + 2u * G::SET;                        // outlier scales of the task: SFA_out 2 x 4 | SFB_out 8
    uint32_t tcount = 0;
    for (int task = pair; task < p.pt_tasks && ok; task += n_pairs, ++tcount) {
      const PairTask t = pair_task<FORM>(p, task);
      const int nu = t.nu;
      const uint32_t T = 32u * (uint32_t)(pair_group0(p, t.mt + 1) - pair_group0(p, t.mt));
      // (two-level scaling: the .block16 kind reads its scale codes as unsigned E4M3 when bit 23 is clear)
      const uint32_t id4[2] = {ptx::idesc_block_scaled(256, T, 1, true, 0, 0) ^ (p.tw ? (1u << 23) : 0u),
                               ptx::idesc_block_scaled(256, T, 1, true, 2, 2)};
      const uint32_t id8 = ptx::idesc_block_scaled(256, T, 0, true, 0, 0);
      const uint32_t idd[2] = {ptx::idesc_block_scaled(256, T, 1, false, 0, 0), ptx::idesc_block_scaled(256, T, 1, false, 2, 2)};
      const bool wide = T > 128u;
      const uint32_t ab = acc2 ? tcount & 1u : 0u, use = acc2 ? tcount >> 1 : tcount;
      const uint32_t acc0 = tmem + ab * TMAX, acc1 = acc0 + TMAX;
      // instructions of the stages k .. k + n - 1 of the task in ring slots s ..., by one elected lane
      // (`stages`: bit 0 inlier, bit 1 outlier ones; DUAL: a run is all the one or all the other, compiled for its ring)
      auto issue = [&](auto units, auto stages, int k, int n) {
        constexpr int NU = decltype(units)::value;
        constexpr bool INL = decltype(stages)::value & 1, OUTL = decltype(stages)::value & 2, outl = !INL;
        uint32_t ss = s, pp = par;
        for (int kk = k; kk < k + n; ++kk) {
          const uint64_t so = (uint64_t)(ss * (outl ? o_slot16 : slot16));
          const uint32_t mb = meta + (pp ? G::SET : 0u);
          pp ^= 1u;
          const uint32_t acc = kk ? 1u : 0u;   // the first MMA of the task overwrites the accumulator
          if (INL && (!OUTL || kk < NI)) {
            // scale words of the tokens: K-block kb, 128 tokens a at SFB + 8 kb + 4 a, staged as [128 tokens][K-block]
            ptx::tc2_cp_32x128b_warpx4(mb + G::SFB, d_sf + so);
            if constexpr (S32) ptx::tc2_cp_32x128b_warpx4(mb + G::SFB + 8, d_sf + so + atom16);
            if (wide) {
              ptx::tc2_cp_32x128b_warpx4(mb + G::SFB + 4, d_sf + so + NA * atom16);
              if constexpr (S32) ptx::tc2_cp_32x128b_warpx4(mb + G::SFB + 12, d_sf + so + 3 * atom16);
            }
#pragma unroll
            for (int u = 0; u < NU; ++u) {
              const uint64_t wo = so + (u ? wib16 : 0u);
              const uint32_t sfa = mb + G::SFA + (u ? 4u * NA : 0u), d = u ? acc1 : acc0;
              [[maybe_unused]] const uint32_t e = mb + (u ? 4u : 0u);
              constexpr uint32_t SFA_OFF = (DENSE ? 2 * A_IN_BYTES : A_IN_BYTES + E_IN_BYTES) >> 4;
              if constexpr (!DENSE) ptx::tc2_cp_128x128b(e, d_cp + wo + (A_IN_BYTES >> 4));
              ptx::tc2_cp_32x128b_warpx4(sfa, d_cp + wo + SFA_OFF);
              if constexpr (S32) ptx::tc2_cp_32x128b_warpx4(sfa + 4, d_cp + wo + SFA_OFF + atom16);
              if constexpr (DENSE) {
#pragma unroll
                for (uint32_t j = 0; j < 4; ++j)
                  ptx::mma2_mxf4(d, d_a + wo + ((4096 * j) >> 4), d_b + so + ((256 * j) >> 4), idd[j & 1], sfa + 4 * (j >> 1),
                                 mb + G::SFB + 8 * (j >> 1), j ? 1u : acc);
              } else if constexpr (B32) {
                ptx::mma2_sp_nvf4(d, d_a + wo, d_b + so, id4[0], e, sfa, mb + G::SFB, acc);
                ptx::mma2_sp_nvf4(d, d_a + wo + (4096 >> 4), d_b + so + (512 >> 4), id4[0], e + 2, sfa + 4, mb + G::SFB + 8, 1u);
              } else {
                ptx::mma2_sp_mxf4(d, d_a + wo, d_b + so, id4[0], e, sfa, mb + G::SFB, acc);
                ptx::mma2_sp_mxf4(d, d_a + wo + (4096 >> 4), d_b + so + (512 >> 4), id4[1], e + 2, sfa, mb + G::SFB, 1u);
              }
            }
          } else {
            if (kk == NI) {
              ptx::tc2_cp_32x128b_warpx4(sfo, d_cp + so + (WO_BYTES >> 4));
              if constexpr (NU == 2) ptx::tc2_cp_32x128b_warpx4(sfo + 4, d_cp + so + o_unit16 + (WO_BYTES >> 4));
              ptx::tc2_cp_32x128b_warpx4(sfo + 8, d_sfo + so);
              if (wide) ptx::tc2_cp_32x128b_warpx4(sfo + 12, d_sfo + so + atom16);
            }
#pragma unroll
            for (int u = 0; u < NU; ++u) {
              const uint64_t wo = so + (u ? o_unit16 : 0u);
              const uint32_t e = mb + (u ? 4u : 0u), d = u ? acc1 : acc0, sfa = sfo + (u ? 4u : 0u);
              ptx::tc2_cp_128x128b(e, d_cp + wo + (A_OUT_BYTES >> 4));
              ptx::mma2_sp_mxf8(d, d_a + wo, d_bo + so, id8, e, sfa, sfo + 8, acc);
              ptx::mma2_sp_mxf8(d, d_a + wo + (4096 >> 4), d_bo + so + (512 >> 4), id8, e + 2, sfa, sfo + 8, 1u);
            }
          }
          // slots ss - 1 and ss may be refilled (both CTAs); DUAL: also the last one of an odd number of inlier stages
          if ((ss & 1) || (DUAL && kk == NI - 1)) ptx::tc2_commit_both(outl ? &empty_o[ss >> 1] : &empty[ss >> 1], both);
          if (kk == S - 1) ptx::tc2_commit_both(&acc_full[ab], both);  // the task's accumulator is complete (both CTAs)
          if (++ss == (outl ? O_NSLOT : NSLOT)) ss = 0;
        }
      };
      int k = 0;
      while (k < S) {
        // lane i: has slot s + i (the i-th next stage of this task) landed in both CTAs?
        const bool outl = DUAL && k >= NI;
        uint64_t* cf = outl ? full_o : full;
        const uint32_t N = outl ? O_NSLOT : NSLOT, idx = s + lane, sl = idx >= N ? idx - N : idx;
        const bool r = (int)lane < min(4, (DUAL && !outl ? NI : S) - k) && ptx::mbar_test(&cf[sl], idx >= N ? ph ^ 1 : ph);
        const int n = __ffs(~__ballot_sync(0xffffffffu, r)) - 1;    // length of the run of ready slots
        if (n == 0) {   // nothing yet: wait for the next slot, then look again (its neighbours tend to land with it)
          ok = __all_sync(0xffffffffu, ptx::mbar_wait(&cf[s], ph));
          if (!ok) break;
          continue;
        }
        if (k == 0 && use > 0) {   // the epilogues of both CTAs must have drained this accumulator's previous task
          ok = __all_sync(0xffffffffu, ptx::mbar_wait(&acc_empty[ab], (use - 1) & 1));
          if (!ok) break;
        }
        ptx::tc_fence_after();
        if (ptx::elect_one()) {
          auto run = [&](auto units) {
            if constexpr (!DUAL) issue(units, std::integral_constant<int, 3>{}, k, n);
            else if (!outl) issue(units, std::integral_constant<int, 1>{}, k, n);
            else issue(units, std::integral_constant<int, 2>{}, k, n);
          };
          if (FORM == PAIR_TWO && nu == 2) run(std::integral_constant<int, FORM == PAIR_TWO ? 2 : 1>{});
          else run(std::integral_constant<int, 1>{});
        }
        __syncwarp();
        k += n;
        par ^= (uint32_t)n & 1u;
        s += (uint32_t)n;
        if (s >= N) { s -= N; ph ^= 1; }
        if (DUAL && k == NI) s = ph = 0;
      }
    }
    // (a kernel whose stage count is odd leaves its last slot unreleased: nobody waits for it)
    if (!ok && lane == 0) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
  } else {
    // ---------------- epilogue (both CTAs): warp w owns TMEM lanes 32 (w % 4) .. + 31 (own weight rows).  Two units: groups 0
    // and 1 take the two halves of unit 0's tokens, groups 2 and 3 unit 1's; one unit: a quarter of the tokens each.
    const uint32_t q = warp & 3, grp = (warp - 4) >> 2, et = tid & 127u;
    uint32_t tcount = 0;
    bool ok = true;
    ptx::griddep_wait();                            // Y may still be in use by the previous kernel
    for (int task = pair; task < p.pt_tasks && ok; task += n_pairs, ++tcount) {
      const PairTask t = pair_task<FORM>(p, task);
      const uint32_t ab = acc2 ? tcount & 1u : 0u, use = acc2 ? tcount >> 1 : tcount;
      const int g0 = pair_group0(p, t.mt);
      const uint32_t unit = t.nu == 2 ? grp >> 1 : 0u, nc = 2u * (uint32_t)(pair_group0(p, t.mt + 1) - g0);   // 16-token chunks
      const uint32_t c_begin = t.nu == 2 ? (grp & 1u) * (nc / 2) : grp * nc / 4, c_end = t.nu == 2 ? (grp & 1u ? nc : nc / 2) : (grp + 1) * nc / 4;
      const int rt = 2 * (t.u0 + (int)unit) + (int)rank;
      const int64_t m0 = (int64_t)g0 * 32 + c_begin * 16;
      // tokens this group stores (a multiple of 16 in tensor memory, fewer at the end of the matrix; none beyond the last row tile)
      const int n_valid = rt < RT ? (int)max((int64_t)0, min((int64_t)(c_end - c_begin) * 16, p.M - m0)) : 0;
      const int64_t n0 = (int64_t)rt * TILE_ROWS;
      const int twr = p.tw && rt < RT ? __ldg(p.tw + n0 + q * 32 + lane) : 0;     // two-level scaling: this thread's row factor
      // The bf16 output is rounded first and multiplied by its power of two when it is stored, which is the rounding of the
      // multiplied value unless that falls below the normal range.  `tiny`: in this group of warps it may.  Accumulators are
      // multiples of 2^-20 (products of two codes and two subnormal E4M3 scales) and of 2^-18 times the outliers' row scale
      [[maybe_unused]] bool tiny = false;
      if constexpr (TWO_LEVEL) {
        if (p.tw && ks == 1 && n_valid) {
          int tx = 127;
          for (int i = (int)lane; i < n_valid; i += 32) tx = min(tx, __ldg(p.tx + m0 + i));
          tx = __reduce_min_sync(0xffffffffu, tx);
          const int e = T1 ? __ldg(reinterpret_cast<const int32_t*>(p.w + p.poff.osexp) + n0 + q * 32 + lane) : 0;
          tiny = max(twr + tx, -126) + min(-20, T1 ? e - twr - 18 : -20) < -126;
        }
      }
      // one thread per group polls the barrier and releases the other 127 through a hardware barrier: hundreds of threads
      // polling one mbarrier notice its completion late and slow the CTA's other barrier traffic down
      if (et == 0 && !ptx::mbar_wait(&acc_full[ab], use & 1)) *timed_out = 1u;
      if constexpr (TWO_LEVEL) tiny = ptx::named_bar_any(1 + grp, 128, tiny);
      else ptx::named_bar_sync(1 + grp, 128);
      if (*timed_out) { ok = false; break; }
      ptx::tc_fence_after();
      const uint32_t tbase = tmem + ((q * 32u) << 16) + (ab + unit) * TMAX + c_begin * 16u;   // (alternating accumulators: one unit)
      auto factor = [&](int64_t m) { return __int_as_float((min(max(twr + __ldg(p.tx + m), -126), 127) + 127) << 23); };
      auto hand_back = [&]() {      // this warp has read its part of the accumulator
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) { if (rank == 0) ptx::mbar_arrive(&acc_empty[ab]); else ptx::mbar_arrive_remote(&acc_empty[ab], lead); }
      };
      if (ks > 1) {
        // K split: this CTA's fp32 partial tile [token][128 rows] goes to shared memory, where the ring is idle by now
        float* dst = reinterpret_cast<float*>(sm) + (size_t)c_begin * 16 * TILE_ROWS + q * 32 + lane;
#pragma unroll 1
        for (int c0 = 0; c0 < n_valid; c0 += 16) {
          uint32_t v[16];
          ptx::tmem_ld_32x32b_x16(tbase + (uint32_t)c0, v);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) dst[(size_t)(c0 + j) * TILE_ROWS] = __uint_as_float(v[j]);
        }
        continue;
      }
      if (F32_OUT || tiny) {
        // fp32 output (tests), or a scaled one that is rounded after the scaling: straight from TMEM
#pragma unroll 1
        for (int c0 = 0; c0 < n_valid; c0 += 16) {
          uint32_t v[16];
          ptx::tmem_ld_32x32b_x16(tbase + (uint32_t)c0, v);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j < n_valid) {
              float f = __uint_as_float(v[j]);
              if (p.tw) f *= factor(m0 + c0 + j);
              const int64_t at = (m0 + c0 + j) * p.ldy + n0 + q * 32 + lane;
              if constexpr (F32_OUT) reinterpret_cast<float*>(p.Y)[at] = f;
              else reinterpret_cast<__nv_bfloat16*>(p.Y)[at] = __float2bfloat16_rn(f);
            }
        }
        hand_back();
      } else {
        // bf16 output: drain the accumulator into registers (one weight row x up to 112 tokens per thread as packed bf16
        // pairs), hand TMEM back, then transpose and store under the next task's K loop
        constexpr int CH = FORM == PAIR_TWO ? (int)FIXED_T / 32 : 4;   // 16-token chunks a group may have
        uint32_t pk[8 * CH];
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          if (16 * c < n_valid) {                   // uniform over the group
            uint32_t v[16];
            ptx::tmem_ld_32x32b_x16(tbase + 16u * (uint32_t)c, v);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
              pk[8 * c + j] = *reinterpret_cast<const uint32_t*>(&h);
            }
          }
        }
        hand_back();
        // transpose through shared memory, 4 tokens at a time per group: [4 tokens][128 features] bf16, then one 8-byte
        // store per thread (a warp writes one token's 256 B).  Two-level scaling: multiplying the rounded value by the power
        // of two is the rounding of the multiplied value (not `tiny`), so the factors go in here, after TMEM has been handed back.
        uint16_t* stg = reinterpret_cast<uint16_t*>(stg_base) + grp * 512u;
        __nv_bfloat16* Y = reinterpret_cast<__nv_bfloat16*>(p.Y);
#pragma unroll
        for (int c0 = 0; c0 < 16 * CH; c0 += 4) {
          if (c0 < n_valid) {                       // uniform over the group
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              uint32_t lo = pk[c0 / 2 + j] << 16, hi = pk[c0 / 2 + j] & 0xFFFF0000u;
              if (p.tw) {
                const int tk = c0 + 2 * j;
                if (tk < n_valid) lo = __float_as_uint(__uint_as_float(lo) * factor(m0 + tk));
                if (tk + 1 < n_valid) hi = __float_as_uint(__uint_as_float(hi) * factor(m0 + tk + 1));
              }
              stg[(2 * j) * 128 + q * 32 + lane] = (uint16_t)(lo >> 16);
              stg[(2 * j + 1) * 128 + q * 32 + lane] = (uint16_t)(hi >> 16);
            }
            ptx::named_bar_sync(1 + grp, 128);
            const uint32_t tok = et >> 5, seg = et & 31;
            if (c0 + (int)tok < n_valid) {
              const uint2 w = *reinterpret_cast<const uint2*>(stg + tok * 128 + seg * 4);
              *reinterpret_cast<uint2*>(Y + (m0 + c0 + tok) * p.ldy + n0 + seg * 4) = w;
            }
            ptx::named_bar_sync(1 + grp, 128);       // the buffer is rewritten by the next chunk
          }
        }
      }
    }
    if (!ok && lane == 0) atomicOr(&p.flags[FLAG_TIMEOUT], 1u);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (FORM == PAIR_FLEX && ks > 1) {
    ptx::cluster_sync();   // every split's partial tile is in shared memory
    const PairTask t = pair_task<FORM>(p, pair);
    const int g0 = pair_group0(p, t.mt), rt = 2 * t.u0 + (int)rank;
    const int64_t m0 = (int64_t)g0 * 32, n0 = (int64_t)rt * TILE_ROWS;
    const int n_valid = rt < RT ? (int)min((int64_t)32 * (pair_group0(p, t.mt + 1) - g0), p.M - m0) : 0;
    // four rows x one token per item: one 16-byte load per split, added in order.  The 32 quads of rows are dealt out over the splits
    const uint32_t q_begin = (uint32_t)(split * 32 / ks), q_per = (uint32_t)((split + 1) * 32 / ks) - q_begin, local = ptx::smem_u32(sm);
    uint32_t part[4];
#pragma unroll
    for (uint32_t sp = 0; sp < 4; ++sp) part[sp] = ptx::mapa_u32(local, sp < (uint32_t)ks ? 2 * sp + rank : crank);
    const uint32_t n_items = q_per * (uint32_t)max(n_valid, 0);
    for (uint32_t idx = tid; idx < n_items; idx += PAIR_THREADS) {
      const uint32_t tok = idx / q_per, row = (q_begin + (idx - tok * q_per)) << 2, off = (tok * TILE_ROWS + row) * 4;
      float4 v[4];
#pragma unroll
      for (uint32_t sp = 0; sp < 4; ++sp)
        v[sp] = sp < (uint32_t)ks ? ptx::ld_cluster_f32x4(part[sp] + off) : make_float4(0.f, 0.f, 0.f, 0.f);
      float4 a = v[0];
#pragma unroll
      for (uint32_t sp = 1; sp < 4; ++sp) { a.x += v[sp].x; a.y += v[sp].y; a.z += v[sp].z; a.w += v[sp].w; }   // absent splits add +0
      if (p.tw) {
        const int4 t4 = __ldg(reinterpret_cast<const int4*>(p.tw + n0 + row));
        const int tx = __ldg(p.tx + m0 + tok);
        auto f = [&](int e) { return __int_as_float((min(max(e + tx, -126), 127) + 127) << 23); };
        a.x *= f(t4.x); a.y *= f(t4.y); a.z *= f(t4.z); a.w *= f(t4.w);
      }
      if constexpr (F32_OUT) {
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.Y) + (m0 + tok) * p.ldy + n0 + row) = a;
      } else {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.Y) + (m0 + tok) * p.ldy + n0 + row) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
      }
    }
  }
  ptx::cluster_sync();     // no CTA leaves (or frees TMEM) while another may still read its shared memory
  if (warp == 1) ptx::tmem_dealloc_pair(tmem, 512);
}

template <bool F32_OUT, bool B32, bool DENSE, int FORM, bool DUAL = false>
static cudaError_t launch_form(const LinearParams& p, int pairs, cudaStream_t stream, std::atomic<uint32_t>* attr_mask)
{
  auto kern = sdq_linear_pair_kernel<F32_OUT, B32, DENSE, FORM, DUAL>;
  const uint32_t bit = 1u << (DUAL ? 18 + (F32_OUT ? 2 : 0) + FORM : ((F32_OUT ? 3 : 0) + (DENSE ? 2 : (B32 ? 1 : 0))) * 3 + FORM);
  if (!(*attr_mask & bit)) {     // once per device and instantiation
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
    if (e != cudaSuccess) return e;
    *attr_mask |= bit;
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)(2 * p.pt_ks * pairs));
  lc.blockDim = dim3(PAIR_THREADS);
  lc.dynamicSmemBytes = (size_t)p.ring_bytes + PAIR_TAIL;
  lc.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)(2 * p.pt_ks);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = 2;
  return cudaLaunchKernelEx(&lc, kern, p);
}
template <bool F32_OUT, bool B32, bool DENSE>
static cudaError_t launch_one(const LinearParams& p, int form, int pairs, cudaStream_t stream, std::atomic<uint32_t>* attr_mask)
{
  if constexpr (DENSE)
    if (p.pt_dual)
      return form == PAIR_TWO ? launch_form<F32_OUT, B32, DENSE, PAIR_TWO, true>(p, pairs, stream, attr_mask)
                              : launch_form<F32_OUT, B32, DENSE, PAIR_FULL, true>(p, pairs, stream, attr_mask);
  if (form == PAIR_TWO) return launch_form<F32_OUT, B32, DENSE, PAIR_TWO>(p, pairs, stream, attr_mask);
  if (form == PAIR_FULL) return launch_form<F32_OUT, B32, DENSE, PAIR_FULL>(p, pairs, stream, attr_mask);
  return launch_form<F32_OUT, B32, DENSE, PAIR_FLEX>(p, pairs, stream, attr_mask);
}

// How a call is cut into tasks: token tiles, one or two units per task, pairs per task (K split).
struct PairPlan { int form, T, mt, acc2, doubles, split, tasks, ks; double us; };

// The plan for `mt` token tiles with one-unit tasks, two-unit tasks or K over two pairs in tiles too wide to alternate; false if tensor
// memory does not hold it or there is none.  Times in us, fitted to measurements (4096 x 4096 to 16384 x 4096, 130 to 8192 tokens): a stage of one unit takes 0.158 (the chain of barrier test
// and issue) or 10.5 ns per KB that an SM stages (12.5 with every SM busy, 11.8 with compile-time geometry), one of two units 0.10 + 0.00188 T (the tensor pipe at the clock it keeps
// under load) or 13.5 ns per KB; a call 4.2 and 0.02 per pair it uses; a task ends with a drain of its accumulator that the next one waits for unless the accumulator alternates.
enum { PLAN_ONE, PLAN_TWO, PLAN_WIDE, PLAN_KINDS };
static bool pair_plan(int groups, int mt, int units, int T1, int T2, int kind, uint32_t wib, bool s32, bool dense, int pairs, const int* max_clusters, PairPlan* out)
{
  const bool dbl = kind == PLAN_TWO;
  PairPlan q;
  const int T = 32 * ((groups + mt - 1) / mt), cols = s32 ? (int)PairGeom<true, false>::COLS : (int)PairGeom<false, false>::COLS;
  q.T = T; q.mt = mt; q.ks = 1;
  if (T > pair_tmax(dbl ? PAIR_TWO : PAIR_FULL, s32)) return false;
  q.acc2 = !dbl && 2 * T + cols <= 512;
  if (kind == PLAN_WIDE && (q.acc2 || units * mt > max_clusters[2] || T2 < 2)) return false;
  q.form = dbl ? PAIR_TWO : (q.acc2 ? PAIR_FLEX : PAIR_FULL);
  const double avgT = 32.0 * groups / mt;
  const double kb1 = !dbl && units * mt < pairs ? 0.0105e-3 : (q.acc2 ? 0.0125e-3 : 0.0118e-3);
  const double s1i = kb1 * (wib + avgT * 64.0), s1o = kb1 * (WO_BYTES + avgT * 64.0), m2 = 0.10 + 0.00188 * avgT;
  const double c1 = T2 * (s1i > 0.158 ? s1i : 0.158) + T1 * (s1o > 0.158 ? s1o : 0.158) + (q.acc2 ? 0.3 : 1.0);
  const double s2i = 0.0135e-3 * (2 * wib + avgT * 64.0), s2o = 0.0135e-3 * (2 * WO_BYTES + avgT * 64.0);
  // dense inliers: a stage has twice the MMAs, 2.0 times as long under load, 1.7 times in a call of one round, which is over before
  // the clock falls.  (Priced like the sparse ones, calls of several rounds took two-unit tasks where one-unit tasks are faster: 4096 x
  // 4096 -> 11008 199 us against 182, 4096 x 16384 -> 4096 306 against 277; one round, 1500 x 11008 -> 4096: 77 us against 83)
  const double m2i = dense ? ((units / 2) * mt > pairs ? 2.0 : 1.7) * m2 : m2;
  const double c2 = T2 * (s2i > m2i ? s2i : m2i) + T1 * (s2o > m2 ? s2o : m2) + 1.0;
  q.doubles = q.split = 0;
  double us;
  if (!dbl) {
    q.tasks = units * mt;
    us = c1 * ((q.tasks + pairs - 1) / pairs);
    // few tasks: as many pairs to each as the clusters that fit the GPU allow (a reduction costs 1 us + 10 ns a token)
    // (tiles too wide for alternating accumulators are split over two pairs at most, 2.0: with few tokens to a CTA's stages the codes' bytes
    // count as much as the weights', and tiles of 256 tokens stage a quarter less than twice as many of 128: 500 x 4096 -> 4096 14.73 ->
    // 14.20 us, 512 x 8192 -> 4096 23.3 -> 19.3, with E4M3 scales 442 x 8704 -> 4096 25.3 -> 20.4; over three pairs 256 x 4096 -> 4096
    // would go from 12.1 to 13.7.  Adding two items of a reduction at a time was slower by 1 to 5 %)
    if (kind == PLAN_WIDE) {
      if (c1 / 2 + 2.0 >= us) return false;
      us = c1 / 2 + 2.0; q.ks = 2; q.form = PAIR_FLEX;
    }
    const double red = 1.0 + 0.01 * avgT;
    for (int k = 2; k <= 4 && q.acc2; ++k)
      if (q.tasks <= max_clusters[k] && k <= T2 && c1 / k + red < us) { us = c1 / k + red; q.ks = k; }
  } else {
    const int D = (units / 2) * mt, odd = (units & 1) * mt;
    const int full = D / pairs * pairs, left = D - full;
    // the last, partial round either as two-unit tasks or cut into one-unit tasks
    const double base = c2 * (D / pairs);
    const int over = odd > pairs - left ? odd - (pairs - left) : 0;         // one-unit tasks that do not fit beside the last two-unit ones
    const double as2 = left ? c2 + c1 * ((over + pairs - 1) / pairs) : c1 * ((odd + pairs - 1) / pairs);
    const double as1 = c1 * ((2 * left + odd + pairs - 1) / pairs);
    if (as1 < as2) { q.doubles = full; q.split = 2 * left; us = base + as1; }
    else { q.doubles = D; us = base + as2; }
    q.tasks = q.doubles + q.split + odd;
    if (!q.doubles) return false;      // nothing but one-unit tasks: the other form has the better slots for them
  }
  const int used = q.tasks * q.ks < pairs ? q.tasks * q.ks : pairs;
  q.us = us + 4.2 + 0.02 * used;
  // the packed weights come from DRAM
  const double stream = 4.2 + 0.02 * used + (double)units * 2 * (T2 * (double)wib + T1 * (double)WO_BYTES) / 5.5e6;
  if (q.us < stream) q.us = stream;
  *out = q;
  return true;
}

static PairPlan pair_best(int64_t M, int64_t N, int64_t K, int out_n, bool b32, bool dense, int sm_count, const int* max_clusters)
{
  const int units = (int)((N + 2 * TILE_ROWS - 1) / (2 * TILE_ROWS)), groups = (int)((M + 31) / 32);
  PairPlan best, wide, q;
  best.us = wide.us = -1.0;
  // from tiles of 256 tokens down to tiles of 128, or of 32 where the call is small (up to 1024 tokens)
  const int mt0 = (groups + 7) / 8, mt1 = groups <= 32 ? groups : 2 * mt0;
  for (int mt = mt0; mt <= mt1; ++mt)
    for (int kind = 0; kind < PLAN_KINDS; ++kind) {
      if (!pair_plan(groups, mt, units, out_n ? (int)(K / K1) : 0, (int)(K / K2), kind, dense ? 17408u : (b32 ? 11264u : 10752u), b32 || dense, dense, sm_count / 2,
                     max_clusters, &q)) continue;
      PairPlan& b = kind == PLAN_WIDE ? wide : best;
      if (b.us < 0 || q.us < b.us) b = q;
    }
  // Dense inliers: alternating tiles of 128 tokens and more take 0.4 to 0.9 us less than their price, and without outliers, where all of a
  // task's stages are of the kind that is priced too high, 1 to 2.  Chosen by price alone, wide tiles made 252 x 7168 -> 7808 without outliers
  // 13.5 us instead of 12.0, 236 x 11520 -> 4864 15.6 instead of 14.6, with them 1259 x 2560 -> 1024 11.8 instead of 11.3.  What they still win: 919 x 5888
  // -> 1920 19.2 -> 17.6, 211 x 9216 -> 7424 28.3 -> 22.8, against tiles of 96 tokens 450 x 4608 -> 2944 15.8 -> 15.0
  const double margin = !dense || best.form != PAIR_FLEX ? 0.0 : (!out_n ? 1.5 : (best.T > 96 ? 0.6 : 0.0));
  return wide.us >= 0 && (best.us < 0 || wide.us + margin < best.us) ? wide : best;
}

// largest grids, in clusters of 4, 6 and 8 CTAs with one CTA per SM, that run at once on the current device: [pairs per cluster]
const int* pair_max_clusters(DeviceInfo* d)
{
  static const int none[5] = {0, 0, 0, 0, 0};
  static std::mutex filling;
  if (!d->clusters_known) {
    std::lock_guard<std::mutex> lock(filling);
    auto kern = sdq_linear_pair_kernel<false, false, false, PAIR_FLEX, false>;
    for (int k = 2; k <= 4 && !d->clusters_known; ++k) {
      cudaLaunchConfig_t lc = {};
      lc.gridDim = dim3((unsigned)(2 * k));
      lc.blockDim = dim3(PAIR_THREADS);
      lc.dynamicSmemBytes = 200 * 1024;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = (unsigned)(2 * k);
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      lc.attrs = attr;
      lc.numAttrs = 1;
      // (not answered: plans without larger clusters, and the next call asks again)
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448) != cudaSuccess ||
          cudaOccupancyMaxActiveClusters(&d->pair_clusters[k], kern, &lc) != cudaSuccess) { (void)cudaGetLastError(); return none; }
    }
    d->clusters_known = 1;
  }
  return d->pair_clusters;
}

double pair_kernel_us(int64_t M, int64_t N, int64_t K, int out_n, bool b32, bool dense, int sm_count, const int* max_clusters)
{ return pair_best(M, N, K, out_n, b32, dense, sm_count, max_clusters).us; }

// do the outlier stages of a call have a ring geometry of their own (see pair_out_slot_bytes)?
static bool pair_dual(const LinearParams& p, const PairPlan& best, int pairs) {
  return p.dense && p.out_n > 0 && best.form != PAIR_FLEX && best.tasks <= pairs && p.K >= (best.form == PAIR_TWO ? 8 : 24) * K2;
}

// the plan's numbers into the launch parameters (p.M, N, K and the format are there); returns the pairs to launch
static int pair_apply(LinearParams& p, const PairPlan& best, int sm_count)
{
  const bool s32 = p.dense || p.b32;
  const int T = best.form == PAIR_FLEX ? best.T : pair_tmax(best.form, s32);
  p.n_tile = T;
  p.pt_units = (int)((p.N + 2 * TILE_ROWS - 1) / (2 * TILE_ROWS)); p.pt_mtiles = best.mt; p.pt_groups = (int)((p.M + 31) / 32);
  p.pt_doubles = best.doubles; p.pt_split = best.split; p.pt_tasks = best.tasks; p.pt_acc2 = best.acc2; p.pt_ks = best.ks;
  p.slot_bytes = (int)pair_slot_bytes(p.dense ? 17408u : (p.b32 ? 11264u : 10752u), s32, best.form == PAIR_TWO ? 2 : 1, T);
  p.nslot = pair_slots((uint32_t)p.slot_bytes);
  p.pt_dual = pair_dual(p, best, sm_count / 2);
  p.ring_bytes = (int)pair_ring_bytes((uint32_t)p.slot_bytes, p.nslot, p.pt_dual != 0, best.form == PAIR_TWO ? 2 : 1, T);
  return p.pt_tasks < sm_count / 2 || best.ks > 1 ? p.pt_tasks : sm_count / 2;
}

void pair_describe(LinearParams p, int sm_count, const int* max_clusters, sdq_diag_plan_t* out, sdq_diag_task_t* tasks, int64_t cap)
{
  const PairPlan best = pair_best(p.M, p.N, p.K, p.out_n, p.b32 != 0, p.dense != 0, sm_count, max_clusters);
  out->ctas = 2 * best.ks * pair_apply(p, best, sm_count);
  out->form = best.form; out->cluster = 2 * best.ks; out->ksplit = best.ks; out->tasks = best.tasks; out->doubles = best.doubles; out->halves = best.split;
  out->alternate = best.acc2; out->token_tile = p.n_tile;
  for (int64_t i = 0; tasks && i < best.tasks && i < cap; ++i) {
    const PairTask t = best.form == PAIR_TWO ? pair_task<PAIR_TWO>(p, (int)i) : pair_task<PAIR_FLEX>(p, (int)i);
    tasks[i] = {0, t.u0, t.nu, pair_group0(p, t.mt), pair_group0(p, t.mt + 1)};
  }
}

void pair_describe_rings(LinearParams p, int sm_count, const int* max_clusters, sdq_diag_rings_t* out)
{
  const PairPlan best = pair_best(p.M, p.N, p.K, p.out_n, p.b32 != 0, p.dense != 0, sm_count, max_clusters);
  (void)pair_apply(p, best, sm_count);
  const uint32_t o = pair_out_slot_bytes(best.form == PAIR_TWO ? 2 : 1, p.n_tile);
  out->slots = p.nslot; out->slot_bytes = p.slot_bytes;
  out->out_slots = p.pt_dual ? pair_slots(o) : p.nslot; out->out_slot_bytes = p.pt_dual ? (int)o : p.slot_bytes;
  out->bytes = p.ring_bytes;
}

cudaError_t launch_linear_pair(LinearParams p, bool f32_out, DeviceInfo* d, cudaStream_t stream)
{
  const PairPlan best = pair_best(p.M, p.N, p.K, p.out_n, p.b32 != 0, p.dense != 0, d->sm_count, pair_max_clusters(d));
  const int pairs = pair_apply(p, best, d->sm_count);
  std::atomic<uint32_t>* attr_mask = &d->pair_attr;
  const int v = (f32_out ? 4 : 0) | (p.dense ? 2 : (p.b32 ? 1 : 0));
  switch (v) {
    case 0: return launch_one<false, false, false>(p, best.form, pairs, stream, attr_mask);
    case 1: return launch_one<false, true, false>(p, best.form, pairs, stream, attr_mask);
    case 2: return launch_one<false, false, true>(p, best.form, pairs, stream, attr_mask);
    case 4: return launch_one<true, false, false>(p, best.form, pairs, stream, attr_mask);
    case 5: return launch_one<true, true, false>(p, best.form, pairs, stream, attr_mask);
    default: return launch_one<true, false, true>(p, best.form, pairs, stream, attr_mask);
  }
}

}  // namespace sdq
