// Launch parameters of the fused GEMM kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sdq_diag.h"
#include "sdq_internal.h"
#include "sdq_layout.h"

namespace sdq {

struct LinearParams {
  const uint8_t* w;      // packed weights
  const uint8_t* x;      // quantized activations
  PackedOffsets poff;
  ActOffsets aoff;
  int64_t M, N, K;
  int out_n;
  int n_tile;            // few tokens: 16, 32, 64 or 128, the one token tile; pairs: tokens of the widest tile
  int total_tiles;       // (N / 128) * ksplit
  int nslot, slot_bytes; // shared-memory ring geometry (depends on n_tile)
  int ring_bytes;        // nslot * slot_bytes (pairs: or what the outlier stages' own slots take, if more); the transpose buffer and the barriers follow
  int release;           // 1: ring slots are reused (producer waits on `empty`, MMA issuer commits to it)
  int tmem_cols;         // TMEM columns to allocate (128, 256 or 512)
  int meta_col;          // first TMEM column of the metadata / scale buffers
  int b32;               // 1: one inlier / activation scale per 32 K (kind::mxf4nvf4 .block16)
  // two-level scaling (E4M3 Q-Vector scale codes): the accumulator of row n and token m is in units of 2^(tw[n] + tx[m]);
  // the epilogue multiplies that factor back in.  tw == nullptr: not in use.
  const int32_t* tw;     // [N] exponents of the rows' inlier factors (packed weights)
  const int32_t* tx;     // [tokens] exponents of the tokens' 8-bit scales (quantized activations)
  int dense;             // 1: dense inliers (no Stage 1): 4 dense kind::mxf4 MMAs of 64 K per stage
  // CTA-pair kernel: a task is one token tile and one or two row units (a unit = 256 weight rows = 128 per CTA).  Token tile i
  // of pt_mtiles covers the 32-token groups [i G / pt_mtiles, (i + 1) G / pt_mtiles) of the G there are; n_tile is the widest.
  int pt_units, pt_mtiles, pt_groups;
  int pt_doubles, pt_split;       // the first tasks, of two units; of the one-unit tasks behind them, the first pt_split are halves of two-unit ones
  int pt_tasks;                   // all tasks
  int pt_ks;                      // pairs that share the K range of a task, in a cluster of 2 pt_ks CTAs (then one task per cluster)
  int pt_acc2;                    // 1: the accumulator alternates between two sets of columns (one-unit tasks only)
  int pt_dual;                    // 1: the outlier stages' ring has a geometry of its own
  int ksplit;            // CTAs sharing the K range of one row tile (1 = no split)
  int cluster_ks;        // > 1: those CTAs form a cluster and reduce through distributed shared memory
  uint32_t* ws_counter;  // split-K workspace: arrival counters [row tile], zero between calls
  float* ws_partial;     // split-K workspace: fp32 partial tiles [row tile][split][token][128 rows]
  void* Y;
  int64_t ldy;
  uint32_t* flags;
};

// Grouped few-token kernel (sdq_linear_group.cu): one persistent launch over the (matrix, 128-row tile) work items of
// up to GROUP_MAX independent linear layers.
constexpr int GROUP_MAX = 32;
struct GroupMat {
  const uint8_t* w;      // packed weights
  const uint8_t* x;      // quantized activations
  void* Y;
  int64_t ldy;
  uint64_t wi, wc, sfa_out;       // sections of w: inlier stages, compact outlier stages, outlier row-scale atoms
  uint64_t xi, xo, sfb_out;       // sections of x: 4-bit stages, 8-bit stages, token-scale atom
  uint64_t wsc, xsc;              // int8 outliers: the fp32 row scales [N] of w and token scales [M] of x
  int M, T2;             // tokens, K / 256
  int item0;             // number of the matrix's first work item (= row tiles of the matrices before it)
};
struct GroupParams {
  int n, n_tile, nslot, total_items;   // nslot: inlier ring positions
  int cluster_log2, rounds, tail_log2; // how the items are dealt out (filled in by launch_linear_group)
  int w_early;           // 1: the packed weights are complete and may be read before the previous launch of the stream has ended
  int out_n;             // outliers per S-Vector, the same for every matrix of the call (0 or 1)
  int out_i8;            // the outlier operands are int8 with fp32 scales (else E4M3 with power-of-two scale atoms)
  // activation-resident variant (launch_linear_group with x_bf16 set): all matrices share one bf16 X [x_M][K], which every
  // CTA quantizes into its own shared memory before it starts; GroupMat::x and its section offsets are then unused
  const void* x_bf16;
  int64_t x_ld;
  int x_M, scale_rule;
  uint32_t* flags;
  GroupMat m[GROUP_MAX];
};
cudaError_t launch_linear_group(GroupParams p, bool f32_out, DeviceInfo* d, cudaStream_t stream);
double group_kernel_us(int64_t items, int T2, int sm_count, const int* max_clusters);   // estimated time of a call of `items` row tiles of 256 T2 K, in us
bool group_xres_fits(int T2, int out_n);   // the activation-resident variant's shared-memory budget for K = 256 T2

// CTA-pair (tcgen05 cta_group::2) many-token kernel (sdq_linear_pair.cu).
// estimated time of a call in us, to choose between the kernels
double pair_kernel_us(int64_t M, int64_t N, int64_t K, int out_n, bool b32, bool dense, int sm_count, const int* max_clusters);
// clusters of k pairs of CTAs, one CTA per SM, that run at once on the current device: entries 2..4
const int* pair_max_clusters(DeviceInfo* d);
// what sdq_diag_linear_plan and sdq_diag_group_plan report (the parameters as for a launch, pointers unset)
void pair_describe_rings(LinearParams p, int sm_count, const int* max_clusters, sdq_diag_rings_t* out);
void pair_describe(LinearParams p, int sm_count, const int* max_clusters, sdq_diag_plan_t* out, sdq_diag_task_t* tasks, int64_t cap);
void group_describe(GroupParams p, int sm_count, const int* max_clusters, sdq_diag_plan_t* out, sdq_diag_task_t* segs, int64_t cap);
cudaError_t launch_linear_pair(LinearParams p, bool f32_out, DeviceInfo* d, cudaStream_t stream);

}  // namespace sdq
