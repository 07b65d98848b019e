/*
 * sdq_diag.h -- measurement and self-test aids of the SDQ library (no counterpart in the paper; not part of the
 * method's C-ABI in sdq.h).  Same conventions as sdq.h: plain pointers, status codes, nothing allocates.
 */
#ifndef SDQ_DIAG_H_
#define SDQ_DIAG_H_

#include "sdq.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Measurement aid: enqueues a copy-only kernel in which every SM keeps `nslot` bulk
 * copies of `slot_bytes` in flight from its own region of `src` (device, 16-byte aligned; walked cyclically) into
 * shared memory, `iters` copies per SM, nothing consuming them.  *bytes_moved receives the bytes the launch stages
 * in total; the caller times the launch with events.  With a source smaller than L2 this is the ceiling of the
 * L2 -> shared-memory path that bounds the many-token product kernel.
 *   slot_bytes a multiple of 128, >= 1024; nslot 1..16; nslot * slot_bytes <= 220 KB; src_bytes / #SMs >= slot_bytes;
 *   issuers 1..4: threads per SM that issue the copies (the slots are dealt out over them).
 *   Asynchronous on `stream`.  Errors: INVALID_ARG, ALIGNMENT, SHAPE, CUDA; a bounded wait that gives up sets the
 *   sticky device status. */
sdq_status_t sdq_diag_l2_copy(const void* src, size_t src_bytes, int slot_bytes, int nslot, int issuers, int iters,
                              size_t* bytes_moved, void* stream);


/* Self-test of the failure detection: every device-side wait of the library is bounded and reports through the sticky
 * status word (packing: through its return value) instead of hanging.  This enqueues a one-thread kernel that waits, for at most `polls` polls (1 .. 4096),
 * on a shared-memory barrier that nothing ever completes; the wait gives up, the kernel sets the status word and
 * returns.  sdq_device_status(stream) then returns SDQ_ERR_TIMEOUT once (and clears it).  Nothing traps, nothing hangs,
 * the context stays usable.  Asynchronous on `stream`.  Errors: SHAPE (polls out of range), CUDA. */
sdq_status_t sdq_diag_wait_timeout(int polls, void* stream);

/* The same of a packing call, which waits for its kernel and so reports by itself: sdq_decompose whose kernel gives its wait for the
 * rows' maxima no polls at all (K <= 16384 and a configuration that sdq_linear accepts; others have no wait).  The thread blocks give
 * up, wait for what their peers still send them, and the call returns SDQ_ERR_TIMEOUT (SDQ_ERR_NONFINITE comes first); what
 * packed_buf then holds is not to be used.  Nothing is left behind for later calls.  Errors: as sdq_decompose. */
sdq_status_t sdq_diag_decompose_timeout(const void* W, int64_t N, int64_t K, int64_t ldw, const sdq_config_t* cfg, void* packed_buf,
                                        size_t packed_bytes, sdq_packed_t* out, void* stream);

/* What a call would run, decided by the functions that decide it in the call itself; nothing is launched.
 *   sm_count > 0: for a GPU of that many SMs, of which max_clusters[k] (k = 2, 3, 4; NULL: none) clusters of 2 k thread blocks, one
 *   per SM, run at once -- host code only; sm_count == 0: for the current device (max_clusters is then ignored).
 *   sdq_diag_linear_plan: sdq_linear (workspace != 0: sdq_linear_ws with one that is large enough) of M tokens and an N x K matrix.
 *   sdq_diag_group_plan: the one launch of sdq_linear_group on n layers N[i] x K[i] in its range.
 *   tasks (may be NULL): the first `cap` of out->tasks pieces of work, in the order that thread blocks take them.  CTA pairs: row units
 *   (256 rows) row .. row + rows - 1 of 32-token groups begin .. end - 1 of the call, all of K.  Grouped kernel: row tile (128 rows)
 *   `row` of layer `layer`, its 256-K units begin .. end - 1.  The few-token kernel has none to tell.
 *   Errors: INVALID_ARG, SHAPE, UNSUPPORTED, CUDA. */
enum { SDQ_DIAG_FEW = 0, SDQ_DIAG_PAIRS = 1, SDQ_DIAG_GROUP = 2 };
typedef struct {
  int32_t kernel;      /* SDQ_DIAG_* */
  int32_t token_tile;  /* tokens of the widest tile there is room for */
  int32_t ksplit;      /* parts of the K range: of a row tile (few-token), of a task (pairs), of a left-over item (grouped) */
  int32_t cluster;     /* thread blocks per cluster (few-token with a workspace: 1) */
  int32_t ctas, tasks; /* (pairs, grouped) */
  int32_t form;        /* pairs: 0 two row units per task, 1 one, 2 one with geometry from the launch */
  int32_t alternate;   /* pairs: the accumulator alternates between two sets of columns */
  int32_t doubles, halves;   /* pairs, form 0: tasks of two units, and the tasks behind them that are halves of such */
  int32_t rounds, tail_items;   /* grouped: whole items per thread block, left-over items per cluster */
} sdq_diag_plan_t;
typedef struct { int32_t layer, row, rows, begin, end; } sdq_diag_task_t;
sdq_status_t sdq_diag_linear_plan(int64_t M, int64_t N, int64_t K, const sdq_config_t* cfg, int workspace, int sm_count,
                                  const int* max_clusters, sdq_diag_plan_t* out, sdq_diag_task_t* tasks, int64_t cap);
/* The shared-memory ring that the CTA pairs of such a call stage their operands in, by stage kind; all zero where the call runs another kernel.
 * out_slots and out_slot_bytes differ from slots and slot_bytes where the outlier stages have a geometry of their own.  Errors as above. */
typedef struct { int32_t slots, slot_bytes, out_slots, out_slot_bytes, bytes; } sdq_diag_rings_t;
sdq_status_t sdq_diag_linear_rings(int64_t M, int64_t N, int64_t K, const sdq_config_t* cfg, int sm_count, const int* max_clusters,
                                   sdq_diag_rings_t* out);
sdq_status_t sdq_diag_group_plan(int n, int64_t M, const int64_t* N, const int64_t* K, int sm_count, const int* max_clusters,
                                 sdq_diag_plan_t* out, sdq_diag_task_t* segs, int64_t cap);

#ifdef __cplusplus
}
#endif

#endif /* SDQ_DIAG_H_ */
