// Internal declarations shared by the host runtime and the kernels of the
// ASAP library.  Nothing here is part of the public ABI (include/asap.h).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "asap.h"

#ifdef __CUDACC__
#define ASAP_HD __host__ __device__
#else
#define ASAP_HD
#endif

namespace asap {

constexpr int kMaxWorkers = 1024;
constexpr int kMaxKp1Sparse = 32;     // neighbours per row for the sparse reduce
constexpr int kMetricsCap = 65536;    // rounds of metrics kept on the device
constexpr int kGraphRing = 64;        // device slots for per-round graphs: two halves of
constexpr int kGraphBatch = kGraphRing / 2;   // rounds uploaded together
constexpr int kThreads = 256;         // block size of every kernel here

// Device-side protocol and error state (one per context).
struct DevState {
  unsigned int err_code;     // first asap_status raised on the device (0 = none)
  unsigned int err_worker;
  unsigned int err_round;
  unsigned int mix_ticket;   // CTAs of the current reduce that have finished
  unsigned long long reduces;
  unsigned long long consistent_inputs;
  unsigned long long timeouts;
  unsigned long long inputs_read;        // (slab, worker) update blocks read by gated reduces
  unsigned long long inputs_current;     // ... whose worker had published NOTIFY for the round
};

// How the stochastic reduce of a sparse model meets its local step.
//   BSP        the reduce starts when the whole local-step grid has finished
//              (the kernel boundary is the barrier)
//   NOTIFY_ACK the reduce is launched while the local step runs; it streams
//              W at once and copies a slab's column sums only after the
//              NOTIFY of every worker with updates in the slab (time-limited)
//   ASYNC      measurement only: as NOTIFY_ACK but without the waits; a
//              block of updates copied before its worker's NOTIFY is stale
constexpr int kSyncBsp = 0;
constexpr int kSyncNotifyAck = 1;
constexpr int kSyncAsync = 2;

constexpr uint32_t kListPad = 0xffffffffu;   // padding entry of a column list

// Where one worker's minibatch lives inside a batch block (byte offsets from
// the block start).  The minibatch's entries are kept in one order only,
// sorted by (column, row); `cpos` indexes the batch's slab-major column list
// (one entry per distinct (worker, column) of the minibatch).  For the
// margins the sorted entries are cut into segments of kSlotSegment (one
// consumer warp's share of a tile); inside a segment every entry has a slot,
// the slots of one row contiguous (rows in order, a row's entries by
// column); the local step puts each entry's product and row at its slot.
// For the column sums the entries are split among the worker's Q CTAs at
// column boundaries (`bnd`).
struct BatchDesc {
  int64_t y;      // float [B]
  int64_t cpos;   // int32 [nnz]: list position of the entry's column
  int64_t cval;   // float [nnz]
  int64_t crow;   // uint16 [nnz]: row within the batch
  int64_t cslot;  // uint16 [nnz]: slot within its segment
  int64_t bnd;    // int32 [Q+1]: column-sum ranges of the worker's CTAs
  int32_t nnz;
  int32_t pad_;
};

// Entries per margin slot segment: a consumer warp's share of a ring stage of
// the local step (a tile of 256 entries per consumer warp).
constexpr int kSlotSegment = 256;
// Per-warp partial margins and r stay in shared memory for minibatches of
// at most this many rows (else in global scratch).
constexpr int kRSmemRows = 2048;
// Local-step threads: 4, 8 or 12 consumer warps, a bulk-copy issuer warp, and a
// gather warp (two beside twelve consumers).
constexpr int local_step_gather_warps(int warps) { return warps > 8 ? 2 : 1; }
constexpr int local_step_threads(int warps) { return 32 * (warps + 1 + local_step_gather_warps(warps)); }
constexpr int kMaxStepCluster = 8;       // CTAs per worker (portable cluster size)

// Arguments of the fused sparse local step (kernels_sparse.cu): one cluster
// of Q CTAs per worker.
struct LocalStepArgs {
  const unsigned char* block;  // batch block of this step
  const BatchDesc* desc;       // [N] descriptors of this step's batch
  const float* wv;             // w values at the step's list positions
  float* gsum;                 // column sums at the step's list positions
  float* mpart_big;            // [N][Q][4][B] per-warp partial margins (B > kRSmemRows only: four warps)
  float* r_big;                // [N][Q][B] r (B > kRSmemRows only)
  float* loss_part;            // [N]: minibatch loss sum per worker
  unsigned int* ready;         // NOTIFY flags [N]
  DevState* st;
  const int* worker_of;        // worker of each cluster (a permutation or, worker-sharded, the owned
                               // workers), or nullptr
  int N, B, Q, stages;         // N: clusters launched (workers stepped)
  unsigned int round;
  int skip_worker;             // fault injection: do not NOTIFY this worker
  float mscale;                // true w = mscale * (stored values): margins are scaled by it
  int notify;                  // publish NOTIFY (last local step of the round)
};

// The entry layout of a minibatch (kernels_entry.cu).  All workers' entries,
// by column slab of the reduce, then worker, column and row; a slab's region
// starts at a multiple of 8 entries and is padded with kListPad codes, at its
// end and before a run of one column that would cross a multiple of 32 entries.
struct EntryList {
  const uint32_t* code;        // row << row_shift | place << 16 | flags | worker * S + column in the slab
  const float* val;
  const uint16_t* place;       // place in the row's products, where the code has no room for it (row_shift 16)
  int row_shift;
  const int* off;              // [n_slabs + 1] slab regions
};

// Row and place share the code's upper 16 bits where they fit (8 bytes an
// entry instead of 10: a host-resident round of the hashed workload, 512 rows of
// 100 entries, copies 27 MB instead of 33).
constexpr uint32_t kEntryOff = 0x3fffu;       // worker * S + column (a slab holds at most 16,384 parameters)
constexpr uint32_t kEntryMore = 0x4000u;      // the next entry has the same worker and column
constexpr uint32_t kEntryNext = 0x8000u;      // so has the entry before (set in padding too)

// It is used when every slab region of every minibatch holds at most
// kEntryRegion entries and no column of a worker's minibatch more than
// kEntryRun.  A region bounds the chain of the reduce's updater warps, which
// look up an r per entry (480 entries in one pass), and takes 10 bytes an entry
// in every stage and 12 in the entry ring: up to 704 entries leave three stages
// of 32 KB slabs, two must fit.  With longer regions (allowed up to 1,300 in a
// copy; us a round, lists and entries, BSP): N = 64, d = 2^20, 660 entries on
// average 168 and 162, 800 181 and 195; N = 4, d = 3,000, 817 17.5 and 19.8; N =
// 256, d = 10^5, 921 89.9 and 92.4; but N = 32, d = 500,000, 838 73.4 and 55.7; N
// = 16, d = 10^6, 838 68.3 and 56.6: one line for all sizes lies where no size
// loses.  A run must fit the 32 entries a warp holds.  The table of products is
// rectangular, kEntryWaste bounds what padding to the longest row may cost (at
// 7.5 times, N = 32, d = 500,000, rows of 2 and 16, 36.7 us against 44.1 with lists).
constexpr int kEntryRegion = 704;
constexpr int kEntryRun = 32;
constexpr int kEntryWaste = 8;
constexpr int kHotRun = 4;               // a run from which a column counts as hot (load_entries)
constexpr int kEntryAhead = 2;           // slabs by which the reduce's entry ring runs ahead of its slabs
constexpr int kRowStepRows = 32;         // rows a local-step CTA works on at once

// Arguments of the local step on the entry layout: Q CTAs per worker, `rows`
// rows (a multiple of kRowStepRows) each.
struct RowStepArgs {
  const float* y;              // [N][B] labels
  const uint16_t* len;         // [N][B] entries of each row
  const float* prod;           // [N][B][row_stride] val * w of each entry
  int64_t row_stride;
  float* r;                    // [N][B]
  float* loss_part;            // [N][Q]
  unsigned int* ticket;        // [N] CTAs of the worker that have finished
  unsigned int* ready;
  const int* worker_of;        // as in LocalStepArgs
  int B, Q, rows;
  unsigned int round;
  int skip_worker;
  float mscale;
  int notify;
  int late_trigger;            // let the next kernel in only once the one before is complete
};

// Arguments of the stochastic reduce.
struct MixArgs {
  float* out;                  // next parameter buffer
  uint16_t* shadow;            // bf16 copy of `out` (softmax) or nullptr
  int64_t ld;                  // row stride of W (floats), multiple of 64
  int N;
  int kp1;                     // neighbours per row (sparse kind)
  const int* nbr;              // [N][kp1]
  const float* wgt;            // [N][kp1]
  float wscale;                // the round's L2 shrink prod_j (1 - eta_j l2) after local steps, else 1
  int uniform_w;               // every weight of the table equals wgt[0]
  int S;                       // slab width (columns)
  int rows_pad;                // smem rows per slab (box_rows * n_boxes)
  int box_rows;
  int n_boxes;
  int stages;
  int depth;                   // slabs in flight at most, <= stages
  long long n_slabs;
  // fused sparse update / export (FUSED kernels only)
  const uint32_t* upd_list;    // this round's column list (slab-major)
  const int* upd_off;          // [n_slabs + 1] slab regions of upd_list
  const float* gsum;           // column sums at upd_list positions
  float upd_scale;             // eta / (B wscale) of the round's last local step
  const uint32_t* exp_list;    // next round's column list
  const int* exp_off;          // [n_slabs + 1]
  float* wv_out;               // w_{t+1} at exp_list positions
  int max_region;              // entries: the largest slab region of any list
  // entry layout (kMixEntries kernels): upd / exp replace the lists above
  EntryList upd, exp;          // this round's minibatch, the next step's
  int list_slots;              // ring slots of upd's regions (0 without entries)
  const float* r;              // [N][B] r of this round's rows
  float* prod_out;             // [N][B][row_stride] products of the next step's entries
  float* step_w;               // entry step (launch_entry_step): the parameters updated in place
  int64_t row_stride;
  int B;
  // metrics and protocol
  float2* cons_part;           // scratch [gridDim.x]: float-float pairs
  const float* loss_part;      // [n_loss_part] from the local step
  int n_loss_part;
  float loss_norm;             // 1 / (N B)
  int have_loss;
  float* metrics_loss;         // ring of kMetricsCap
  float* metrics_cons;
  unsigned int* ready;
  unsigned int* consumed;
  unsigned int* stamp_next;    // [N] stamp of the buffer being written
  DevState* st;
  unsigned int round;
  int expect_notify;
  unsigned long long wait_ns;
  int sync_mode;               // kSync* (FUSED reduces; others are BSP)
  int own_lo, own_n;           // workers stepped in this context: the NOTIFY waits and the counters cover
                               // [own_lo, own_lo + own_n); a worker-sharded context learns of the others'
                               // NOTIFY on the host, when their rows are delivered
};

// Arguments of the dense softmax-regression step (kernels_dense.cu).
struct DenseFwdArgs {
  int C, Cq, d, B, nb, t;      // Cq = ceil(C / 256) CTAs per cluster
  int N;                       // workers (set by the launcher)
  const int* y;                // [N][nb*B] class ids
  uint16_t* RT;                // [N][Cq*256][B] bf16: R^T
  float* loss_part;            // [N][B/128][Cq]
  float inv_B;
  DevState* st;
  unsigned int round;
};

struct DenseGradArgs {
  int C, Cq, d, B, nb, t;
  int N;                       // workers (set by the launcher)
  float* W;                    // fp32 master [N][ld], worker row = C x d class-major
  int64_t ld;
  float lr;
  float decay;                 // 1 - lr * l2
  unsigned int* ready;
  unsigned int* worker_ticket;
  int skip_worker;
  DevState* st;
  unsigned int round;
};

asap_status build_graph_host(asap_graph_kind kind, int N, int k, uint64_t seed, int64_t round,
                             int32_t* nbr, const char** why);

// Launchers (kernels_*.cu).  Each returns the cudaError_t of the launch.
cudaError_t launch_local_step(const LocalStepArgs& a, int loss, int warps, size_t smem, cudaStream_t s);
size_t local_step_smem_bytes(int B, int stages, int warps);
cudaError_t local_step_configure(int loss, int warps);
// Clusters of Q local-step CTAs that the device holds at once (0: none).
cudaError_t local_step_clusters(int loss, int warps, int Q, size_t smem, int* clusters);
cudaError_t launch_apply_update(float* W, int64_t ld, const uint32_t* list, const int* slab_off, long long n_slabs,
                                int S, int max_region, const float* gsum, float scale, int sm_count, cudaStream_t s);
cudaError_t launch_gather_wv(const float* W, int64_t ld, const uint32_t* list, const int* slab_off, long long n_slabs,
                             int S, int max_region, float* wv, int sm_count, cudaStream_t s);
constexpr int kMixComputeWarps = 16;
constexpr int kMixUpdaterWarps = 3;
// compute warps + one TMA producer warp + the warps that apply the fused update
constexpr int kMixThreads = (kMixComputeWarps + 1 + kMixUpdaterWarps) * 32;
// What a reduce does to a slab beside mixing it: nothing; a sparse model's
// update and export through the column list; or through its entries.
constexpr int kMixPlain = 0;
constexpr int kMixLists = 1;
constexpr int kMixEntries = 2;
cudaError_t launch_mix(const CUtensorMap& tmap, const MixArgs& a, bool complete, int mode, int grid, size_t smem,
                       cudaStream_t s);
ASAP_HD size_t mix_stage_bytes(int S, int rows_pad, int max_region, int mode);
size_t mix_smem_bytes(int N, int kp1, int S, int rows_pad, int stages, int max_region, int mode, int list_slots);
cudaError_t mix_configure(bool complete, int mode, int kp1, bool shadow);
cudaError_t mix_occupancy(bool complete, int mode, int kp1, bool shadow, size_t smem, int* blocks);
// The update of a local step before a round's last, in place, and the products
// of the next step, with the slabs streamed as by the reduce (a.upd, a.exp, a.r,
// a.upd_scale, a.prod_out, a.step_w; shared memory as for a kMixEntries reduce).
cudaError_t entry_step_configure();
cudaError_t launch_entry_step(const CUtensorMap& tmap, const MixArgs& a, int grid, size_t smem, cudaStream_t s);
cudaError_t launch_row_step(const RowStepArgs& a, int loss, int workers, cudaStream_t s);
cudaError_t launch_entry_products(const float* W, int64_t ld, const EntryList& x, long long n_slabs, int S,
                                  int max_region, float* prod, int B, int64_t stride, int sm_count, cudaStream_t s);
cudaError_t launch_entry_update(float* W, int64_t ld, const EntryList& x, long long n_slabs, int S, int max_region,
                                const float* r, int B, float scale, int sm_count, cudaStream_t s);

// How the kernels that walk a step's slab regions are laid out: one CTA per
// slab while the CTAs of one wave cover all slabs (nothing is gained by
// packing slabs then) or where a region is longer than a CTA's four entries a
// thread; else one warp per slab, whose walk is a few latencies long and which
// needs an eighth of the CTAs.
inline bool slab_per_cta(long long n_slabs, int max_region, int sm_count) {
  return n_slabs <= 8LL * sm_count || max_region > 4 * kThreads;
}

// CTAs of such a kernel, at most one wave.
inline int slab_grid(long long n_slabs, int sm_count, int slabs_per_cta) {
  const long long ctas = (n_slabs + slabs_per_cta - 1) / slabs_per_cta;
  const long long cap = 8LL * sm_count;
  const long long g = ctas < cap ? ctas : cap;
  return static_cast<int>(g > 0 ? g : 1);
}
size_t dense_smem_bytes();
cudaError_t dense_configure();
cudaError_t launch_dense_fwd(const CUtensorMap& tmX, const CUtensorMap& tmW, const DenseFwdArgs& f, int N,
                             cudaStream_t s);
cudaError_t launch_dense_grad(const CUtensorMap& tmR, const CUtensorMap& tmXT, const CUtensorMap& tmWf,
                              const DenseGradArgs& g, int N, int sm_count, cudaStream_t s);
cudaError_t launch_cast_bf16(const float* src, uint16_t* dst, int64_t n, cudaStream_t s);

}  // namespace asap
