// Local minibatch SGD step for sparse linear models whose columns are spread
// evenly (Eq. A.1, first line): the entry layout.
//
// The minibatch is stored once, cut into the column slabs of the stochastic
// reduce: per slab its entries by (worker, column, row), each a code (row,
// run flags, worker * S + column in the slab), a value and a place in its row.  The
// kernels that hold a slab do all the work that is indexed by column:
//   * the reduce of the round before (or the gather below) multiplies each
//     entry's value by w at its column and stores the product at the entry's
//     place in a row-major table, products[worker][row][place];
//   * the local step (k_row_step) only adds up each row of that table --
//     a margin -- and leaves r = d loss / d margin, one float per row;
//   * the round's reduce (or the update below) subtracts eta / B * r * value
//     at each entry's column, a column's entries added up in row order by
//     the thread that holds the first of them.
// Against the list layout (kernels_sparse.cu), which fetches w by list
// position, exchanges partial margins across a cluster and scans column sums,
// the local step of hashed logistic regression (N = 64, d = 2^20, B = 512, 100
// entries a row) went from 47 to 11.5 us and the reduce from 106 to 128 us (150
// to 132 us a round), and a minibatch takes 8 or 10 instead of 16 bytes an entry
// (250 to 140 us a round with host-resident shards, which the copy bounds).  The
// layout is for minibatches whose slabs all hold few entries and whose columns
// have short runs (kEntryRegion, kEntryRun, load_entries); skewed columns stay
// with the list layout.
#include <cuda_runtime.h>

#include <cstdint>

#include "asap_internal.h"

namespace asap {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRowLanes = 8;                             // lanes that add up one row
constexpr int kRowsAtOnce = kThreads / kRowLanes;        // rows a CTA works on at once
static_assert(kRowsAtOnce == kRowStepRows, "a CTA's share of rows is a whole number of passes");

__device__ __forceinline__ void st_release_u32(unsigned int* p, unsigned int v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

// loss(y, m) and r = d loss / d m.
template <int LOSS>
__device__ __forceinline__ void loss_and_r(float y, float m, float& l, float& r) {
  const float z = y * m;
  if (LOSS == ASAP_LOSS_HINGE) {
    l = fmaxf(0.f, 1.f - z);
    r = (z < 1.f) ? -y : 0.f;                 // strict: the corner z = 1 takes r = 0
  } else {
    // ln(1 + e^{-z}) = max(-z, 0) + ln(1 + e^{-|z|});  sigmoid(-z) = 1 / (1 + e^{z})
    l = fmaxf(-z, 0.f) + log1pf(expf(-fabsf(z)));
    r = -y / (1.f + expf(z));
  }
}

// Margins, loss and r of `rows` consecutive rows of one worker per CTA, then
// NOTIFY by the worker's last CTA.  Eight lanes add up a row, 16 bytes a load
// and four loads ahead, so that a row of 100 entries is one round trip to L2,
// where the products are: the kernel is one such trip plus its launch.  Every
// sum has a fixed order (lane by lane, then a shuffle tree; the loss over the
// CTA's warps in order), so the result does not depend on the schedule.
template <int LOSS>
__global__ void __launch_bounds__(kThreads) k_row_step(const RowStepArgs a) {
  __shared__ float red[kThreads / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, l8 = tid & (kRowLanes - 1);
  const int wq = static_cast<int>(blockIdx.x) / a.Q, q = static_cast<int>(blockIdx.x) - wq * a.Q;
  const int i = a.worker_of ? a.worker_of[wq] : wq;
  const int b_end = min((q + 1) * a.rows, a.B);
  // The stochastic reduce that follows is a programmatic dependent; this
  // grid is one of the previous round's reduce.  Labels and row lengths are
  // static batch data, read before that reduce is waited for.  A gated reduce
  // does not wait for the grids before it: one that follows a streamed update
  // of W is let in only when that grid's writes are known to be there.
  if (!a.late_trigger) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  float lsum = 0.f;
  bool waited = false;
  for (int b0 = q * a.rows; b0 < b_end; b0 += kRowsAtOnce) {
    const int b = b0 + tid / kRowLanes;
    const bool in = b < b_end;
    const int64_t row = static_cast<int64_t>(i) * a.B + b;
    const int len = in ? a.len[row] : 0;
    const float y = in ? a.y[row] : 0.f;
    if (!waited) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      waited = true;
      if (a.late_trigger) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    const float* p = a.prod + row * a.row_stride;
    float m = 0.f;
    constexpr int kU = 4, kStep = 4 * kRowLanes;
    for (int j0 = 4 * l8; j0 < len; j0 += kU * kStep) {
      float4 v[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u)
        v[u] = j0 + u * kStep < len ? __ldcg(reinterpret_cast<const float4*>(p + j0 + u * kStep))
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int n = len - (j0 + u * kStep);    // places past the row's end hold no product
        if (n > 0) m += v[u].x;
        if (n > 1) m += v[u].y;
        if (n > 2) m += v[u].z;
        if (n > 3) m += v[u].w;
      }
    }
#pragma unroll
    for (int o = kRowLanes / 2; o > 0; o >>= 1) m += __shfl_xor_sync(kFull, m, o);
    if (in && l8 == 0) {
      float l, r;
      loss_and_r<LOSS>(y, m * a.mscale, l, r);
      a.r[row] = r;
      lsum += l;
    }
  }
  if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
  for (int o = 16; o >= kRowLanes; o >>= 1) lsum += __shfl_xor_sync(kFull, lsum, o);
  if (lane == 0) red[warp] = lsum;
  __syncthreads();
  if (tid != 0) return;
  float tot = 0.f;
  for (int w = 0; w < kThreads / 32; ++w) tot += red[w];
  a.loss_part[i * a.Q + q] = tot;
  if (!a.notify) return;
  // The CTA's r are ordered before its ticket (the barrier above, then a
  // fence), the worker's tickets before its NOTIFY.
  __threadfence();
  if (atomicAdd(&a.ticket[i], 1u) == static_cast<unsigned>(a.Q) - 1u) {
    a.ticket[i] = 0u;
    __threadfence();
    if (i != a.skip_worker) st_release_u32(&a.ready[i], a.round + 1u);
  }
}

// The parameter of an entry's code in slab s.
__device__ __forceinline__ int64_t param_of(uint32_t code, long long s, int lS, int64_t ld) {
  const uint32_t off = code & kEntryOff;
  return static_cast<int64_t>(off >> lS) * ld + (s << lS) + (off & ((1u << lS) - 1u));
}

// products[worker][row][place] = value * W at the entry's column, for every
// entry of a step (parameters written by the caller, or changed by an earlier
// local step of the round).  TPS threads walk a slab, four entries each in
// flight.
template <int TPS>
__device__ __forceinline__ void slab_products(const float* W, int64_t ld, const EntryList& x, int a0, int a1,
                                              long long s, int lS, int t, float* prod, int B, int64_t stride) {
  constexpr int kU = 4;
  for (int e0 = a0 + t; e0 < a1; e0 += kU * TPS) {
    uint32_t code[kU];
    float v[kU], w[kU];
    int k[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = e0 + TPS * u;
      code[u] = e < a1 ? x.code[e] : kListPad;
      v[u] = e < a1 ? x.val[e] : 0.f;
      k[u] = e >= a1 ? 0
             : x.place ? x.place[e]
                       : static_cast<int>((code[u] >> 16) & ((1u << (x.row_shift - 16)) - 1u));
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) w[u] = code[u] != kListPad ? __ldcg(W + param_of(code[u], s, lS, ld)) : 0.f;
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (code[u] != kListPad)
        prod[(static_cast<int64_t>((code[u] & kEntryOff) >> lS) * B + (code[u] >> x.row_shift)) * stride + k[u]] =
            v[u] * w[u];
  }
}

// W -= scale * sum of r * value over a column's entries (consecutive in the
// list, in row order): the thread that holds the first of them adds them up
// and writes, so every parameter has one writer.
template <int TPS>
__device__ __forceinline__ void slab_update(float* W, int64_t ld, const EntryList& x, int a0, int a1, long long s,
                                            int lS, int t, const float* r, int B, float scale) {
  constexpr int kU = 4;
  for (int e0 = a0 + t; e0 < a1; e0 += kU * TPS) {
    uint32_t code[kU];
    float g[kU], w[kU];
    bool head[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = e0 + TPS * u;
      code[u] = e < a1 ? x.code[e] : kListPad;
      head[u] = (code[u] & kEntryNext) == 0u;
      g[u] = head[u] ? x.val[e] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (head[u]) {
        g[u] *= __ldcg(r + static_cast<int64_t>((code[u] & kEntryOff) >> lS) * B + (code[u] >> x.row_shift));
        w[u] = W[param_of(code[u], s, lS, ld)];
      }
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (head[u]) {
        const int64_t r0 = static_cast<int64_t>((code[u] & kEntryOff) >> lS) * B;
        uint32_t c = code[u];
        for (int e = e0 + TPS * u + 1; c & kEntryMore; ++e) {
          c = x.code[e];
          g[u] = fmaf(__ldcg(r + r0 + (c >> x.row_shift)), x.val[e], g[u]);
        }
        W[param_of(code[u], s, lS, ld)] = fmaf(-scale, g[u], w[u]);
      }
  }
}

template <int TPS>
__global__ void __launch_bounds__(kThreads, 4) k_entry_products(const float* W, int64_t ld, const EntryList x,
                                                             long long n_slabs, int lS, float* prod, int B,
                                                             int64_t stride) {
  const int t = threadIdx.x % TPS;
  const long long ng = static_cast<long long>(gridDim.x) * (kThreads / TPS);
  for (long long s = static_cast<long long>(blockIdx.x) * (kThreads / TPS) + threadIdx.x / TPS; s < n_slabs; s += ng)
    slab_products<TPS>(W, ld, x, x.off[s], x.off[s + 1], s, lS, t, prod, B, stride);
}

template <int TPS>
__global__ void __launch_bounds__(kThreads, 4) k_entry_update(float* W, int64_t ld, const EntryList x,
                                                           long long n_slabs, int lS, const float* r, int B,
                                                           float scale) {
  const int t = threadIdx.x % TPS;
  const long long ng = static_cast<long long>(gridDim.x) * (kThreads / TPS);
  for (long long s = static_cast<long long>(blockIdx.x) * (kThreads / TPS) + threadIdx.x / TPS; s < n_slabs; s += ng)
    slab_update<TPS>(W, ld, x, x.off[s], x.off[s + 1], s, lS, t, r, B, scale);
}

}  // namespace

cudaError_t launch_row_step(const RowStepArgs& a, int loss, int workers, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(workers * a.Q);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (loss == ASAP_LOSS_HINGE) return cudaLaunchKernelEx(&cfg, k_row_step<ASAP_LOSS_HINGE>, a);
  return cudaLaunchKernelEx(&cfg, k_row_step<ASAP_LOSS_LOGISTIC>, a);
}

cudaError_t launch_entry_products(const float* W, int64_t ld, const EntryList& x, long long n_slabs, int S,
                                  int max_region, float* prod, int B, int64_t stride, int sm_count, cudaStream_t s) {
  const int lS = __builtin_ctz(static_cast<unsigned>(S));
  if (slab_per_cta(n_slabs, max_region, sm_count))
    k_entry_products<kThreads><<<slab_grid(n_slabs, sm_count, 1), kThreads, 0, s>>>(W, ld, x, n_slabs, lS, prod, B,
                                                                                    stride);
  else
    k_entry_products<32><<<slab_grid(n_slabs, sm_count, kThreads / 32), kThreads, 0, s>>>(W, ld, x, n_slabs, lS, prod,
                                                                                          B, stride);
  return cudaGetLastError();
}

cudaError_t launch_entry_update(float* W, int64_t ld, const EntryList& x, long long n_slabs, int S, int max_region,
                                const float* r, int B, float scale, int sm_count, cudaStream_t s) {
  const int lS = __builtin_ctz(static_cast<unsigned>(S));
  if (slab_per_cta(n_slabs, max_region, sm_count))
    k_entry_update<kThreads><<<slab_grid(n_slabs, sm_count, 1), kThreads, 0, s>>>(W, ld, x, n_slabs, lS, r, B, scale);
  else
    k_entry_update<32><<<slab_grid(n_slabs, sm_count, kThreads / 32), kThreads, 0, s>>>(W, ld, x, n_slabs, lS, r, B,
                                                                                        scale);
  return cudaGetLastError();
}

}  // namespace asap
