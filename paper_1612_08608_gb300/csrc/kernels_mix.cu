// Stochastic reduce (Eq. A.1, second line; Section 3):
//   W_next[i, :] = sum_{m < k+1} wgt[i, m] * W_half[nbr[i, m], :]
// plus, fused, the round's metrics (consensus error ||W_next - 1 wbar^T||_F
// and the mean minibatch loss) and the NOTIFY-ACK bookkeeping of Section 4.
//
// Data movement.  W is [N][ld] fp32 (ld a multiple of 64).  The kernel is
// persistent: CTA b walks column slabs b, b + grid, ...  A slab is S columns
// (8 to 1024, about 32 KB) of *all* N rows.  One producer warp brings slabs into a ring of
// shared-memory stages with TMA 2-D tiled loads (one box per 256 rows), so
// every element of W is read from HBM exactly once however many neighbours
// use it; sixteen compute warps mix and write the outputs straight from
// registers.  A stage goes back to the producer when all the compute warps
// have arrived on its "empty" mbarrier: no CTA-wide barrier in steady state.
//
// Sparse models (FUSED): the local step left, per distinct (worker, column)
// of the minibatch, the column sum g of r_b x_b (kernels_sparse.cu).  The
// producer also copies the slab's part of that list (and of the next
// round's list) into the stage; once a slab has landed the updater warps
// apply the round's last local update to it, w -= eta / (B s) g, and release
// it to the compute warps through a "ready" mbarrier -- so w_{t+1/2} exists
// only in shared memory.  s is the round's L2 shrink, prod_j (1 - eta_j l2)
// over its local steps, which also scales the mixing weights (true w =
// s * stored w).  After mixing the compute warps export w_{t+1} at the next
// round's columns, which is all the next margin kernel reads.  On the entry
// layout (kMixEntries, kernels_entry.cu) the updaters form each column's sum
// of r * value themselves (update_entries), and the export is value * w_{t+1}
// of every entry of the next step.
//
// Consensus error per column: with K the column's value in row 0 (a shift
// against cancellation), sum_i (w_i - wbar)^2 = sum_i (w_i - K)^2 -
// (sum_i (w_i - K))^2 / N.  Squares accumulate per thread in fp32 (a few
// dozen slabs per thread; GB300's fp64 pipe is narrow), the per-column sums
// are combined across warps by the producer warp when the stage comes back,
// and the block and launch totals are formed in float-float pairs (fp32 hi +
// lo, a fixed order).  The complete graph (all-reduce, equal weights) writes
// the column mean to every row and adds nothing.
//
// Protocol (Section 4, NOTIFY-ACK): before it writes anything each CTA waits,
// with a time limit, until ready[j] == round+1 for every worker j and
// consumed[j] >= round (a gated reduce: before it reads).  The last CTA to
// finish (ticket) reduces the metric partials in a fixed order and ACKs:
// consumed[j] = round+1, stamp_next[j] = round+1.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "asap_internal.h"

namespace asap {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned long long kTmaWaitNs = 2000000000ull;   // 2 s: a TMA load never takes this long
// The compute warps work in groups, on alternate slabs.  A slab costs a warp a
// chain of shared-memory accesses, a few hundred cycles each: one group of
// sixteen warps goes through every slab's chain in step, the pipe idle at its
// ends.  Two groups overlap two chains, and with half the threads a thread
// has twice the rows, hence loads, in flight (N = 256, d = 10^6, k = 4: 414 ->
// 363 us a reduce).  On the entry layout, where the stages' turnaround is the
// bound, the shorter life of a slab in one group is worth more (hashed workload,
// N = 64, d = 2^20, k = 4: 127 us against 160 with two groups; no other shape
// was tried).  The number of stages is a multiple of the groups, so that a stage
// always belongs to the same group (its warps wait for every phase of the
// stage's barriers, which parities need).
constexpr int mix_groups(int mode) { return mode == kMixEntries ? 1 : 2; }
// Threads of a group: at least the 256 column quads of the widest slab.
constexpr int mix_group_threads(int mode) { return kMixComputeWarps * 32 / mix_groups(mode); }
constexpr int kProducerWarp = kMixComputeWarps;
constexpr int kUpdater0 = kMixComputeWarps + 1;             // first updater warp

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release_u32(unsigned int* p, unsigned int v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

// 4-byte asynchronous copy global -> shared.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src))
               : "memory");
}

__device__ __forceinline__ int ld_acquire_cta(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}

__device__ __forceinline__ void st_release_cta(int* p, int v) {
  asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" :: "r"(smem_u32(p)), "r"(v) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// Adds to the bytes the current phase waits for, without an arrival.
__device__ __forceinline__ void mbar_expect_only(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}

// Bounded wait on an mbarrier phase; false if the limit ran out.  The timer
// is read every 256 polls only (each try_wait already suspends the thread
// for a while), so waiting warps take few issue slots.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (unsigned n = 1;; ++n) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((n & 255u) == 0 && globaltimer_ns() - t0 > kTmaWaitNs) return false;
  }
}

// L2 policy for the parameter stream: each element is read once and written
// once per round, so it should not push the round's small lists out of L2.
__device__ __forceinline__ uint64_t evict_first_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y,
                                            uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;"
      :: "r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// The next round's w values (a few MB) should stay in L2 for the margin
// kernel's gathers.
__device__ __forceinline__ uint64_t evict_last_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ void st_f32_hint(float* p, float v, uint64_t policy) {
  asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" :: "l"(p), "f"(v), "l"(policy) : "memory");
}

__device__ __forceinline__ void st_f4_hint(float* p, float4 v, uint64_t policy) {
  asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;"
               :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "l"(policy) : "memory");
}

// Untiled bulk copy global -> shared (16-byte aligned, size a multiple of 16).
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               :: "r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void record_error(DevState* st, unsigned code, unsigned worker, unsigned round) {
  if (atomicCAS(&st->err_code, 0u, code) == 0u) {
    st->err_worker = worker;
    st->err_round = round;
  }
}

// Wait until *flag >= target (time-limited).  Returns 0 on success,
// ASAP_ERR_TIMEOUT if the limit ran out, ASAP_ERR_STATE if exact and the
// flag went past target.
__device__ unsigned wait_flag(const unsigned int* flag, unsigned target, bool exact, unsigned long long limit_ns) {
  unsigned v = ld_acquire_u32(flag);
  if (v < target) {
    const unsigned long long t0 = globaltimer_ns();
    do {
      __nanosleep(128);
      v = ld_acquire_u32(flag);
      if (v < target && globaltimer_ns() - t0 > limit_ns) return ASAP_ERR_TIMEOUT;
    } while (v < target);
  }
  return (exact && v != target) ? ASAP_ERR_STATE : 0u;
}

__device__ __forceinline__ float4 f4_fma(float w, float4 x, float4 acc) {
  acc.x = fmaf(w, x.x, acc.x);
  acc.y = fmaf(w, x.y, acc.y);
  acc.z = fmaf(w, x.z, acc.z);
  acc.w = fmaf(w, x.w, acc.w);
  return acc;
}

__device__ __forceinline__ float4 f4_add(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// A float-float value hi + lo (|lo| at most half an ulp of hi): the block
// sums are carried in fp32 pairs, since this GPU's fp64 pipe is narrow (an
// fp64 tree over the block took ~2 us, in the last CTA's finalisation ~7).
struct F2 {
  float hi, lo;
};

// hi + lo of a + b: the rounding error of hi_a + hi_b is recovered exactly
// by Knuth's two-sum, the low parts are added to it, and the pair is
// renormalised.  The result does not depend on the order of a and b.
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  const float s = a.hi + b.hi;
  const float bv = s - a.hi;
  const float e = ((a.hi - (s - bv)) + (b.hi - bv)) + (a.lo + b.lo);
  const float hi = s + e;
  return F2{hi, e - (hi - s)};
}

__device__ __forceinline__ F2 warp_sum_f2(F2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = f2_add(v, F2{__shfl_xor_sync(kFull, v.hi, o), __shfl_xor_sync(kFull, v.lo, o)});
  return v;
}

// Sum over all threads of the block (kMixThreads) in a fixed order, a warp
// tree over the lanes and one over the warps; valid in thread 0.
__device__ __forceinline__ F2 block_sum_f2(F2 v, F2* scratch) {
  constexpr int kW = kMixThreads / 32;
  static_assert(kW <= 32, "one lane per warp");
  v = warp_sum_f2(v);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) scratch[warp] = v;
  __syncthreads();
  return warp == 0 ? warp_sum_f2(lane < kW ? scratch[lane] : F2{0.f, 0.f}) : F2{0.f, 0.f};
}

// Two block sums at once, each in the order block_sum_f2 takes; valid in
// thread 0.  `scratch` holds two pairs per warp.
__device__ __forceinline__ void block_sum2_f2(F2& u, F2& v, F2* scratch) {
  constexpr int kW = kMixThreads / 32;
  u = warp_sum_f2(u);
  v = warp_sum_f2(v);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) {
    scratch[warp] = u;
    scratch[kW + warp] = v;
  }
  __syncthreads();
  if (warp == 0) {
    u = warp_sum_f2(lane < kW ? scratch[lane] : F2{0.f, 0.f});
    v = warp_sum_f2(lane < kW ? scratch[kW + lane] : F2{0.f, 0.f});
  }
}

// Barrier of all warps but the producer's, and at its own time the
// producer's, that also returns the OR of `v` over them.
__device__ __forceinline__ bool start_bar_or(bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 4, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r) : "r"(static_cast<uint32_t>(v)), "n"(kMixThreads) : "memory");
  return r != 0;
}

// Barrier of a compute group.
template <int THREADS>
__device__ __forceinline__ void compute_bar(int group) {
  asm volatile("bar.sync %0, %1;" :: "r"(group + 1), "n"(THREADS) : "memory");
}

// Barrier of a compute group that also returns the OR of `v` over it.
template <int THREADS>
__device__ __forceinline__ bool compute_bar_or(int group, bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, %3, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r) : "r"(static_cast<uint32_t>(v)), "n"(THREADS), "r"(group + 1) : "memory");
  return r != 0;
}

struct MixSmem {
  unsigned char* stage0;
  size_t stage_bytes;
  uint64_t* full;
  uint64_t* empty;
  uint64_t* ready;   // FUSED: the producer has applied the slab's update
  float4* part;      // [stages][kCompute]: per-thread column sums (consensus / complete-graph mean)
  int* info;         // [stages][4]: n_upd, n_exp, exp_base
  // entry layout: ring of a.list_slots slots of code, value and r [max_region]
  unsigned char* lists;
  size_t list_bytes;
  uint64_t* lfull;
  int* linfo;        // [list_slots]: entries of the slab
  int* nbr;
  float* wgt;
  F2* scratch;       // two pairs per warp
  int* flags;        // [0]: fail, [1]: last, [2]: failed CTAs of the launch (last CTA), [3]: slabs whose workers'
                     // NOTIFY the producer has seen (gated reduces on the entry layout)
  unsigned* seen;    // [32]: bitmap of workers whose NOTIFY this CTA has seen (gated reduces)
};

// Shared-memory layout; every region starts 16-byte aligned (the slab
// stages 1024-byte aligned).  mix_smem_bytes() mirrors it.
// Regions are formed from `raw` by pointer arithmetic (offsets only), so that
// the compiler keeps the pointers in the shared address space and emits
// plain shared-memory accesses.
__device__ __forceinline__ MixSmem carve(unsigned char* raw, const MixArgs& a, int kp1, int mode) {
  MixSmem m;
  auto a16 = [](size_t v) { return (v + 15) & ~static_cast<size_t>(15); };
  size_t off = (1024u - (smem_u32(raw) & 1023u)) & 1023u;   // 1024-byte aligned stages
  m.stage_bytes = mix_stage_bytes(a.S, a.rows_pad, a.max_region, mode);
  m.stage0 = raw + off;
  off += m.stage_bytes * a.stages;
  m.lists = raw + off;
  m.list_bytes = 12 * static_cast<size_t>(a.max_region);
  off = (off + m.list_bytes * a.list_slots + 15) & ~static_cast<size_t>(15);
  m.full = reinterpret_cast<uint64_t*>(raw + off);
  off += 8 * a.stages;
  m.empty = reinterpret_cast<uint64_t*>(raw + off);
  off += 8 * a.stages;
  m.ready = reinterpret_cast<uint64_t*>(raw + off);
  off += 8 * a.stages;
  m.lfull = reinterpret_cast<uint64_t*>(raw + off);
  off += 8 * a.list_slots;
  m.linfo = reinterpret_cast<int*>(raw + off);
  off = a16(off + 4 * a.list_slots);
  m.scratch = reinterpret_cast<F2*>(raw + off);
  off = a16(off + 16 * (kMixThreads / 32));
  m.flags = reinterpret_cast<int*>(raw + off);
  off = a16(off + 16);
  m.seen = reinterpret_cast<unsigned*>(raw + off);
  off = a16(off + 4 * 32);
  m.info = reinterpret_cast<int*>(raw + off);
  off = a16(off + 16 * a.stages);
  m.part = reinterpret_cast<float4*>(raw + off);
  off = a16(off + 16 * static_cast<size_t>(a.stages) * mix_group_threads(mode));
  m.nbr = reinterpret_cast<int*>(raw + off);
  off = a16(off + 4 * static_cast<size_t>(a.N) * kp1);
  m.wgt = reinterpret_cast<float*>(raw + off);
  return m;
}

// The updater warps' walk on the entry layout: once a slab has landed, w -=
// upd_scale * sum of r * value at every column of this round's entries.  Its
// pace is a chain of shared-memory accesses, a few hundred cycles each while
// the compute warps keep that pipe two thirds busy, so the chain is kept short:
// the entries run ahead of the slabs in a ring of their own; a thread keeps
// its entries' codes in registers and fetches the r they name (4-byte
// cp.async from L2) kAhead slabs early; a landed slab costs it one round of
// loads (w, value, r) and one of stores.  A column's entries lie in one
// 32-entry group, so its run is added up by shuffles, in row order, into the
// lane of its first entry, the column's only writer.  Hashed workload (N =
// 64, d = 2^20, ~400 entries a slab, 1.6 us a slab streamed): codes and r looked
// up in the landed slab 167 us a reduce; r early, runs read in a loop 144; so,
// 140 us then, 128 us now that the producer issues a slab before it adds up the
// last one's column sums.  In a gated reduce r is read only after the NOTIFY of
// its worker: early for slabs the producer has passed, and for all once it has
// seen every worker (sm.flags[3]), else in the landed slab.
// STORE: each updated value also goes to the stored parameters (a.step_w).
template <bool STORE>
__device__ __forceinline__ void update_entries(const MixSmem& sm, const MixArgs& a, int n_slabs, bool gated, int lS,
                                               int lqb, int box_col, bool& failed) {
  constexpr int kUpd = kMixUpdaterWarps * 32, kU = 5, kAhead = 2;
  const int ut = threadIdx.x - kUpdater0 * 32, lane = threadIdx.x & 31;
  const int S = 1 << lS, QB = 1 << lqb;
  auto r_at = [&](uint32_t c) {
    return a.r + static_cast<int64_t>((c & kEntryOff) >> lS) * a.B + (c >> a.upd.row_shift);
  };
  int fsl = 0, sl = 0, st = 0;         // ring positions: entries being fetched, entries and stage being used
  uint32_t fph = 0, ph = 0;            // and phases
  uint32_t early = 0;                  // bit d: r of the slab d ahead is on its way
  uint32_t code[kAhead + 1][kU];       // this thread's first kU entries of the slab d ahead
  // Entries of slab it into code[d], their r on the way; false if they never came.
  auto fetch = [&](int it, int d) {
    uint32_t (&c)[kU] = code[d];
#pragma unroll
    for (int u = 0; u < kU; ++u) c[u] = kListPad;
    if (it >= n_slabs) return true;
    if (!__all_sync(kFull, mbar_wait_bounded(sm.lfull + fsl, fph))) return false;
    const uint32_t* list = reinterpret_cast<const uint32_t*>(sm.lists + fsl * sm.list_bytes);
    float* r = reinterpret_cast<float*>(sm.lists + fsl * sm.list_bytes) + 2 * a.max_region;
    const int n = sm.linfo[fsl];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (ut + u * kUpd < n) c[u] = list[ut + u * kUpd];
    if (!gated || __all_sync(kFull, ld_acquire_cta(sm.flags + 3) > it)) {
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (c[u] != kListPad) cp_async4(r + ut + u * kUpd, r_at(c[u]));
      for (int e = ut + kU * kUpd; e < n; e += kUpd)
        if (list[e] != kListPad) cp_async4(r + e, r_at(list[e]));
      early |= 1u << d;
    }
    if (++fsl == a.list_slots) {
      fsl = 0;
      fph ^= 1u;
    }
    return true;
  };
  bool ok = true;
#pragma unroll
  for (int d = 0; d < kAhead; ++d) {
    ok = ok && fetch(d, d);
    asm volatile("cp.async.commit_group;" ::: "memory");   // one group per slab, empty ones included
  }
  for (int it = 0; it < n_slabs && ok; ++it) {
    ok = __all_sync(kFull, mbar_wait_bounded(sm.full + st, ph));
    if (!ok) break;
    asm volatile("cp.async.wait_group %0;" :: "n"(kAhead - 1) : "memory");   // all but the slabs after this one
    float* x = reinterpret_cast<float*>(sm.stage0 + st * sm.stage_bytes);
    const uint32_t* list = reinterpret_cast<const uint32_t*>(sm.lists + sl * sm.list_bytes);
    const float* val = reinterpret_cast<const float*>(list) + a.max_region;
    const float* r = val + a.max_region;
    const bool have_r = early & 1u;
    const int n = sm.linfo[sl];
    for (int e0 = ut; e0 - lane < n; e0 += kU * kUpd) {    // one turn unless the region is longer than kU * kUpd
      uint32_t c[kU];
      float g[kU], w[kU];
      int off[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int e = e0 + u * kUpd;
        c[u] = e0 == ut ? code[0][u] : e < n ? list[e] : kListPad;
        const int i = static_cast<int>((c[u] & kEntryOff) >> lS), cl = static_cast<int>(c[u]) & (S - 1), q = cl >> 2;
        off[u] = 4 * ((i << lqb) + (q >> lqb) * box_col + (q & (QB - 1))) + (cl & 3);
        g[u] = 0.f;
        w[u] = 0.f;
        if (c[u] != kListPad) g[u] = (have_r ? r[e] : __ldcg(r_at(c[u]))) * val[e];
        if ((c[u] & kEntryNext) == 0u) w[u] = x[off[u]];
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        // add the run's later products: step d brings that of the entry d on
        // while the run (kEntryMore up to there) reaches it
        float sum = g[u];
        uint32_t more = c[u] == kListPad ? 0u : c[u] & kEntryMore;
        for (int d = 1; __any_sync(kFull, more != 0u); ++d) {
          const float gd = __shfl_down_sync(kFull, g[u], d);
          const uint32_t cd = __shfl_down_sync(kFull, c[u], d);
          if (more) {
            sum += gd;
            more = cd & kEntryMore;
          }
        }
        if ((c[u] & kEntryNext) == 0u) {
          const float v = fmaf(-a.upd_scale, sum, w[u]);
          x[off[u]] = v;
          if (STORE) {
            const long long slab = blockIdx.x + static_cast<long long>(it) * gridDim.x;
            const uint32_t o = c[u] & kEntryOff;
            a.step_w[static_cast<int64_t>(o >> lS) * a.ld + (slab << lS) + (o & (S - 1))] = v;
          }
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before this stage's next TMA
    __syncwarp();
    if (lane == 0) mbar_arrive(sm.ready + st);
    if (++sl == a.list_slots) sl = 0;
    if (++st == a.stages) {
      st = 0;
      ph ^= 1u;
    }
    ok = fetch(it + kAhead, kAhead);
    asm volatile("cp.async.commit_group;" ::: "memory");
    early >>= 1;
#pragma unroll
    for (int d = 0; d < kAhead; ++d)
#pragma unroll
      for (int u = 0; u < kU; ++u) code[d][u] = code[d + 1][u];
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (!ok) {
    if (lane == 0) record_error(a.st, ASAP_ERR_CUDA, 0xfffffffdu, a.round);
    failed = true;
  }
}

// KP1 > 0: sparse graph with KP1 neighbours per row (compile-time);
// KP1 == 0: sparse graph, runtime a.kp1 (<= kMaxKp1Sparse);
// KP1 == -1: complete graph with equal weights;
// KP1 == kStepOnly (entry layout): no mixing, but the update of a local step
// before a round's last, stored in place, and the next step's products.  The
// slabs are streamed whole: touched one by one (kernels_entry.cu), a third of a
// hashed slab's 32-byte sectors cost a 64-byte DRAM access each, twice (N = 64,
// d = 2^20, ~400 entries a slab: update 75.5 us, products 57.3; so, both 105.8
// us).  Where entries are few it is the other way round (load_entries).
constexpr int kStepOnly = -2;

template <int KP1, bool SHADOW, int MODE>
__global__ void __launch_bounds__(kMixThreads, 1) k_mix(const __grid_constant__ CUtensorMap tmap, const MixArgs a) {
  extern __shared__ unsigned char smem_raw[];
  constexpr bool FUSED = MODE != kMixPlain;
  constexpr bool ENTRIES = MODE == kMixEntries;
  constexpr bool STEP = KP1 == kStepOnly;
  constexpr int kGroups = mix_groups(MODE), kCompute = mix_group_threads(MODE);
  const int kp1 = KP1 > 0 ? KP1 : (KP1 == 0 ? a.kp1 : 0);
  MixSmem sm = carve(smem_raw, a, kp1, MODE);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = a.S, nq = S >> 2;            // column quads per slab, a power of two <= 256
  const int lq = __ffs(nq) - 1;
  const int lS = lq + 2;
  const int QB = nq < 64 ? nq : 64;           // quads per TMA box row (a box spans <= 256 columns)
  const int lqb = __ffs(QB) - 1;
  const int box_col = a.rows_pad << lqb;      // float4s per column box of a slab
  const int G = kCompute >> lq;               // row groups: compute threads that share a column quad
  const size_t slab_floats = static_cast<size_t>(a.rows_pad) * S;
  const size_t list_off = (slab_floats * 4 + 15) & ~static_cast<size_t>(15);
  const size_t list_bytes = (static_cast<size_t>(a.max_region) * 4 + 15) & ~static_cast<size_t>(15);

  // Before the previous kernel is waited for: barriers, and the mixing table,
  // which is complete on the device before the kernels of its round begin.
  // (With these and the flags after the wait and before the first loads, and
  // slabs of 32 KB for every size, a reduce of N = 8, d = 10^5 took 10.8 us in a
  // row of reduces, now 9.7; the RCV1-shaped one 18.5 us, now 16.7.)
  if (tid == 0) {
    sm.flags[0] = 0;
    sm.flags[1] = 0;
    sm.flags[3] = 0;
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(sm.full + s, 1);
      mbar_init(sm.empty + s, kMixComputeWarps / kGroups);
      mbar_init(sm.ready + s, kMixUpdaterWarps);
    }
    for (int s = 0; s < a.list_slots; ++s) mbar_init(sm.lfull + s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 32) sm.seen[tid] = 0u;
  if (KP1 >= 0) {
    for (int idx = tid; idx < a.N * kp1; idx += kMixThreads) {
      sm.nbr[idx] = a.nbr[idx] * QB;       // float4 offset of the neighbour's row within a box column
      sm.wgt[idx] = a.wgt[idx] * a.wscale;
    }
  }
  __syncthreads();
  // A gated reduce (NOTIFY_ACK or ASYNC, sparse models) runs while the local
  // step may still be running: it reads the column sums of worker j only
  // after j's NOTIFY (or, ASYNC, counts the read as stale).  Otherwise
  // (BSP) it starts once the local step's grid has finished.
  const bool gated = FUSED && a.sync_mode != kSyncBsp;
  if (!gated) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // The next round's local step (a programmatic dependent) may now be
    // scheduled as this grid drains; it waits for this grid before it reads
    // what this grid writes.  A gated reduce leaves the trigger to its exit,
    // since the local step it overlaps is still running; so does the update of
    // an intermediate local step, or a gated reduce, let in by the next local
    // step's own trigger, could read parameters this grid has yet to update.
    if constexpr (!STEP) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }

  // ---- NOTIFY / ACK checks (time-limited waits) ----
  // A gated reduce checks the ACKs before it reads anything.  Otherwise the
  // grid before has finished and its flags are final: they are checked while
  // the first slabs fly, by all warps but the producer's, and before anything
  // is written.
  auto check_flags = [&](int first, int step) {
    bool bad = false;
    for (int j = first; j < a.N; j += step) {
      unsigned e = 0;
      const bool own = j >= a.own_lo && j < a.own_lo + a.own_n;
      if (a.expect_notify && !gated && own) e = wait_flag(a.ready + j, a.round + 1u, true, a.wait_ns);
      if (!e) e = wait_flag(a.consumed + j, a.round, false, a.wait_ns);
      if (e) {
        record_error(a.st, e, j, a.round);
        if (e == ASAP_ERR_TIMEOUT) atomicAdd(&a.st->timeouts, 1ull);
        atomicOr(&sm.flags[0], 1);
        bad = true;
      }
    }
    __syncwarp();
    return bad;
  };
  if (gated) {
    check_flags(tid, kMixThreads);
    __syncthreads();
    // W is there by the ACKs; the copies read it through the async proxy.
    if (warp == kProducerWarp) asm volatile("fence.proxy.async.global;" ::: "memory");
  }
  bool failed = gated && sm.flags[0] != 0;
  bool quiet = false;                    // a flag was missing: pass the slabs on, write nothing
  if (!STEP && !gated && warp != kProducerWarp)
    quiet = start_bar_or(check_flags(tid < kProducerWarp * 32 ? tid : tid - 32, kMixThreads - 32));

  float s2 = 0.f;      // compute threads: sum of (w - K)^2;  producer lanes: -sum of S1^2 / N
  if (!failed) {
    const long long stride = gridDim.x;
    const int n_my = static_cast<int>((a.n_slabs - blockIdx.x + stride - 1) / stride);   // slabs of this CTA
    const float inv_n = 1.0f / static_cast<float>(a.N);

    const uint64_t policy = evict_first_policy();
    if (warp == kProducerWarp) {
      // ================= producer warp =================
      float term = 0.f;
      const float inv_n_term = 1.0f / static_cast<float>(a.N);
      unsigned long long n_read = 0, n_current = 0;   // gated: (slab, worker) inputs, and those current
      int n_seen = 0;                                 // gated: workers whose NOTIFY this CTA has seen
      // List offsets of the next 32 slabs, one slab per lane, loaded ahead so
      // that issuing a stage never waits on a global load.
      int4 offs = make_int4(0, 0, 0, 0);
      int2 loffs = make_int2(0, 0);                   // entry ring: the same, list_slots - stages slabs ahead
      int st = 0, done_st = 0;                        // stages of slab it, and of the slab that came back
      uint32_t done_ph = 0;
      // a.depth slabs are asked for at most: a slab goes out when the one
      // a.depth before has come back (its own stage has by then, a.stages >= a.depth).
      for (int it = 0; it < n_my + a.depth; ++it) {
        if (!STEP && !gated && it == min(a.depth, n_my)) start_bar_or(false);
        if (FUSED && (it & 31) == 0 && it < n_my) {
          const long long sl = blockIdx.x + static_cast<long long>(it + lane) * stride;
          if (it + lane < n_my)
            offs = ENTRIES ? make_int4(__ldg(a.upd.off + sl), __ldg(a.upd.off + sl + 1), __ldg(a.exp.off + sl),
                                       __ldg(a.exp.off + sl + 1))
                           : make_int4(__ldg(a.upd_off + sl), __ldg(a.upd_off + sl + 1), __ldg(a.exp_off + sl),
                                       __ldg(a.exp_off + sl + 1));
        }
        int4 o = make_int4(0, 0, 0, 0);
        if (FUSED) {
          const int src = it & 31;
          o.x = __shfl_sync(kFull, offs.x, src);
          o.y = __shfl_sync(kFull, offs.y, src);
          o.z = __shfl_sync(kFull, offs.z, src);
          o.w = __shfl_sync(kFull, offs.w, src);
        }
        if (it >= a.depth) {
          bool ok = (lane == 0) ? mbar_wait_bounded(sm.empty + done_st, done_ph) : true;
          ok = __shfl_sync(kFull, ok, 0) != 0;   // warp-uniform outcome
          __syncwarp();
          if (!ok) {
            if (lane == 0) record_error(a.st, ASAP_ERR_CUDA, 0xfffffffeu, a.round);
            failed = true;
            // A slab that never comes back: those who wait for copies may have
            // given up, and the CTA's shared memory must not be given back with
            // one in flight.  (A slab that comes back has landed, its entries too.)
            const int slabs = min(it, n_my), lists = min(it + a.list_slots - a.stages, n_my);
            if (lane < a.stages && lane < slabs)
              mbar_wait_bounded(sm.full + lane, static_cast<uint32_t>((slabs - 1 - lane) / a.stages) & 1u);
            if (ENTRIES && lane < a.list_slots && lane < lists)
              mbar_wait_bounded(sm.lfull + lane, static_cast<uint32_t>((lists - 1 - lane) / a.list_slots) & 1u);
            __syncwarp();
            break;
          }
        }
        if (FUSED && gated && it < n_my) {
          // The slab's updates come from workers w0 .. w1 (a region is sorted
          // by worker): their NOTIFY for the round before the slab's column
          // sums are copied (NOTIFY_ACK, time-limited waits), or just noted
          // (ASYNC).  The warp checks 32 workers at a time; a worker seen
          // once stays seen for the rest of the launch.
          const int nu = o.y - o.x;
          if (n_seen == a.N) {
            n_read += static_cast<unsigned long long>(a.N);
            n_current += static_cast<unsigned long long>(a.N);
          } else if (nu > 0) {
            const uint32_t* codes = ENTRIES ? a.upd.code : a.upd_list;
            auto worker_of = [&](uint32_t c) { return ENTRIES ? (c & kEntryOff) >> lS : c >> 16; };
            const unsigned w0 = worker_of(__ldg(codes + o.x));
            unsigned w1 = w0;
            for (int e = nu - 1; e >= 0 && e >= nu - 8; --e) {   // past the region's padding
              const uint32_t c = __ldg(codes + o.x + e);
              if (c != kListPad) { w1 = worker_of(c); break; }
            }
            bool acquired = false;
            for (unsigned j0 = w0; j0 <= w1 && j0 < static_cast<unsigned>(a.N); j0 += 32) {
              const unsigned j = j0 + lane;
              const bool in = j <= w1 && j < static_cast<unsigned>(a.N);
              const unsigned bit = 1u << (j & 31u);
              bool cur = in && (sm.seen[j >> 5] & bit) != 0;
              bool fresh = false;
              if (in && !cur && !failed) {
                if (a.sync_mode == kSyncNotifyAck) {
                  const unsigned er = wait_flag(a.ready + j, a.round + 1u, true, a.wait_ns);
                  if (er) {
                    record_error(a.st, er, j, a.round);
                    if (er == ASAP_ERR_TIMEOUT) atomicAdd(&a.st->timeouts, 1ull);
                    failed = true;
                  } else {
                    fresh = true;
                  }
                } else {
                  fresh = ld_acquire_u32(a.ready + j) == a.round + 1u;
                }
                if (fresh) atomicOr(sm.seen + (j >> 5), bit);
                cur = fresh;
              }
              n_seen += __popc(__ballot_sync(kFull, fresh));
              acquired = acquired || __any_sync(kFull, fresh);
              n_read += __popc(__ballot_sync(kFull, in));
              n_current += __popc(__ballot_sync(kFull, in && cur));
            }
            failed = __any_sync(kFull, failed);
            __syncwarp();
            // newly acquired column sums, to the bulk copy's async proxy
            if (acquired && lane == 0) asm volatile("fence.proxy.async.global;" ::: "memory");
          }
        }
        // The updater warps may look up r for the slabs passed, and for all of them
        // once every worker has been seen.  (Only ever the slabs passed, the early
        // look-up mostly missed its turn: N = 64, d = 2^20, 110 entries a row 150
        // us a NOTIFY_ACK round, now 123; 150 entries a row 170, now 155.)
        if (ENTRIES && gated && it < n_my && lane == 0)
          st_release_cta(sm.flags + 3, n_seen == a.N ? 0x7fffffff : it + 1);
        if (it < n_my && lane == 0) {
          const long long slab = blockIdx.x + it * stride;
          unsigned char* base = sm.stage0 + st * sm.stage_bytes;
          uint32_t bytes = static_cast<uint32_t>(a.n_boxes) * a.box_rows * S * 4u;
          int n_upd = 0, n_exp = 0, x0 = 0, u0 = 0;
          if (FUSED) {
            u0 = o.x;
            n_upd = o.y - o.x;
            x0 = o.z;
            n_exp = o.w - o.z;
            bytes += ENTRIES ? (a.exp.place ? 10u : 8u) * n_exp : 8u * n_upd + 4u * n_exp;
          }
          *reinterpret_cast<int4*>(sm.info + 4 * st) = make_int4(n_upd, n_exp, x0, u0);
          mbar_expect_only(sm.full + st, bytes);
          // Slab layout in shared memory: [column box][row][QB quads].
          for (int xb = 0; xb < nq / QB; ++xb)
            for (int b = 0; b < a.n_boxes; ++b)
              tma_load_2d(base + (static_cast<size_t>(xb) * a.rows_pad + static_cast<size_t>(b) * a.box_rows) * QB * 16,
                          &tmap, sm.full + st, static_cast<int>(slab * S + xb * QB * 4), b * a.box_rows, policy);
          if (ENTRIES) {
            if (n_exp > 0) {
              bulk_load(base + list_off, a.exp.code + x0, 4u * n_exp, sm.full + st);
              bulk_load(base + list_off + list_bytes, a.exp.val + x0, 4u * n_exp, sm.full + st);
              if (a.exp.place)
                bulk_load(base + list_off + 2 * list_bytes, a.exp.place + x0, 2u * n_exp, sm.full + st);
            }
          } else if (FUSED) {
            if (n_upd > 0) {
              bulk_load(base + list_off, a.upd_list + u0, 4u * n_upd, sm.full + st);
              bulk_load(base + list_off + list_bytes, a.gsum + u0, 4u * n_upd, sm.full + st);
            }
            if (n_exp > 0) bulk_load(base + list_off + 2 * list_bytes, a.exp_list + x0, 4u * n_exp, sm.full + st);
          }
        }
        if (ENTRIES) {
          // The entries of the slab list_slots - stages ahead: their slot is
          // that of the slab whose stage has just come back.  (At first, also
          // those of the slabs before.)
          const int ahead = a.list_slots - a.stages;
          for (int j = it > 0 ? it + ahead : 0; j <= it + ahead && j < n_my; ++j) {
            if ((j & 31) == 0) {
              const long long sl = blockIdx.x + static_cast<long long>(j + lane) * stride;
              if (j + lane < n_my) loffs = make_int2(__ldg(a.upd.off + sl), __ldg(a.upd.off + sl + 1));
            }
            const int u0 = __shfl_sync(kFull, loffs.x, j & 31);
            const int n = __shfl_sync(kFull, loffs.y, j & 31) - u0;
            if (lane != 0) continue;
            const int slot = j % a.list_slots;
            unsigned char* dst = sm.lists + slot * sm.list_bytes;
            sm.linfo[slot] = n;
            mbar_expect_tx(sm.lfull + slot, 8u * n);
            if (n > 0) {
              bulk_load(dst, a.upd.code + u0, 4u * n, sm.lfull + slot);
              bulk_load(dst + 4 * static_cast<size_t>(a.max_region), a.upd.val + u0, 4u * n, sm.lfull + slot);
            }
          }
          __syncwarp();
        }
        // The column sums of the slab that came back, while the next one's
        // copies fly: its stage cannot be handed on before the arrival below.
        // (Added up before the copies were issued, they lengthened every
        // stage's turnaround by about a microsecond: the hashed workload's
        // reduce took 141 us instead of 128.)
        if (it >= a.depth && KP1 >= 0) {
          const float4* p = sm.part + done_st * kCompute;
          for (int q = lane; q < nq; q += 32) {
            float4 t = p[q];
            for (int g = 1; g < G; ++g) t = f4_add(t, p[g * nq + q]);
            term = fmaf(fmaf(t.x, t.x, fmaf(t.y, t.y, fmaf(t.z, t.z, t.w * t.w))), inv_n_term, term);
          }
        }
        __syncwarp();
        if (it < n_my && lane == 0) mbar_arrive(sm.full + st);
        if (it >= a.depth && ++done_st == a.stages) {
          done_st = 0;
          done_ph ^= 1u;
        }
        if (++st == a.stages) st = 0;
      }
      s2 = -term;
      if (gated && lane == 0 && n_read) {
        atomicAdd(&a.st->inputs_read, n_read);
        atomicAdd(&a.st->inputs_current, n_current);
      }
    } else if (warp >= kUpdater0) {
      // ================= updater warps (FUSED) =================
      // Once a slab has landed, apply w -= eta/B (1 - eta l2)^-1 g to it and
      // release it to the compute warps.
      if (FUSED && quiet) {
        // The entry ring goes round with the stages: a slot is armed again when
        // its slab's stage comes back, so its entries must have landed too.
        int st = 0, sl = 0;
        uint32_t ph = 0, lph = 0;
        for (int it = 0; it < n_my; ++it) {
          bool here = mbar_wait_bounded(sm.full + st, ph);
          if (ENTRIES) here = mbar_wait_bounded(sm.lfull + sl, lph) && here;
          if (!__all_sync(kFull, here)) break;
          if (ENTRIES && ++sl == a.list_slots) {
            sl = 0;
            lph ^= 1u;
          }
          if (lane == 0) mbar_arrive(sm.ready + st);
          if (++st == a.stages) {
            st = 0;
            ph ^= 1u;
          }
        }
      } else if constexpr (ENTRIES) {
        update_entries<STEP>(sm, a, n_my, gated, lS, lqb, box_col, failed);
      } else if (FUSED) {
        const int ut = tid - kUpdater0 * 32;
        int st = 0;
        uint32_t ph = 0;
        for (int it = 0; it < n_my; ++it) {
          const bool ok = __all_sync(kFull, mbar_wait_bounded(sm.full + st, ph));
          if (!ok) {
            if (lane == 0) record_error(a.st, ASAP_ERR_CUDA, 0xfffffffdu, a.round);
            failed = true;
            break;
          }
          unsigned char* bj = sm.stage0 + st * sm.stage_bytes;
          float* xj = reinterpret_cast<float*>(bj);
          const uint32_t* ul = reinterpret_cast<const uint32_t*>(bj + list_off);
          const float* ug = reinterpret_cast<const float*>(bj + list_off + list_bytes);
          const int n_upd = sm.info[4 * st];
          // Four entries per thread in flight: the (worker, column) pairs of
          // one list are distinct, so the four read-modify-writes never alias.
          constexpr int kUpd = kMixUpdaterWarps * 32, kU = 4;
          for (int e0 = ut; e0 < n_upd; e0 += kU * kUpd) {
            uint32_t code[kU];
            float gv[kU], wv[kU] = {};
            int off[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
              const int e = e0 + u * kUpd;
              code[u] = e < n_upd ? ul[e] : kListPad;
              gv[u] = e < n_upd ? ug[e] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
              const int i = static_cast<int>(code[u] >> 16), cl = static_cast<int>(code[u] & 0xffffu);
              const int q = cl >> 2;
              off[u] = 4 * ((i << lqb) + (q >> lqb) * box_col + (q & (QB - 1))) + (cl & 3);
              if (code[u] != kListPad) wv[u] = xj[off[u]];
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
              if (code[u] != kListPad) xj[off[u]] = fmaf(-a.upd_scale, gv[u], wv[u]);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before this stage's next TMA
          __syncwarp();
          if (lane == 0) mbar_arrive(sm.ready + st);
          if (++st == a.stages) {
            st = 0;
            ph ^= 1u;
          }
        }
      }
    } else {
      // ================= compute warps =================
      // Group k takes the slabs k, k + kGroups, ... of the CTA; its thread t
      // owns column quad q = t mod nq of them for the rows i = g, g + G, ...
      // (g = t / nq): with ~32 KB slabs that is 4 or 8 rows.
      const int group = tid / kCompute, gt = tid - group * kCompute;
      const int q_t = gt & (nq - 1), g_t = gt >> lq;
      const uint64_t keep = evict_last_policy();
      const int qoff = (q_t >> lqb) * box_col + (q_t & (QB - 1));   // float4 offset of (row 0, quad q_t)
      const int rows_t = (a.N - g_t + G - 1) / G;
      auto xq = [&](int q) { return (q >> lqb) * box_col + (q & (QB - 1)); };
      // Entry layout: value * w of the stage's export entry e, to its row.
      auto export_product = [&](uint32_t code, int e, const unsigned char* base, float w) {
        const float val = reinterpret_cast<const float*>(base + list_off + list_bytes)[e];
        const uint32_t place = a.exp.place ? reinterpret_cast<const uint16_t*>(base + list_off + 2 * list_bytes)[e]
                                           : (code >> 16) & ((1u << (a.exp.row_shift - 16)) - 1u);
        const int64_t row = static_cast<int64_t>((code & kEntryOff) >> lS) * a.B + (code >> a.exp.row_shift);
        st_f32_hint(a.prod_out + row * a.row_stride + place, val * w, keep);
      };
      // With a compile-time neighbour count and at most kCacheRows rows per
      // thread, the neighbour offsets of the thread's rows (its quad folded
      // in) stay in registers as 16-bit pairs, and an equal weight in one
      // register: the slab loop then reads only the slab from shared memory.
      constexpr int kCacheRows = 4 * kGroups;   // all of a thread's rows, with 32 KB slabs
      constexpr int kC = KP1 > 0 ? KP1 : 1;
      constexpr int kPk = (kCacheRows * kC + 1) / 2;
      const bool cached = KP1 > 0 && rows_t <= kCacheRows;
      uint32_t pko[kPk];
#pragma unroll
      for (int u = 0; u < kPk; ++u) pko[u] = 0u;
      if (KP1 > 0 && cached) {
#pragma unroll
        for (int rr = 0; rr < kCacheRows; ++rr)
#pragma unroll
          for (int m = 0; m < kC; ++m) {
            const int e = rr * kC + m;
            const uint32_t off = rr < rows_t ? static_cast<uint32_t>(sm.nbr[(g_t + rr * G) * kC + m] + qoff) : 0u;
            pko[e >> 1] |= (off & 0xffffu) << (16 * (e & 1));
          }
      }
      const bool uni = a.uniform_w != 0;
      const float wu = uni && KP1 >= 0 ? sm.wgt[0] : 0.f;
      int st = group;
      uint32_t ph = 0;
      for (int it = group; it < n_my; it += kGroups) {
        if (st >= a.stages) {
          st = group;
          ph ^= 1u;
        }
        const long long slab = blockIdx.x + it * stride;
        bool ok = __all_sync(kFull, mbar_wait_bounded(FUSED ? sm.ready + st : sm.full + st, ph));
        unsigned char* base = sm.stage0 + st * sm.stage_bytes;
        float* x = reinterpret_cast<float*>(base);
        const float4* x4 = reinterpret_cast<const float4*>(base);
        const int* info = sm.info + 4 * st;
        float4* part = sm.part + st * kCompute;
        const long long c0 = slab * S;
        if (quiet) {                     // the same for every compute thread
          __syncwarp();
          if (lane == 0) mbar_arrive(sm.empty + st);
          st += kGroups;
          if (!ok) break;
          continue;
        }
        if (ok && KP1 == -1) {
          // Complete graph: this thread's share of its column's sum.
          float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int r = 0; r < rows_t; ++r) cs = f4_add(cs, x4[(g_t + r * G) * QB + qoff]);
          part[gt] = cs;
        }
        if (KP1 == -1) ok = !compute_bar_or<kCompute>(group, !ok);   // uniform decision; the column sums are visible
        if (!ok) {
          if (lane == 0) record_error(a.st, ASAP_ERR_CUDA, 0xffffffffu, a.round);
          failed = true;
          break;
        }
        if constexpr (STEP) {
          const uint32_t* xl = reinterpret_cast<const uint32_t*>(base + list_off);
          for (int e = gt; e < info[1]; e += kCompute) {
            const uint32_t code = xl[e];
            if (code == kListPad) continue;
            const int cl = static_cast<int>(code & static_cast<uint32_t>(S - 1));
            const int i = static_cast<int>((code & kEntryOff) >> lS);
            export_product(code, e, base, x[4 * ((i << lqb) + xq(cl >> 2)) + (cl & 3)]);
          }
        } else if constexpr (KP1 == -1) {
          // Complete graph: column means (threads t < nq), then every row gets them.
          if (gt < nq) {
            float4 t = part[gt];
            for (int g = 1; g < G; ++g) t = f4_add(t, part[g * nq + gt]);
            const float sc = inv_n * a.wscale;
            part[gt] = make_float4(t.x * sc, t.y * sc, t.z * sc, t.w * sc);
          }
          compute_bar<kCompute>(group);
          const float4 mean = part[q_t];
          for (int r = 0; r < rows_t; ++r) {
            const int i = g_t + r * G;
            const long long c = c0 + 4 * q_t;
            if (c < a.ld) {
              st_f4_hint(a.out + static_cast<int64_t>(i) * a.ld + c, mean, policy);
              if (SHADOW) {
                __nv_bfloat162 lo = __floats2bfloat162_rn(mean.x, mean.y);
                __nv_bfloat162 hi = __floats2bfloat162_rn(mean.z, mean.w);
                uint2 pk;
                pk.x = *reinterpret_cast<uint32_t*>(&lo);
                pk.y = *reinterpret_cast<uint32_t*>(&hi);
                *reinterpret_cast<uint2*>(a.shadow + static_cast<int64_t>(i) * a.ld + c) = pk;
              }
            }
          }
          if (FUSED) {
            const uint32_t* xl = reinterpret_cast<const uint32_t*>(base + list_off + (ENTRIES ? 0 : 2 * list_bytes));
            const int n_exp = info[1], xbase = info[2];
            const float* means = reinterpret_cast<const float*>(part);
            for (int e = gt; e < n_exp; e += kCompute) {
              const uint32_t code = xl[e];
              if (code == kListPad) continue;
              if constexpr (ENTRIES)
                export_product(code, e, base, means[code & static_cast<uint32_t>(S - 1)]);
              else
                a.wv_out[xbase + e] = means[code & 0xffffu];
            }
          }
          compute_bar<kCompute>(group);   // the means are read before the next slab's sums overwrite them
        } else {
          const float4 K = x4[qoff];        // shift: row 0 of the (updated) slab
          float4 s1 = make_float4(0.f, 0.f, 0.f, 0.f);
          float sq = 0.f;
          auto mix_one = [&](int i) -> float4 {
            const int* nb = sm.nbr + i * kp1;
            const float* wt = sm.wgt + i * kp1;
            const float4 xa = x4[nb[0] + qoff];
            float4 acc = make_float4(wt[0] * xa.x, wt[0] * xa.y, wt[0] * xa.z, wt[0] * xa.w);
#pragma unroll
            for (int m = 1; m < (KP1 > 0 ? KP1 : kMaxKp1Sparse); ++m) {
              if (KP1 == 0 && m >= kp1) break;
              acc = f4_fma(wt[m], x4[nb[m] + qoff], acc);
            }
            return acc;
          };
          auto emit = [&](int i, float4 acc) {
            const long long c = c0 + 4 * q_t;
            if (c < a.ld) {
              st_f4_hint(a.out + static_cast<int64_t>(i) * a.ld + c, acc, policy);
              if (SHADOW) {
                __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y);
                __nv_bfloat162 hi = __floats2bfloat162_rn(acc.z, acc.w);
                uint2 pk;
                pk.x = *reinterpret_cast<uint32_t*>(&lo);
                pk.y = *reinterpret_cast<uint32_t*>(&hi);
                *reinterpret_cast<uint2*>(a.shadow + static_cast<int64_t>(i) * a.ld + c) = pk;
              }
            }
            const float dx = acc.x - K.x, dy = acc.y - K.y, dz = acc.z - K.z, dw = acc.w - K.w;
            s1 = f4_add(s1, make_float4(dx, dy, dz, dw));
            sq = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, fmaf(dw, dw, sq))));
          };
          if (KP1 > 0 && cached) {
            // the same operations in the same order as mix_one, offsets from registers
            auto mix_c = [&](int rr) -> float4 {
              const float* wt = sm.wgt + (g_t + rr * G) * kC;
              auto xo = [&](int m) {
                const int e = rr * kC + m;
                return static_cast<int>((pko[e >> 1] >> (16 * (e & 1))) & 0xffffu);
              };
              const float w0 = uni ? wu : wt[0];
              const float4 xa = x4[xo(0)];
              float4 acc = make_float4(w0 * xa.x, w0 * xa.y, w0 * xa.z, w0 * xa.w);
#pragma unroll
              for (int m = 1; m < kC; ++m) acc = f4_fma(uni ? wu : wt[m], x4[xo(m)], acc);
              return acc;
            };
#pragma unroll
            for (int rr = 0; rr < kCacheRows; rr += 2) {   // two rows in flight
              if (rr + 1 < rows_t) {
                const float4 a0 = mix_c(rr);
                const float4 a1 = mix_c(rr + 1);
                emit(g_t + rr * G, a0);
                emit(g_t + (rr + 1) * G, a1);
              } else if (rr < rows_t) {
                emit(g_t + rr * G, mix_c(rr));
              }
            }
          } else {
            int r = 0;
            for (; r + 1 < rows_t; r += 2) {      // two rows in flight
              const int i0 = g_t + r * G, i1 = i0 + G;
              const float4 a0 = mix_one(i0);
              const float4 a1 = mix_one(i1);
              emit(i0, a0);
              emit(i1, a1);
            }
            if (r < rows_t) emit(g_t + r * G, mix_one(g_t + r * G));
          }
          s2 += sq;
          part[gt] = s1;
          if (FUSED) {
            // w_{t+1} at the next round's columns, recomputed with the same
            // operations in the same order as the stored outputs.
            const uint32_t* xl = reinterpret_cast<const uint32_t*>(base + list_off + (ENTRIES ? 0 : 2 * list_bytes));
            const int n_exp = info[1], xbase = info[2];
            for (int e = gt; e < n_exp; e += kCompute) {
              const uint32_t code = xl[e];
              if (code == kListPad) continue;
              const int i = static_cast<int>(ENTRIES ? (code & kEntryOff) >> lS : code >> 16);
              const int cl = static_cast<int>(ENTRIES ? code & static_cast<uint32_t>(S - 1) : code & 0xffffu);
              const int* nb = sm.nbr + i * kp1;
              const float* wt = sm.wgt + i * kp1;
              const int xo = xq(cl >> 2), comp = cl & 3;
              float v = (uni ? wu : wt[0]) * x[4 * (nb[0] + xo) + comp];
#pragma unroll
              for (int m = 1; m < (KP1 > 0 ? KP1 : kMaxKp1Sparse); ++m) {
                if (KP1 == 0 && m >= kp1) break;
                v = fmaf(uni ? wu : wt[m], x[4 * (nb[m] + xo) + comp], v);
              }
              if constexpr (ENTRIES) export_product(code, e, base, v);
              else st_f32_hint(a.wv_out + xbase + e, v, keep);
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(sm.empty + st);
        st += kGroups;
      }
    }
  }

  if constexpr (STEP) return;

  // ---- per-CTA partial, ticket, and the last CTA's finalisation ----
  F2* scratch = sm.scratch;
  if (failed && lane == 0) atomicOr(&sm.flags[0], 1);
  const F2 csum = block_sum_f2(F2{s2, 0.f}, scratch);
  if (tid == 0) a.cons_part[blockIdx.x] = make_float2(csum.hi, csum.lo);
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    if (sm.flags[0]) atomicAdd(&a.st->mix_ticket, 0x10000u);   // high half counts failed CTAs
    // Every CTA adds its failure before its ticket, to the same word: the
    // last ticket's old value already holds every CTA's failure count.
    const unsigned t = atomicAdd(&a.st->mix_ticket, 1u);
    sm.flags[1] = ((t & 0xffffu) == gridDim.x - 1) ? 1 : 0;
    sm.flags[2] = static_cast<int>(t >> 16);
    // The next reduce's tickets may come as soon as the ACK below is out.
    if (sm.flags[1]) a.st->mix_ticket = 0u;
  }
  __syncthreads();
  if (!sm.flags[1]) return;
  __threadfence();
  bool any_fail = sm.flags[2] != 0;
  // Consensus partials of every CTA, and the loss partials: read together
  // unless NOTIFY_ACK must first see every worker's NOTIFY (the loss
  // partials of workers without any update in this launch's slabs).
  const bool loss_after_notify = gated && a.sync_mode == kSyncNotifyAck;
  const int n_cons = static_cast<int>(gridDim.x);
  const int n_lp = a.have_loss ? a.n_loss_part : 0;
  F2 ctot{0.f, 0.f}, ltot{0.f, 0.f};
  for (int b = tid; b < (loss_after_notify ? n_cons : max(n_cons, n_lp)); b += kMixThreads) {
    if (b < n_cons) {
      const float2 p = __ldcg(a.cons_part + b);
      ctot = f2_add(ctot, F2{p.x, p.y});
    }
    if (!loss_after_notify && b < n_lp) ltot = f2_add(ltot, F2{__ldcg(a.loss_part + b), 0.f});
  }
  if (loss_after_notify) {
    if (!any_fail) {
      for (int j = tid; j < a.N; j += kMixThreads) {
        const unsigned er = wait_flag(a.ready + j, a.round + 1u, true, a.wait_ns);
        if (er) {
          record_error(a.st, er, j, a.round);
          atomicOr(&sm.flags[0], 2);
        }
      }
      __syncthreads();
      any_fail = (sm.flags[0] & 2) != 0;
    }
    for (int b = tid; b < n_lp; b += kMixThreads) ltot = f2_add(ltot, F2{__ldcg(a.loss_part + b), 0.f});
  }
  block_sum2_f2(ctot, ltot, scratch);   // its barriers: every partial is read, the ticket reset, before the ACK
  if (!any_fail)
    for (int j = tid; j < a.N; j += kMixThreads) {
      a.stamp_next[j] = a.round + 1u;
      st_release_u32(a.consumed + j, a.round + 1u);
    }
  if (tid == 0) {
    const int slot = static_cast<int>(a.round % kMetricsCap);
    // Rounding may leave a little below 0; a NaN (parameters that are not
    // finite) stays one.
    const float c2 = ctot.hi + ctot.lo;
    a.metrics_cons[slot] = any_fail ? __int_as_float(0x7fc00000) : sqrtf(c2 < 0.f ? 0.f : c2);
    a.metrics_loss[slot] = (a.have_loss && !any_fail) ? (ltot.hi + ltot.lo) * a.loss_norm
                                                      : __int_as_float(0x7fc00000);
    if (!any_fail) {
      atomicAdd(&a.st->reduces, static_cast<unsigned long long>(a.own_n));
      if (a.expect_notify)
        atomicAdd(&a.st->consistent_inputs, static_cast<unsigned long long>(a.own_n) * (KP1 < 0 ? a.N : kp1));
    }
  }
}

template <int KP1, bool SHADOW, int MODE>
struct MixKernel {
  // The limit is the function's, not a launch's: contexts of other sizes
  // share it, so it is always the device's (227 KB).
  static cudaError_t attr() {
    return cudaFuncSetAttribute(k_mix<KP1, SHADOW, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 << 10);
  }
  static cudaError_t occ(size_t smem, int* blocks) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k_mix<KP1, SHADOW, MODE>, kMixThreads, smem);
  }
  static cudaError_t launch(const CUtensorMap& tmap, const MixArgs& a, int grid, size_t smem, cudaStream_t s) {
    // A programmatic dependent of the local step's last kernel.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kMixThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_mix<KP1, SHADOW, MODE>, tmap, a);
  }
};

// Dispatch over (complete / k+1, shadow, mode); K is a functor template.
template <template <int, bool, int> class K, bool SHADOW, int MODE>
struct ByKp1 {
  template <typename F>
  static cudaError_t go(bool complete, int kp1, F&& f) {
    if (complete) return f(K<-1, SHADOW, MODE>());
    switch (kp1) {
      case 1: return f(K<1, SHADOW, MODE>());
      case 2: return f(K<2, SHADOW, MODE>());
      case 3: return f(K<3, SHADOW, MODE>());
      case 5: return f(K<5, SHADOW, MODE>());
      default: return f(K<0, SHADOW, MODE>());
    }
  }
};

template <typename F>
cudaError_t dispatch(bool complete, int mode, int kp1, bool shadow, F&& f) {
  if (shadow) {
    if (mode != kMixPlain) return cudaErrorInvalidValue;   // dense models never fuse a sparse update
    return ByKp1<MixKernel, true, kMixPlain>::go(complete, kp1, f);
  }
  switch (mode) {
    case kMixLists: return ByKp1<MixKernel, false, kMixLists>::go(complete, kp1, f);
    case kMixEntries: return ByKp1<MixKernel, false, kMixEntries>::go(complete, kp1, f);
    default: return ByKp1<MixKernel, false, kMixPlain>::go(complete, kp1, f);
  }
}

__global__ void k_cast_bf16(const float* __restrict__ src, uint16_t* __restrict__ dst, int64_t n) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    __nv_bfloat16 b = __float2bfloat16_rn(src[i]);
    dst[i] = *reinterpret_cast<uint16_t*>(&b);
  }
}

}  // namespace

ASAP_HD size_t mix_stage_bytes(int S, int rows_pad, int max_region, int mode) {
  const size_t slab = (static_cast<size_t>(rows_pad) * S * 4 + 15) & ~static_cast<size_t>(15);
  const size_t list = (static_cast<size_t>(max_region) * 4 + 15) & ~static_cast<size_t>(15);
  // lists: update codes and sums, export codes; entries: the export's codes,
  // values and places
  const size_t lists = mode == kMixEntries ? 2 * list + ((list / 2 + 15) & ~static_cast<size_t>(15)) : 3 * list;
  return (slab + lists + 1023) & ~static_cast<size_t>(1023);
}

size_t mix_smem_bytes(int N, int kp1, int S, int rows_pad, int stages, int max_region, int mode, int list_slots) {
  auto a16 = [](size_t v) { return (v + 15) & ~static_cast<size_t>(15); };
  size_t b = 1024 + mix_stage_bytes(S, rows_pad, max_region, mode) * stages;   // alignment slack + stages
  b = a16(b + 12 * static_cast<size_t>(max_region) * list_slots);        // entry ring
  b = a16(b + 24 * static_cast<size_t>(stages) + 12 * static_cast<size_t>(list_slots));   // mbarriers, entry counts
  b = a16(b + 16 * (kMixThreads / 32));                                   // block-sum scratch (two fp32 pairs a warp)
  b = a16(b + 16);                                                        // flags
  b = a16(b + 4 * 32);                                                    // NOTIFY bitmap
  b = a16(b + 16 * static_cast<size_t>(stages));                          // stage info
  b = a16(b + 16 * static_cast<size_t>(stages) * mix_group_threads(mode));   // partial sums
  b = a16(b + 4 * static_cast<size_t>(N) * kp1);                          // neighbour offsets
  return b + 4 * static_cast<size_t>(N) * kp1;                            // weights
}

cudaError_t mix_configure(bool complete, int mode, int kp1, bool shadow) {
  return dispatch(complete, mode, kp1, shadow, [&](auto k) { return decltype(k)::attr(); });
}

cudaError_t mix_occupancy(bool complete, int mode, int kp1, bool shadow, size_t smem, int* blocks) {
  return dispatch(complete, mode, kp1, shadow, [&](auto k) { return decltype(k)::occ(smem, blocks); });
}

cudaError_t launch_mix(const CUtensorMap& tmap, const MixArgs& a, bool complete, int mode, int grid, size_t smem,
                       cudaStream_t s) {
  return dispatch(complete, mode, a.kp1, a.shadow != nullptr,
                  [&](auto k) { return decltype(k)::launch(tmap, a, grid, smem, s); });
}

cudaError_t entry_step_configure() { return MixKernel<kStepOnly, false, kMixEntries>::attr(); }

cudaError_t launch_entry_step(const CUtensorMap& tmap, const MixArgs& a, int grid, size_t smem, cudaStream_t s) {
  return MixKernel<kStepOnly, false, kMixEntries>::launch(tmap, a, grid, smem, s);
}

cudaError_t launch_cast_bf16(const float* src, uint16_t* dst, int64_t n, cudaStream_t s) {
  const int grid = static_cast<int>(std::min<int64_t>((n + kThreads - 1) / kThreads, 4096));
  k_cast_bf16<<<grid > 0 ? grid : 1, kThreads, 0, s>>>(src, dst, n);
  return cudaGetLastError();
}

}  // namespace asap
