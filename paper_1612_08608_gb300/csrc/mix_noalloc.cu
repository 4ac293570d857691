// asap_mix_noalloc: the stochastic reduce with its consensus error, for
// callers that must not allocate device memory.
//
// Some callers cannot call cudaMalloc: a host framework that reserves
// (nearly) all of HBM for its own pool and tracks every byte, where an
// untracked cudaMalloc fails or breaks its budget; or a latency-critical
// loop, where cudaMalloc / cudaFree may synchronise the device and take an
// unbounded time.  The context API allocates its scratch at creation, so it
// does not suit them.  This entry point takes only caller-owned inputs and
// outputs.  Its one piece of scratch (a ticket counter and per-slab partial
// sums of the consensus error) is the file-scope array below, which every
// GPU that loads this library holds until the process exits.
//
// Compared with the context's reduce kernel it has no NOTIFY-ACK flags, at
// most 256 workers and the column means of its input, not its output (the
// weights need not be doubly stochastic); weights apply in row order.
//
// The kernel is bound by HBM: W is read and written once.  One CTA per SM
// walks column slabs (about 32 KB of all rows) that a producer warp brings into
// a ring of four stages by TMA (the tensor map is encoded on the host at each
// call and passed by value); two groups of eight warps mix alternate slabs.
// N = 32, d = 4 10^6, k = 2: 178 us, 5.7 TB/s; loaded slab by slab with plain
// loads, one slab in flight per CTA, 280 us.  A small call is launch latency: N =
// 8, d = 4,093 8.1 us, 9.5 us while a memset cleared the ticket before each
// launch (now the last CTA leaves it at zero).
//
// Every wait is time-limited.  A CTA in which one runs out stops mixing, waits
// (time-limited again) for its own copies in flight and turns the consensus
// error into NaN, the only word a call can pass on.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "asap_internal.h"

namespace asap {
void set_thread_error(const char* msg);
}

namespace {

using namespace asap;

constexpr int kNoAllocMaxN = 256;
constexpr int kNoAllocMaxSlabs = 32768;               // consensus partials: one per column slab
constexpr int kNoAllocTicketBytes = 256;
constexpr size_t kNoAllocScratchBytes = kNoAllocTicketBytes + 8u * kNoAllocMaxSlabs;   // 262,400 bytes
constexpr int kNoAllocMaxDevices = 64;

// [0, 256): ticket counters; [256, 256 + 8 * kNoAllocMaxSlabs): double
// partials, one per CTA.  (The largest ld that a call takes is 32,768 slabs of at
// most 16 KB: the partials were one per slab when it was set.)  Calls take
// kSlots slots of both in turn.  A call's last CTA leaves its own ticket at zero,
// and clears the one half the slots away: calls that overlapped against the
// rules (their stream order is the caller's business) cannot spoil more than the
// calls right after them.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kSlots = 32;
constexpr int kSlotPartials = kNoAllocMaxSlabs / kSlots;
constexpr int kStages = 4;
constexpr int kGroups = 2;                             // compute groups, on alternate slabs
constexpr int kGroupThreads = 256;
constexpr int kBlock = kGroups * kGroupThreads + 32;   // and the producer warp
constexpr size_t kSlabBytes = 32768;                   // at most
constexpr unsigned long long kWaitNs = 2000000000ull;  // a wait's limit: a TMA load never takes this long
static_assert(kStages % kGroups == 0, "a stage belongs to one group: its warps wait for each of its phases");

struct NoAllocArgs {
  float* out;
  int64_t ld;
  int N;
  int kp1;
  const int* nbr;
  const float* wgt;
  int S;           // slab width (columns), a power of two from 32 to 1024
  long long n_slabs;
  float* consensus_out;
  unsigned int* tickets;
  int slot;
  double* partial;
  unsigned long long wait_ns;
  long long drop_slab;   // tests: the slab whose copy is left out, so that its wait runs out (-1: none)
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(smem_u32(bar)), "r"(bytes)
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

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Time-limited wait on an mbarrier phase; false if the limit ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = now_ns();
  for (unsigned n = 1;; ++n) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((n & 255u) == 0 && now_ns() - t0 > limit_ns) return false;
  }
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      :: "r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void group_bar(int group) {
  asm volatile("bar.sync %0, %1;" :: "r"(group + 1), "n"(kGroupThreads) : "memory");
}

// The same barrier, which also returns the OR of `v` over the group.
__device__ __forceinline__ bool group_bar_or(int group, bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, %3, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r) : "r"(static_cast<uint32_t>(v)), "n"(kGroupThreads), "r"(group + 1) : "memory");
  return r != 0;
}

// Sums are carried as float-float pairs hi + lo in fp32 arithmetic (this
// GPU's fp64 pipe is narrow): the rounding error of each addition of the high
// parts is recovered exactly (Knuth's two-sum) and kept in lo.
struct Pair {
  float hi, lo;
};

__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
  const float s = a.hi + b.hi;
  const float bv = s - a.hi;
  const float e = ((a.hi - (s - bv)) + (b.hi - bv)) + (a.lo + b.lo);
  const float hi = s + e;
  return Pair{hi, e - (hi - s)};
}

// Sum over the block in a fixed order; valid in thread 0.
__device__ __forceinline__ Pair block_sum(Pair v, Pair* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = pair_add(v, Pair{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)});
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  Pair t{0.f, 0.f};
  if (threadIdx.x == 0)
    for (int w = 0; w < kBlock / 32; ++w) t = pair_add(t, red[w]);
  return t;
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

__device__ __forceinline__ float4 fma4(float w, float4 x, float4 c) {
  return make_float4(fmaf(w, x.x, c.x), fmaf(w, x.y, c.y), fmaf(w, x.z, c.z), fmaf(w, x.w, c.w));
}

// Shared memory: stages (1024-byte aligned), barriers, block-sum scratch, the
// groups' column sums, the mixing table.  noalloc_smem() mirrors it.
struct Smem {
  unsigned char* stage0;
  size_t stage_bytes;
  uint64_t *full, *empty;
  Pair* red;
  int* flag;
  float4* part;                       // [kGroups][kGroupThreads]
  int* nbr;                           // float4 offset of the neighbour's row within a column box
  float* wgt;
};

__host__ __device__ inline size_t noalloc_stage_bytes(int N, int S) {
  return (static_cast<size_t>(N) * S * 4 + 1023) & ~static_cast<size_t>(1023);
}

constexpr size_t kFixedSmem = 1024 + 16 * kStages + 8 * 32 + 16 + 16 * kGroups * kGroupThreads;

inline size_t noalloc_smem(int N, int S, int kp1) {
  return noalloc_stage_bytes(N, S) * kStages + kFixedSmem + 8 * static_cast<size_t>(N) * kp1;
}

__device__ __forceinline__ Smem carve(unsigned char* raw, const NoAllocArgs& a) {
  Smem m;
  size_t off = (1024u - (smem_u32(raw) & 1023u)) & 1023u;
  m.stage_bytes = noalloc_stage_bytes(a.N, a.S);
  m.stage0 = raw + off;
  off += m.stage_bytes * kStages;
  m.full = reinterpret_cast<uint64_t*>(raw + off);
  m.empty = m.full + kStages;
  off += 16 * kStages;
  m.red = reinterpret_cast<Pair*>(raw + off);
  off += 8 * 32;
  m.flag = reinterpret_cast<int*>(raw + off);
  off += 16;
  m.part = reinterpret_cast<float4*>(raw + off);
  off += 16 * kGroups * kGroupThreads;
  m.nbr = reinterpret_cast<int*>(raw + off);
  m.wgt = reinterpret_cast<float*>(raw + off + 4 * static_cast<size_t>(a.N) * a.kp1);
  return m;
}

// KP1 > 0: that many inputs per row; 0: a.kp1.
template <int KP1>
__global__ void __launch_bounds__(kBlock, 1) k_mix_noalloc(const __grid_constant__ CUtensorMap tmap,
                                                           const NoAllocArgs a) {
  extern __shared__ unsigned char smem_raw[];
  const Smem sm = carve(smem_raw, a);
  const int kp1 = KP1 > 0 ? KP1 : a.kp1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nq = a.S >> 2, lq = __ffs(nq) - 1;     // column quads of a slab
  const int QB = nq < 64 ? nq : 64;                // quads per TMA box row
  const int lqb = __ffs(QB) - 1;
  const int n_my = static_cast<int>((a.n_slabs - blockIdx.x + gridDim.x - 1) / gridDim.x);
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(sm.full + s, 1);
      mbar_init(sm.empty + s, kGroupThreads / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  Pair total{0.f, 0.f};
  bool failed = false;                             // a wait of this thread's (or its group's) ran out
  if (warp == kBlock / 32 - 1) {
    // ---- producer ----
    if (lane == 0) {
      int st = 0, it = 0;
      uint32_t ph = 1;                             // "empty" passes at once the first time round
      for (; it < n_my; ++it) {
        if (!mbar_wait(sm.empty + st, ph, a.wait_ns)) {
          failed = true;
          break;
        }
        const long long slab = blockIdx.x + static_cast<long long>(it) * gridDim.x, c0 = slab * a.S;
        mbar_expect_tx(sm.full + st, static_cast<uint32_t>(a.N) * a.S * 4u);
        for (int b = 0; b < nq / QB && slab != a.drop_slab; ++b)   // [column box][row][QB quads]
          tma_load_2d(sm.stage0 + st * sm.stage_bytes + static_cast<size_t>(b) * a.N * QB * 16, &tmap, sm.full + st,
                      static_cast<int>(c0 + b * QB * 4), 0);
        if (++st == kStages) {
          st = 0;
          ph ^= 1u;
        }
      }
      // The CTA's shared memory is given back with no copy in flight: the last
      // one into each stage has landed (as the groups see too, unless one gave up).
      for (int s = 0; s < kStages && s < it; ++s)
        failed = !mbar_wait(sm.full + s, static_cast<uint32_t>((it - 1 - s) / kStages) & 1u, a.wait_ns) || failed;
    }
    __syncwarp();
  } else {
    // ---- compute: thread gt of a group owns quad gt mod nq of the rows g, g + G, ... (g = gt / nq) ----
    for (int idx = tid; idx < a.N * kp1; idx += kGroups * kGroupThreads) {
      // Ids outside [0, N) are clamped so that a bad table cannot read
      // outside the slab; the caller must pass valid ids.
      sm.nbr[idx] = min(max(a.nbr[idx], 0), a.N - 1) << lqb;
      sm.wgt[idx] = a.wgt[idx];
    }
    asm volatile("bar.sync 3, %0;" :: "n"(kGroups * kGroupThreads) : "memory");
    const int group = tid / kGroupThreads, gt = tid - group * kGroupThreads;
    const int q = gt & (nq - 1), g = gt >> lq, G = kGroupThreads >> lq;
    const int qoff = (q >> lqb) * (a.N << lqb) + (q & (QB - 1));
    const float inv_n = 1.0f / static_cast<float>(a.N);
    float4* part = sm.part + group * kGroupThreads;
    int st = group;
    uint32_t ph = 0;
    for (int it = group; it < n_my; it += kGroups) {
      const bool landed = __all_sync(0xffffffffu, mbar_wait(sm.full + st, ph, a.wait_ns));
      const float4* x = reinterpret_cast<const float4*>(sm.stage0 + st * sm.stage_bytes) + qoff;
      // column means of the input
      float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int i = g; i < a.N; i += G) cs = add4(cs, x[i << lqb]);
      part[gt] = cs;
      // The group goes on or gives up as one: a warp that left alone would keep
      // the others at their next barrier for good.
      if (group_bar_or(group, !landed)) {
        failed = true;
        break;
      }
      cs = part[q];
      for (int u = 1; u < G; ++u) cs = add4(cs, part[(u << lq) + q]);
      const float4 mu = make_float4(cs.x * inv_n, cs.y * inv_n, cs.z * inv_n, cs.w * inv_n);
      const long long c = (blockIdx.x + static_cast<long long>(it) * gridDim.x) * a.S + 4 * q;
      float dev = 0.f;
      auto mix = [&](int i) {
        const int* nb = sm.nbr + i * kp1;
        const float* wt = sm.wgt + i * kp1;
        const float4 x0 = x[nb[0]];
        float4 acc = make_float4(wt[0] * x0.x, wt[0] * x0.y, wt[0] * x0.z, wt[0] * x0.w);
        if (KP1 > 0) {
#pragma unroll
          for (int m = 1; m < (KP1 > 0 ? KP1 : 1); ++m) acc = fma4(wt[m], x[nb[m]], acc);
        } else {
          for (int m = 1; m < kp1; ++m) acc = fma4(wt[m], x[nb[m]], acc);
        }
        return acc;
      };
      auto emit = [&](int i, float4 v) {
        const float dx = v.x - mu.x, dy = v.y - mu.y, dz = v.z - mu.z, dw = v.w - mu.w;
        dev = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, fmaf(dw, dw, dev))));
        if (c < a.ld) *reinterpret_cast<float4*>(a.out + static_cast<int64_t>(i) * a.ld + c) = v;
      };
      int i = g;
      for (; i + G < a.N; i += 2 * G) {            // two rows in flight
        const float4 v0 = mix(i), v1 = mix(i + G);
        emit(i, v0);
        emit(i + G, v1);
      }
      if (i < a.N) emit(i, mix(i));
      group_bar(group);                            // the column sums are read
      if (lane == 0) mbar_arrive(sm.empty + st);
      total = pair_add(total, Pair{dev, 0.f});
      st += kGroups;
      if (st >= kStages) {
        st = group;
        ph ^= 1u;
      }
    }
  }

  // The last CTA sums the partials in a fixed order (the result does not
  // depend on which CTA finishes last).
  if (failed) total = Pair{__int_as_float(0x7fc00000), 0.f};
  const Pair ps = block_sum(total, sm.red);
  if (tid == 0) {
    a.partial[blockIdx.x] = static_cast<double>(ps.hi) + static_cast<double>(ps.lo);
    __threadfence();
    sm.flag[0] = (atomicAdd(a.tickets + a.slot, 1u) == gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!sm.flag[0]) return;
  __threadfence();
  Pair v{0.f, 0.f};
  for (int b = tid; b < static_cast<int>(gridDim.x); b += kBlock) {
    const double p = __ldcg(a.partial + b);
    const float h = static_cast<float>(p);
    v = pair_add(v, Pair{h, static_cast<float>(p - static_cast<double>(h))});
  }
  const Pair sum = block_sum(v, sm.red);
  if (tid == 0) {
    const float c2 = sum.hi + sum.lo;
    a.consensus_out[0] = sqrtf(c2 < 0.f ? 0.f : c2);   // a NaN stays one
    a.tickets[a.slot] = 0u;
    a.tickets[(a.slot + kSlots / 2) % kSlots] = 0u;
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct DeviceSlot {
  void* scratch = nullptr;
  int sm_count = 0;
  unsigned calls = 0;              // calls on this device so far
  EncodeTiledFn encode = nullptr;
  unsigned long long ctx_id = 0;   // the CUDA context the address belongs to
};

// Unique id of the calling thread's current CUDA context (0: none current).
// A device reset, or a host framework that resets its primary context,
// reloads this library's module at a new address; the id tells the cached
// scratch address apart from a stale one.  The driver entry points are
// looked up through the runtime, so the library needs no link to libcuda.
unsigned long long current_context_id() {
  typedef CUresult (*GetCurrentFn)(CUcontext*);
  typedef CUresult (*GetIdFn)(CUcontext, unsigned long long*);
  static GetCurrentFn get_current = nullptr;
  static GetIdFn get_id = nullptr;
  static bool looked_up = false;
  if (!looked_up) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 4000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<GetCurrentFn>(p);
    p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<GetIdFn>(p);
    looked_up = true;
  }
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
    return 0;
  return id;
}

// The kernel's shared-memory limit on the current device: 227 KB.
template <int KP1>
bool allow_smem() {
  return cudaFuncSetAttribute(k_mix_noalloc<KP1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 << 10) !=
         cudaSuccess;
}

std::mutex g_noalloc_mu;
DeviceSlot g_noalloc_dev[kNoAllocMaxDevices];

asap_status reject(asap_status s, const char* msg) {
  set_thread_error(msg);
  return s;
}

asap_status mix_noalloc(const float* W_in, float* W_out, int N, int64_t d, int64_t ld, const int32_t* nbr,
                        const float* wgt, int kp1, float* consensus_out, void* cuda_stream,
                        unsigned long long wait_ns, long long drop_slab) {
  if (!W_in || !W_out || !nbr || !wgt || !consensus_out)
    return reject(ASAP_ERR_ARG, "asap_mix_noalloc: NULL pointer");
  if (N < 1 || N > kNoAllocMaxN) return reject(ASAP_ERR_ARG, "asap_mix_noalloc: need 1 <= N <= 256");
  if (kp1 < 1 || kp1 > kMaxKp1Sparse) return reject(ASAP_ERR_ARG, "asap_mix_noalloc: need 1 <= k+1 <= 32");
  if (d < 1 || ld < d || ld % 4 != 0)
    return reject(ASAP_ERR_ARG, "asap_mix_noalloc: need d >= 1, ld >= d and ld a multiple of 4");
  if ((reinterpret_cast<uintptr_t>(W_in) | reinterpret_cast<uintptr_t>(W_out)) & 15u)
    return reject(ASAP_ERR_ARG, "asap_mix_noalloc: W_in and W_out must be 16-byte aligned");
  {
    // ld is limited to 32,768 slabs of at most 16 KB.
    int S_max = 256;
    while (S_max > 4 && static_cast<size_t>(N) * S_max * 4 > 16384) S_max >>= 1;
    if ((ld + S_max - 1) / S_max > kNoAllocMaxSlabs)
      return reject(ASAP_ERR_ARG, "asap_mix_noalloc: ld beyond the range its scratch was laid out for "
                                  "(at most 32768 slabs of 256 columns for N <= 16, 16 columns for N = 256)");
  }
  {
    // Every CTA reads rows of W_in that other CTAs may already have written
    // to W_out: the two ranges must not overlap at all.
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(W_in), b0 = reinterpret_cast<uintptr_t>(W_out);
    const uintptr_t bytes = static_cast<uintptr_t>(N) * static_cast<uintptr_t>(ld) * sizeof(float);
    if (a0 < b0 + bytes && b0 < a0 + bytes)
      return reject(ASAP_ERR_ARG, "asap_mix_noalloc: W_in and W_out must not overlap");
  }

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices)
    return reject(ASAP_ERR_CUDA, "asap_mix_noalloc: no usable current device");
  DeviceSlot slot;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    DeviceSlot& ds = g_noalloc_dev[dev];
    const unsigned long long cur = current_context_id();
    if (!ds.scratch || cur == 0 || cur != ds.ctx_id) {
      // First call on this device (or in a new context of it): resolve the
      // device address of the file-scope scratch (the host-side name is only
      // a stand-in).  This also makes the device's primary context current.
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p)
        return reject(ASAP_ERR_CUDA, "asap_mix_noalloc: cudaGetSymbolAddress failed for the scratch array");
      int sms = 0;
      if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return reject(ASAP_ERR_CUDA, "asap_mix_noalloc: cannot query the SM count");
      void* enc = nullptr;
      cudaDriverEntryPointQueryResult q;
      if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &enc, 12000, cudaEnableDefault, &q) !=
              cudaSuccess ||
          q != cudaDriverEntryPointSuccess)
        return reject(ASAP_ERR_CUDA, "asap_mix_noalloc: cuTensorMapEncodeTiled is not available from the driver");
      if (allow_smem<0>() || allow_smem<2>() || allow_smem<3>() || allow_smem<5>())
        return reject(ASAP_ERR_CUDA, "asap_mix_noalloc: configuring the kernel failed");
      ds.encode = reinterpret_cast<EncodeTiledFn>(enc);
      ds.scratch = p;
      ds.sm_count = sms;
      ds.ctx_id = current_context_id();
    }
    slot = ds;
    ++ds.calls;
  }
  // Slab: S columns of all rows, at most 32 KB; narrower (down to 128-byte
  // rows) while that leaves SMs without two slabs, one for each group.
  int S = 1024;
  while (static_cast<size_t>(N) * S * 4 > kSlabBytes) S >>= 1;
  while (S > 32 && (ld + S - 1) / S < 2LL * slot.sm_count) S >>= 1;
  CUtensorMap tmap;
  {
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(ld), static_cast<cuuint64_t>(N)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * 4};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(std::min(S, 256)), static_cast<cuuint32_t>(N)};
    const cuuint32_t estr[2] = {1, 1};
    if (slot.encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(W_in), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return reject(ASAP_ERR_CUDA, "asap_mix_noalloc: cuTensorMapEncodeTiled failed");
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  unsigned char* base = static_cast<unsigned char*>(slot.scratch);
  NoAllocArgs a;
  a.out = W_out;
  a.ld = ld;
  a.N = N;
  a.kp1 = kp1;
  a.nbr = nbr;
  a.wgt = wgt;
  a.S = S;
  a.n_slabs = (ld + S - 1) / S;
  a.consensus_out = consensus_out;
  a.tickets = reinterpret_cast<unsigned int*>(base);
  a.slot = static_cast<int>(slot.calls % kSlots);
  a.wait_ns = wait_ns;
  a.drop_slab = drop_slab;
  a.partial = reinterpret_cast<double*>(base + kNoAllocTicketBytes) + static_cast<size_t>(a.slot) * kSlotPartials;
  const size_t smem = noalloc_smem(N, S, kp1);
  const int grid = static_cast<int>(std::min<long long>(a.n_slabs, std::min(slot.sm_count, kSlotPartials)));
  switch (kp1) {
    case 2: k_mix_noalloc<2><<<grid, kBlock, smem, s>>>(tmap, a); break;
    case 3: k_mix_noalloc<3><<<grid, kBlock, smem, s>>>(tmap, a); break;
    case 5: k_mix_noalloc<5><<<grid, kBlock, smem, s>>>(tmap, a); break;
    default: k_mix_noalloc<0><<<grid, kBlock, smem, s>>>(tmap, a); break;
  }
  if (cudaGetLastError() != cudaSuccess) return reject(ASAP_ERR_CUDA, "asap_mix_noalloc: launch failed");
  return ASAP_OK;
}

}  // namespace

extern "C" asap_status asap_mix_noalloc(const float* W_in, float* W_out, int N, int64_t d, int64_t ld,
                                        const int32_t* nbr, const float* wgt, int kp1, float* consensus_out,
                                        void* cuda_stream) {
  return mix_noalloc(W_in, W_out, N, d, ld, nbr, wgt, kp1, consensus_out, cuda_stream, kWaitNs, -1);
}

extern "C" asap_status asap_debug_mix_noalloc(const float* W_in, float* W_out, int N, int64_t d, int64_t ld,
                                              const int32_t* nbr, const float* wgt, int kp1, float* consensus_out,
                                              void* cuda_stream, uint64_t wait_ns, int64_t drop_slab) {
  if (wait_ns == 0) return reject(ASAP_ERR_ARG, "asap_debug_mix_noalloc: need wait_ns > 0");
  return mix_noalloc(W_in, W_out, N, d, ld, nbr, wgt, kp1, consensus_out, cuda_stream, wait_ns, drop_slab);
}
