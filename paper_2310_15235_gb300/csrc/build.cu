// Radiation tree build on the GPU (TREVR2, Sec. 2.3 and Sec. 2.6):
// FP64 normalisation + 63-bit Morton keys, a stable sort, bisection level by
// level (a node splits while it holds more than `bucket` elements; empty
// halves become empty leaves), and a bottom-up pass for the summed luminosity
// per band, the centre of luminosity (one band-summed centre per cell), B =
// largest centre-to-corner distance (Sec. 2.5.2) and the bucket absorption
// sum(kappa m)/V_box (Sec. 2.6).  Sums run in FP64 and are rounded once to FP32
// for the walk.
//
// Small and middle trees were bound by launches and read-backs, not by the
// kernels: the levels' sizes went to the host one by one.  The whole build is
// now eight launches and one read-back.  Whole steps, with the pool below and the
// walk of few receivers by blocks: 33k elements 2.21 -> 0.87 ms, 4k 1.45 -> 0.41,
// 2.1M and a 1000-receiver rung 5.96 -> 2.78.
#include <cuda.h>

#include <atomic>
#include <climits>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>
#include <string>

#include "internal.cuh"

namespace trevr2 {

// ---------------------------------------------------------------------------
// Errors
static thread_local char g_err[512];

void set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}

// The pool of the entry point that runs on this thread, once it has looked it up.
static thread_local cudaMemPool_t g_call_pool;

void clear_error() {
  g_err[0] = 0;
  g_call_pool = nullptr;
}

static std::atomic<unsigned long long> g_launches{0};
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

int cuda_fail(cudaError_t e, const char* what) {
  set_error("%s failed: %s", what, cudaGetErrorString(e));
  cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? TREVR2_ENOMEM : TREVR2_ECUDA;
}

// ---------------------------------------------------------------------------
// Device allocations, and the failures a test can ask for (testing aids).
static std::atomic<int64_t> g_fail_alloc_after{-1};   // -1: off
static std::atomic<int> g_source_stack_cap{0};        // 0: off
static std::atomic<uint32_t> g_barrier_polls{kBarrierSpins};
static std::atomic<int> g_cell_cap{INT_MAX}, g_team_hits{INT_MAX};

// True for the one allocation a test asked to fail (then off again).
static bool injected_alloc_failure() {
  int64_t v = g_fail_alloc_after.load();
  while (v >= 0)
    if (g_fail_alloc_after.compare_exchange_weak(v, v - 1)) return v == 0;
  return false;
}

// The library's memory pool of the current device.  The default pool gives
// every freed byte back at the next synchronisation, so that each step's trees
// were mapped anew (about 0.4 ms of a 4k-element step, 1 ms of a 2.1M one); this
// one keeps up to kPoolKeep free bytes (a 2.1M-element tree with its tables and
// walk buffers; 0.7 % of the card), and gives them back when an allocation
// fails.
constexpr uint64_t kPoolKeep = uint64_t(2) << 30;
constexpr int kMaxDevices = 64;

// The driver's ids of contexts, which no later context gets again.
struct ContextIds {
  CUresult (*current)(CUcontext*) = nullptr;
  CUresult (*id)(CUcontext, unsigned long long*) = nullptr;
  CUresult (*retain)(CUcontext*, CUdevice) = nullptr;
  CUresult (*release)(CUdevice) = nullptr;
  template <class F>
  static bool find(const char* name, int version, F* fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion(name, &p, version, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return false;
    }
    *fn = reinterpret_cast<F>(p);
    return true;
  }
  bool known;
  ContextIds()
      : known(find("cuCtxGetCurrent", 4000, &current) && find("cuCtxGetId", 12000, &id) &&
              find("cuDevicePrimaryCtxRetain", 7000, &retain) &&
              find("cuDevicePrimaryCtxRelease", 11000, &release)) {}
  // 0 where there is none
  unsigned long long of_thread() const {
    CUcontext ctx = nullptr;
    unsigned long long v = 0;
    if (!known || current(&ctx) != CUDA_SUCCESS || !ctx || id(ctx, &v) != CUDA_SUCCESS) return 0;
    return v;
  }
  unsigned long long of_primary(int dev) const {
    CUcontext ctx = nullptr;
    unsigned long long v = 0;
    if (!known || retain(&ctx, dev) != CUDA_SUCCESS) return 0;
    if (id(ctx, &v) != CUDA_SUCCESS) v = 0;
    release(dev);
    return v;
  }
};

// The pool outlives a reset of the device's (primary) context, with the blocks it
// keeps (CUDA 13.0: the handle stays good, 1 GiB kept stays reserved), but nothing
// says that blocks mapped before may be used after: a pool is used in the
// context it was made in, and replaced after a reset.  Checked by the first
// allocation of every entry point (each of a build's thirty cost 0.3 us): by the
// thread's current context where that was seen before, else by the primary
// context itself.
static int library_pool(cudaMemPool_t* pool) {
  if (g_call_pool) {
    *pool = g_call_pool;
    return TREVR2_OK;
  }
  struct Kept {
    cudaMemPool_t pool = nullptr;
    unsigned long long primary = 0, seen = 0;
  };
  static std::mutex lock;
  static Kept kept[kMaxDevices];
  static const ContextIds ids;
  int dev = 0;
  T2_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    T2_CUDA(cudaDeviceGetDefaultMemPool(pool, dev));
    return TREVR2_OK;
  }
  std::lock_guard<std::mutex> hold(lock);
  Kept& k = kept[dev];
  unsigned long long now = ids.of_thread();
  if (!k.pool || !now || now != k.seen) {
    T2_CUDA(cudaFree(nullptr));  // the runtime's context, current to this thread
    now = ids.of_thread();
    const unsigned long long primary = ids.of_primary(dev);
    if (k.pool && primary != k.primary) {
      if (cudaMemPoolDestroy(k.pool) != cudaSuccess) cudaGetLastError();
      k.pool = nullptr;
    }
    k.primary = primary;
    k.seen = now;
  }
  if (!k.pool) {
    cudaMemPoolProps props;
    std::memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t fresh = nullptr;
    T2_CUDA(cudaMemPoolCreate(&fresh, &props));
    uint64_t keep = kPoolKeep;
    const cudaError_t e = cudaMemPoolSetAttribute(fresh, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(fresh);
      return cuda_fail(e, "cudaMemPoolSetAttribute");
    }
    k.pool = fresh;
  }
  *pool = g_call_pool = k.pool;
  return TREVR2_OK;
}

int device_alloc(void** p, size_t bytes, cudaStream_t st, const char* what) {
  *p = nullptr;
  if (injected_alloc_failure()) {
    set_error("%s of %zu bytes failed: out of memory (failure requested by "
              "trevr2_debug_set)", what, bytes);
    return TREVR2_ENOMEM;
  }
  cudaMemPool_t pool = nullptr;
  T2_CHECK(library_pool(&pool));
  cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, st);
  if (e == cudaErrorMemoryAllocation) {  // give back what the pool keeps, and try once more
    cudaGetLastError();
    cudaMemPoolTrimTo(pool, 0);
    e = cudaMallocFromPoolAsync(p, bytes, pool, st);
  }
  if (e != cudaSuccess) {
    *p = nullptr;
    cudaGetLastError();
    set_error("%s of %zu bytes failed: %s", what, bytes, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? TREVR2_ENOMEM : TREVR2_ECUDA;
  }
  return TREVR2_OK;
}

int debug_source_stack_cap() { return g_source_stack_cap.load(); }
uint32_t barrier_polls() { return g_barrier_polls.load(); }
int debug_cell_cap() { return g_cell_cap.load(); }
int debug_team_hits() { return g_team_hits.load(); }

// ---------------------------------------------------------------------------
// Exclusive scan (block scan of 2048 values + recursive scan of block sums).
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 2 * kScanThreads;

__global__ void k_scan_block(int* d, int64_t n, int* block_sums) {
  __shared__ int s[kScanItems];
  const int64_t base = int64_t(blockIdx.x) * kScanItems;
  const int t = threadIdx.x;
  int64_t i0 = base + 2 * t, i1 = i0 + 1;
  int a = i0 < n ? d[i0] : 0;
  int b = i1 < n ? d[i1] : 0;
  s[2 * t] = a;
  s[2 * t + 1] = b;
  // Blelloch up-sweep / down-sweep
  int offset = 1;
  for (int w = kScanItems >> 1; w > 0; w >>= 1) {
    __syncthreads();
    if (t < w) {
      int ai = offset * (2 * t + 1) - 1, bi = offset * (2 * t + 2) - 1;
      s[bi] += s[ai];
    }
    offset <<= 1;
  }
  __syncthreads();
  if (t == 0) {
    if (block_sums) block_sums[blockIdx.x] = s[kScanItems - 1];
    s[kScanItems - 1] = 0;
  }
  for (int w = 1; w < kScanItems; w <<= 1) {
    offset >>= 1;
    __syncthreads();
    if (t < w) {
      int ai = offset * (2 * t + 1) - 1, bi = offset * (2 * t + 2) - 1;
      int tmp = s[ai];
      s[ai] = s[bi];
      s[bi] += tmp;
    }
  }
  __syncthreads();
  if (i0 < n) d[i0] = s[2 * t];
  if (i1 < n) d[i1] = s[2 * t + 1];
}

__global__ void k_scan_add(int* d, int64_t n, const int* block_offsets) {
  const int64_t base = int64_t(blockIdx.x) * kScanItems;
  int add = block_offsets[blockIdx.x];
  for (int k = threadIdx.x; k < kScanItems; k += blockDim.x) {
    int64_t i = base + k;
    if (i < n) d[i] += add;
  }
}

__global__ void k_scan_total(const int* scanned, const int* orig_last, int64_t n, int* total) {
  *total = n ? scanned[n - 1] + *orig_last : 0;
}

__global__ void k_copy_last(const int* d, int64_t n, int* out) { *out = n ? d[n - 1] : 0; }

size_t scan_ws_ints(int64_t n) {
  const int64_t nblocks = (n + kScanItems - 1) / kScanItems;
  return 1 + (nblocks > 1 ? size_t(nblocks) + scan_ws_ints(nblocks) : 0);
}

// ws: the last input value, then the block sums of each recursion level.
int scan_exclusive_i32(int* d, int64_t n, int* d_total, cudaStream_t st, int* ws) {
  int* last = ws;
  k_copy_last<<<1, 1, 0, st>>>(d, n, last); note_launch();
  if (n > 0) {
    int64_t nblocks = (n + kScanItems - 1) / kScanItems;
    if (nblocks == 1) {
      k_scan_block<<<1, kScanThreads, 0, st>>>(d, n, nullptr); note_launch();
    } else {
      int* sums = ws + 1;
      k_scan_block<<<unsigned(nblocks), kScanThreads, 0, st>>>(d, n, sums); note_launch();
      T2_CHECK(scan_exclusive_i32(sums, nblocks, nullptr, st, sums + nblocks));
      k_scan_add<<<unsigned(nblocks), 256, 0, st>>>(d, n, sums); note_launch();
    }
  }
  if (d_total) k_scan_total<<<1, 1, 0, st>>>(d, last, n, d_total); note_launch();
  T2_CUDA(cudaGetLastError());
  return TREVR2_OK;
}

// ---------------------------------------------------------------------------
// Stable sort of 64-bit keys with a 32-bit payload.
//
// Up to kSmallSort keys: one block, a merge sort in shared memory, every key
// finding its place in the neighbouring run by a binary search (4097 keys: 56
// us by itself and cold; a bitonic network's 91 steps took 1.7 times as long),
// bound by shared-memory loads.  More: one cooperative
// launch does every pass of an LSD radix sort (8 bits a pass), with a grid
// barrier where a pass needs all blocks' counts or keys: a launch for each
// step of each pass left the GPU idle between them for longer than the steps
// took (33k elements: 47 launches; now 1).
constexpr int kSmallSort = 8192;
constexpr int kSmallSortThreads = 1024;

// With `active`, the receivers' order: the keys are their elements' sorted
// positions (N for an index outside [0, N)), the payload their slots.
__global__ void __launch_bounds__(kSmallSortThreads)
    k_sort_small(uint64_t* keys, int* vals, int n, const int64_t* __restrict__ active,
                 const int* __restrict__ inv, int64_t N) {
  extern __shared__ uint64_t sort_smem[];
  uint64_t *ka = sort_smem, *kb = ka + n;
  uint16_t *pa = reinterpret_cast<uint16_t*>(kb + n), *pb = pa + n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    uint64_t key;
    if (active) {
      const int64_t io = active[i];
      key = io >= 0 && io < N ? uint64_t(inv[io]) : uint64_t(N);
    } else {
      key = keys[i];
    }
    ka[i] = key;
    pa[i] = uint16_t(i);
  }
  for (int run = 1; run < n; run <<= 1) {
    __syncthreads();
    // four keys a thread at a time, their searches side by side
    for (int i0 = threadIdx.x; i0 < n; i0 += 4 * blockDim.x) {
      uint64_t key[4];
      int lo[4], hi[4];
      bool left[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = min(i0 + u * int(blockDim.x), n - 1);
        key[u] = ka[i];
        left[u] = (i & run) == 0;
        // the other run; its equal keys go before a right one, after a left one
        const int first = left[u] ? (i & ~(run - 1)) + run : (i & ~(2 * run - 1));
        lo[u] = min(first, n);
        hi[u] = min(first + run, n);
      }
      for (int len = run; len > 0; len >>= 1)  // the last half steps are empty for some
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (lo[u] < hi[u]) {
            const int mid = (lo[u] + hi[u]) >> 1;
            const uint64_t other = ka[mid];
            if (left[u] ? other < key[u] : other <= key[u]) lo[u] = mid + 1; else hi[u] = mid;
          }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * int(blockDim.x);
        if (i >= n) break;
        const int first = left[u] ? (i & ~(run - 1)) + run : (i & ~(2 * run - 1));
        const int at = left[u] ? i + lo[u] - min(first, n) : i - run + lo[u] - first;
        kb[at] = key[u];
        pb[at] = pa[i];
      }
    }
    uint64_t* const tk = ka;
    ka = kb;
    kb = tk;
    uint16_t* const tp = pa;
    pa = pb;
    pb = tp;
  }
  __syncthreads();
  // the payload is permuted in place: read by everybody before it is written
  int v[kSmallSort / kSmallSortThreads];
#pragma unroll
  for (int r = 0; r < kSmallSort / kSmallSortThreads; ++r) {
    const int i = threadIdx.x + r * blockDim.x;
    if (i < n) v[r] = active ? int(pa[i]) : vals[pa[i]];
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSmallSort / kSmallSortThreads; ++r) {
    const int i = threadIdx.x + r * blockDim.x;
    if (i < n) {
      keys[i] = ka[i];
      vals[i] = v[r];
    }
  }
}

// One block per chunk of consecutive keys.  A pass counts the chunk's digits,
// waits for all blocks, places its own digits after those of smaller digits
// and earlier blocks, and scatters 512 keys a round: warps rank their lanes
// with __match_any_sync and per-warp digit counts, so equal digits keep their
// order.  Keys are read past the L1, which other blocks' writes do not reach.
constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;

__global__ void __launch_bounds__(kSortThreads)
    k_radix_sort(uint64_t* ka, int* va, uint64_t* kb, int* vb, int64_t n, int passes, int* hist,
                 uint32_t* bar, uint32_t* status, uint32_t polls) {
  __shared__ int base[256];
  __shared__ int wh[kSortWarps][256];
  __shared__ int tot2[2][256], bef2[2][256];
  __shared__ int wsum[8];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, nb = gridDim.x, b = blockIdx.x;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t per = (n + nb - 1) / nb;
  const int64_t lo = min(n, b * per), hi = min(n, lo + per);
  for (int pass = 0; pass < passes; ++pass) {
    const int shift = 8 * pass;
    if (t < 256) base[t] = 0;
    __syncthreads();
    for (int64_t i = lo + t; i < hi; i += kSortThreads)
      atomicAdd(&base[(__ldcg(ka + i) >> shift) & 255u], 1);
    __syncthreads();
    if (t < 256) __stcg(hist + b * 256 + t, base[t]);
    if (!grid_barrier(bar, nb, status, polls)) return;
    {
      const int d = t & 255, h = t >> 8;
      int tot = 0, bef = 0;
      for (int o = h; o < nb; o += 2) {
        const int c = __ldcg(hist + o * 256 + d);
        tot += c;
        if (o < b) bef += c;
      }
      tot2[h][d] = tot;
      bef2[h][d] = bef;
    }
    __syncthreads();
    int run = 0, mine = 0;
    if (t < 256) {  // exclusive scan of the digits' totals
      mine = tot2[0][t] + tot2[1][t];
      run = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, run, o);
        if (lane >= o) run += u;
      }
      if (lane == 31) wsum[warp] = run;
    }
    __syncthreads();
    if (t < 256) {
      for (int w = 0; w < warp; ++w) run += wsum[w];
      base[t] = run - mine + bef2[0][t] + bef2[1][t];
    }
    for (int64_t r0 = lo; r0 < hi; r0 += kSortThreads) {
#pragma unroll
      for (int w = 0; w < kSortWarps * 256; w += kSortThreads) (&wh[0][0])[w + t] = 0;
      __syncthreads();
      const int64_t i = r0 + t;
      const bool valid = i < hi;
      const uint64_t key = valid ? __ldcg(ka + i) : 0;
      const int val = valid ? __ldcg(va + i) : 0;
      const int digit = valid ? int((key >> shift) & 255u) : 256;
      const unsigned peers = __match_any_sync(0xffffffffu, digit);
      const int intra = __popc(peers & lt);
      if (valid && intra == 0) wh[warp][digit] = __popc(peers);
      __syncthreads();
      if (t < 256) {
        int at = base[t];
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
          const int c = wh[w][t];
          wh[w][t] = at;
          at += c;
        }
        base[t] = at;
      }
      __syncthreads();
      if (valid) {
        const int dst = wh[warp][digit] + intra;
        __stcg(kb + dst, key);
        __stcg(vb + dst, val);
      }
      __syncthreads();
    }
    uint64_t* const tk = ka;
    ka = kb;
    kb = tk;
    int* const tv = va;
    va = vb;
    vb = tv;
    if (!grid_barrier(bar, nb, status, polls)) return;
  }
}

// SMs of the stream's green context, 0 where it has none (or the driver does
// not know them): a stream of one runs on some of the device's SMs, and a
// cooperative launch sized by the device could not be resident there at once.
static int green_context_sms(cudaStream_t st) {
  using GetCtx = CUresult (*)(CUstream, CUcontext*, CUgreenCtx*);
  using GetResource = CUresult (*)(CUgreenCtx, CUdevResource*, CUdevResourceType);
  struct Entry {
    GetCtx ctx = nullptr;
    GetResource resource = nullptr;
    Entry() {
      cudaDriverEntryPointQueryResult found;
      void *c = nullptr, *r = nullptr;
      if (cudaGetDriverEntryPointByVersion("cuStreamGetCtx", &c, 12050, cudaEnableDefault, &found) ==
              cudaSuccess && found == cudaDriverEntryPointSuccess &&
          cudaGetDriverEntryPointByVersion("cuGreenCtxGetDevResource", &r, 12040, cudaEnableDefault,
                                           &found) == cudaSuccess &&
          found == cudaDriverEntryPointSuccess) {
        ctx = reinterpret_cast<GetCtx>(c);
        resource = reinterpret_cast<GetResource>(r);
      } else {
        cudaGetLastError();
      }
    }
  };
  static const Entry entry;
  if (!entry.ctx) return 0;
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  if (entry.ctx(st, &ctx, &green) != CUDA_SUCCESS || !green) return 0;
  CUdevResource r;
  std::memset(&r, 0, sizeof(r));
  if (entry.resource(green, &r, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS) return 0;
  return int(r.sm.smCount);
}

int coop_blocks(int64_t work, int64_t per_block, int per_sm, cudaStream_t st, int* out) {
  int dev = 0, sms = 0;
  T2_CUDA(cudaGetDevice(&dev));
  T2_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (const int green = green_context_sms(st)) sms = std::min(sms, green);
  const int64_t most = std::min<int64_t>(int64_t(sms) * per_sm, kMaxCoopBlocks);
  *out = int(std::max<int64_t>(1, std::min<int64_t>(most, (work + per_block - 1) / per_block)));
  return TREVR2_OK;
}

constexpr int64_t kSortPerBlock = 2048;

static int64_t sort_blocks_bound(int64_t n) {
  return std::min<int64_t>(kMaxCoopBlocks, std::max<int64_t>(1, (n + kSortPerBlock - 1) / kSortPerBlock));
}

size_t radix_ws_bytes(int64_t n) {
  if (n <= kSmallSort) return 256;
  auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
  return up(sizeof(uint64_t) * size_t(n)) + up(sizeof(int) * size_t(n)) +
         up(sizeof(int) * 256 * size_t(sort_blocks_bound(n))) + 256;
}

static int sort_small(uint64_t* keys, int* vals, int n, cudaStream_t st, const int64_t* active,
                      const int* inv, int64_t N) {
  const size_t smem = size_t(n) * 2 * (sizeof(uint64_t) + sizeof(uint16_t)) + 8;
  T2_CUDA(cudaFuncSetAttribute(k_sort_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               kSmallSort * 20 + 8));
  // at most kSmallSort / kSmallSortThreads keys a thread
  const int threads = std::min(kSmallSortThreads, (n + 31) & ~31);
  k_sort_small<<<1, threads, smem, st>>>(keys, vals, n, active, inv, N);
  note_launch();
  T2_CUDA(cudaGetLastError());
  return TREVR2_OK;
}

__global__ void k_order_keys(const int64_t* __restrict__ active, int64_t A, int64_t N,
                             const int* __restrict__ inv, uint64_t* __restrict__ keys,
                             int* __restrict__ slots) {
  const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= A) return;
  const int64_t io = active[i];
  keys[i] = (io >= 0 && io < N) ? uint64_t(inv[io]) : uint64_t(N);
  slots[i] = int(i);
}

int order_receivers(const Tree* t, const int64_t* active, int64_t A, uint64_t* keys, int* slots,
                    cudaStream_t st) {
  if (A <= kSmallSort) return sort_small(keys, slots, int(A), st, active, t->inv, t->N);
  k_order_keys<<<unsigned((A + 255) / 256), 256, 0, st>>>(active, A, t->N, t->inv, keys, slots);
  note_launch();
  int bits = 1;
  while ((int64_t(1) << bits) <= t->N) ++bits;
  return radix_sort_u64_i32(keys, slots, A, st, t->status, bits);
}

int radix_sort_u64_i32(uint64_t* keys, int* vals, int64_t n, cudaStream_t st, uint32_t* status,
                       int key_bits, void* ws) {
  if (n <= 1) return TREVR2_OK;
  if (n <= kSmallSort) return sort_small(keys, vals, int(n), st, nullptr, nullptr, 0);
  // an even number of 8-bit passes, so the result ends in the caller's buffers
  int passes = (std::min(std::max(key_bits, 1), 64) + 7) / 8;
  passes += passes & 1;
  DeviceTemp<char> own(st);
  if (!ws) {
    T2_CHECK(device_alloc(reinterpret_cast<void**>(&own.p), radix_ws_bytes(n), st, "sort workspace"));
    ws = own.p;
  }
  int nb = 0;
  T2_CHECK(coop_blocks(n, kSortPerBlock, 1, st, &nb));
  auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
  char* p = static_cast<char*>(ws);
  uint64_t* k2 = reinterpret_cast<uint64_t*>(p);
  p += up(sizeof(uint64_t) * size_t(n));
  int* v2 = reinterpret_cast<int*>(p);
  p += up(sizeof(int) * size_t(n));
  int* hist = reinterpret_cast<int*>(p);
  p += up(sizeof(int) * 256 * size_t(sort_blocks_bound(n)));
  uint32_t* bar = reinterpret_cast<uint32_t*>(p);
  T2_CUDA(cudaMemsetAsync(bar, 0, sizeof(uint32_t), st));
  uint32_t polls = barrier_polls();
  void* args[] = {&keys, &vals, &k2, &v2, &n, &passes, &hist, &bar, &status, &polls};
  T2_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_radix_sort), dim3(unsigned(nb)),
                                      dim3(kSortThreads), args, 0, st));
  note_launch();
  return TREVR2_OK;
}

// ---------------------------------------------------------------------------
// Input validation and bounds.
// What the build's kernels find out and the host reads once at the end.
constexpr int kMaxLevels = kMaxDepth + 2;
struct BuildState {
  double lo[3];      // root cube
  double size;
  float h_default;   // (V_root / N_gas)^(1/3), used without h
  int n_luminous;
  int n_nodes, n_internal, levels;
  int need;          // nodes that did not fit (0: all did)
  int level_begin[kMaxLevels + 1];
  unsigned long long n_gas;
  unsigned int tickets;
  uint32_t bar;      // grid barrier of the tree kernel
};

// Checks the inputs (status bits) and, from the last block done, the root
// cube: the explicit one, or the bounding cube of the positions.
__global__ void __launch_bounds__(256)
    k_validate(const double* __restrict__ pos, const float* __restrict__ mass,
               const float* __restrict__ kappa, const float* __restrict__ lum,
               const float* __restrict__ h, int64_t N, int nb, bool explicit_box, double lo0,
               double lo1, double lo2, double box_size, double* partial /*[grid][6]*/,
               BuildState* S, uint32_t* status) {
  __shared__ double smin[3][256], smax[3][256];
  __shared__ bool last;
  double mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
  bool bad = false;
  int gas = 0;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < N;
       i += int64_t(gridDim.x) * blockDim.x) {
    for (int a = 0; a < 3; ++a) {
      double x = pos[3 * i + a];
      bad |= !isfinite(x);
      mn[a] = fmin(mn[a], x);
      mx[a] = fmax(mx[a], x);
    }
    float m = mass[i];
    bad |= !(m >= 0.0f) || !isfinite(m);
    gas += m > 0.0f;
    if (h) bad |= !(h[i] > 0.0f) || !isfinite(h[i]);
    for (int b = 0; b < nb; ++b) {
      float k = kappa[i * nb + b], l = lum[i * nb + b];
      bad |= !(k >= 0.0f) || !isfinite(k) || !(l >= 0.0f) || !isfinite(l);
    }
  }
  if (bad) atomicOr(status, kStatusBadInput);
  gas = __reduce_add_sync(0xffffffffu, gas);
  if ((threadIdx.x & 31) == 0 && gas) atomicAdd(&S->n_gas, (unsigned long long)(gas));
  auto reduce = [&]() {
    for (int a = 0; a < 3; ++a) {
      smin[a][threadIdx.x] = mn[a];
      smax[a][threadIdx.x] = mx[a];
    }
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if (threadIdx.x < w)
        for (int a = 0; a < 3; ++a) {
          smin[a][threadIdx.x] = fmin(smin[a][threadIdx.x], smin[a][threadIdx.x + w]);
          smax[a][threadIdx.x] = fmax(smax[a][threadIdx.x], smax[a][threadIdx.x + w]);
        }
      __syncthreads();
    }
  };
  reduce();
  if (threadIdx.x == 0) {
    for (int a = 0; a < 3; ++a) {
      __stcg(partial + 6 * blockIdx.x + a, smin[a][0]);
      __stcg(partial + 6 * blockIdx.x + 3 + a, smax[a][0]);
    }
    __threadfence();
    last = atomicAdd(&S->tickets, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int a = 0; a < 3; ++a) {
    mn[a] = INFINITY;
    mx[a] = -INFINITY;
  }
  for (int b = threadIdx.x; b < gridDim.x; b += blockDim.x)
    for (int a = 0; a < 3; ++a) {
      mn[a] = fmin(mn[a], __ldcg(partial + 6 * b + a));
      mx[a] = fmax(mx[a], __ldcg(partial + 6 * b + 3 + a));
    }
  reduce();
  if (threadIdx.x != 0) return;
  double lo[3] = {lo0, lo1, lo2}, size = box_size;
  if (explicit_box) {
    for (int a = 0; a < 3; ++a)
      if (N > 0 && (smin[a][0] < lo[a] || smax[a][0] > lo[a] + box_size))
        atomicOr(status, kStatusOutsideBox);
  } else {
    double ext = 0.0;
    for (int a = 0; a < 3; ++a) {
      lo[a] = N > 0 ? smin[a][0] : 0.0;
      if (N > 0) ext = fmax(ext, smax[a][0] - smin[a][0]);
    }
    size = ext > 0.0 ? ext : 1.0;
  }
  for (int a = 0; a < 3; ++a) S->lo[a] = lo[a];
  S->size = size;
  const unsigned long long g = atomicAdd(&S->n_gas, 0ull);
  S->h_default = float(cbrt(size * size * size / double(g ? g : 1ull)));
}

// Sec. 2.3: normalise in FP64 and interleave the 21-bit cell indices,
// bit 62 = x MSB, then y, then z.
__device__ inline uint64_t spread3(uint64_t v) {
  v &= 0x1fffffull;
  v = (v | (v << 32)) & 0x1f00000000ffffull;
  v = (v | (v << 16)) & 0x1f0000ff0000ffull;
  v = (v | (v << 8)) & 0x100f00f00f00f00full;
  v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
  v = (v | (v << 2)) & 0x1249249249249249ull;
  return v;
}

// (x - lo) / size, exactly as the division rounds it: a product where 1 / size
// is a power of two (then both are exact).
__device__ __forceinline__ double normalised(double x, double lo, double size, double inv,
                                             bool exact_inv) {
  const double d = __dsub_rn(x, lo);
  return exact_inv ? d * inv : __ddiv_rn(d, size);
}
__device__ __forceinline__ bool power_of_two(double size) {
  const long long bits = __double_as_longlong(size);
  const int e = int((bits >> 52) & 0x7ff);
  return (bits & 0xfffffffffffffll) == 0 && e > 1 && e < 0x7fd;
}

__global__ void k_morton(const double* __restrict__ pos, int64_t N,
                         const BuildState* __restrict__ S, uint64_t* __restrict__ keys,
                         int* __restrict__ vals) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= N) return;
  const double lo[3] = {S->lo[0], S->lo[1], S->lo[2]}, size = S->size;
  const bool p2 = power_of_two(size);
  const double inv = p2 ? 1.0 / size : 0.0;
  uint64_t k[3];
  for (int a = 0; a < 3; ++a) {
    double u = normalised(pos[3 * i + a], lo[a], size, inv, p2);
    double f = floor(__dmul_rn(u, 2097152.0));
    f = fmin(fmax(f, 0.0), 2097151.0);
    k[a] = uint64_t(f);
  }
  keys[i] = (spread3(k[0]) << 2) | (spread3(k[1]) << 1) | spread3(k[2]);
  vals[i] = int(i);
}

// Sorted element data used by the walk.
__global__ void k_gather_elements(const double* __restrict__ pos, const float* __restrict__ mass,
                                  const float* __restrict__ kappa, const float* __restrict__ lum,
                                  const float* __restrict__ h, const int* __restrict__ perm,
                                  int64_t N, int nb, int nbp, BuildState* __restrict__ S,
                                  int* __restrict__ inv,
                                  double* __restrict__ pos64, float4* __restrict__ pos32,
                                  float* __restrict__ Lelem, float* __restrict__ km,
                                  float* __restrict__ hn, float* __restrict__ ms) {
  int64_t s = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (s >= N) return;
  int i = perm[s];
  inv[i] = int(s);
  const double lo[3] = {S->lo[0], S->lo[1], S->lo[2]}, size = S->size;
  const bool p2 = power_of_two(size);
  const double isize = p2 ? 1.0 / size : 0.0;
  double u[3];
  for (int a = 0; a < 3; ++a) {
    u[a] = normalised(pos[3 * int64_t(i) + a], lo[a], size, isize, p2);
    pos64[3 * s + a] = u[a];
  }
  double lt = 0.0;
  for (int b = 0; b < nbp; ++b) {
    float l = b < nb ? lum[int64_t(i) * nb + b] : 0.0f;
    float k = b < nb ? kappa[int64_t(i) * nb + b] : 0.0f;
    Lelem[s * nbp + b] = l;
    km[s * nbp + b] = k * mass[i];
    lt = __dadd_rn(lt, double(l));
  }
  pos32[s] = make_float4(float(u[0]), float(u[1]), float(u[2]), float(lt));
  const double hh = double(h ? h[i] : S->h_default);
  hn[s] = float(p2 ? hh * isize : hh / size);
  ms[s] = mass[i];
  const unsigned lit = __ballot_sync(__activemask(), lt > 0.0);
  if (lt > 0.0 && (lit & ((1u << (threadIdx.x & 31)) - 1u)) == 0u)
    atomicAdd(&S->n_luminous, __popc(lit));
}

// ---------------------------------------------------------------------------
// Level-by-level bisection and the bottom-up aggregates.  A launch per level,
// with the host reading each level's size, cost more than the work (33k
// elements: 80 launches and 13 synchronisations; now 3 and none).
// Topology, one cooperative launch: block 0 alone while levels are small (block barriers
// only); from then on every block takes a chunk of consecutive nodes of the
// level, counts its splits, and after a grid barrier places its children
// behind those of the blocks before it.  A node splits while it holds more
// than `bucket` elements; nodes are numbered by depth, by prefix within a
// depth.  Aggregates: the leaves' sums at once, then in one cooperative launch
// the internal nodes' (additions only), deepest depth first; runs of small
// depths stay in block 0; then every node's centre, B and record at once.
// Values another block wrote are read past the L1.
struct TreeArgs {
  const uint64_t* keys;
  int64_t N;
  int bucket, nb, nbp;
  int cap;            // nodes the arrays hold
  uint64_t* prefix;
  int* depth;
  int* first;
  int* count;
  int* child;
  int* parent;
  int* int_index;
  int* mid;           // [cap] a splitting node's first upper element, else -1
  int* block_count;   // [blocks]
  const double* pos64;
  const float* Lelem;
  const int* perm;
  const float* kappa;
  const float* mass;
  double* L64;        // [cap][4]
  double* cs64;       // [cap][4] sum Lt x, sum Lt
  uint32_t* flags;    // [cap]
  float* Lnode;
  float4* csrc;
  double* c64;
  double* B64;
  float* alpha_leaf;
  uint32_t* lmask;
  NodeW* nodes;
  BuildState* S;
  uint32_t* status;
  uint32_t polls;     // of a grid barrier
};
constexpr int kTreeThreads = 512;
constexpr int kSmallLevel = 1024;  // nodes of a level that block 0 does alone

// The element that starts the upper half of a node, or -1 when it is a leaf.
__device__ __forceinline__ int split_at(const TreeArgs& A, int d, int f, int c) {
  if (!(c > A.bucket && d < kMaxDepth)) return -1;
  // keys in [f, f+c) share the node's prefix, so bit (62 - d) is monotone
  const int bit = kMaxDepth - 1 - d;
  int lo = f, hi = f + c;  // first index with the bit set
  while (lo < hi) {
    const int m = lo + ((hi - lo) >> 1);
    if ((A.keys[m] >> bit) & 1ull) hi = m; else lo = m + 1;
  }
  return lo;
}

// The same for one node by a whole warp: 32 probes a step instead of one.
__device__ __forceinline__ int split_at_warp(const TreeArgs& A, int d, int f, int c) {
  if (!(c > A.bucket && d < kMaxDepth)) return -1;
  const int bit = kMaxDepth - 1 - d, lane = threadIdx.x & 31;
  int lo = f, hi = f + c;  // first index with the bit set lies in [lo, hi]
  while (lo < hi) {
    const int step = (hi - lo + 31) >> 5;
    const int at = lo + lane * step;  // probes lo, lo + step, ...
    const bool set = at >= hi || ((A.keys[at] >> bit) & 1ull);
    const unsigned m = __ballot_sync(0xffffffffu, set);
    if (m & 1u) return lo;
    const int k = m ? __ffs(m) - 1 : 32;  // clear at probe k - 1, set at probe k
    hi = min(hi, lo + k * step);
    lo = lo + (k - 1) * step + 1;
  }
  return lo;
}

__device__ __forceinline__ void emit_halves(const TreeArgs& A, int q, int c, int d, int f, int n,
                                            int m) {
  const uint64_t p = __ldcg(A.prefix + q);
  A.child[q] = c;
  A.prefix[c] = p;
  A.prefix[c + 1] = p | (1ull << (kMaxDepth - 1 - d));
  A.depth[c] = A.depth[c + 1] = d + 1;
  A.first[c] = f;
  A.count[c] = m - f;
  A.first[c + 1] = m;
  A.count[c + 1] = f + n - m;
  A.parent[c] = A.parent[c + 1] = q;
}

// Running rank of the set flags of a block, in thread order: this thread's
// rank in the tile, the tile's total to `total`.
__device__ __forceinline__ int tile_rank(bool flag, int& total) {
  __shared__ int warp_sum[kTreeThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned m = __ballot_sync(0xffffffffu, flag);
  __syncthreads();
  if (lane == 0) warp_sum[warp] = __popc(m);
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kTreeThreads / 32; ++w) {
    const int c = warp_sum[w];
    before += w < warp ? c : 0;
    all += c;
  }
  total = all;
  return before + __popc(m & ((1u << lane) - 1u));
}

// The sums of a leaf's elements: luminosity per band, L-weighted position and
// total, bucket absorption; whether it absorbs or shines.
__device__ __forceinline__ void leaf_sums(const TreeArgs& A, int64_t q, double inv_size2) {
  const int nb = A.nb, nbp = A.nbp;
  const int f = A.first[q], n = A.count[q];
  double Lb[4] = {0, 0, 0, 0}, kmb[4] = {0, 0, 0, 0}, cs[4] = {0, 0, 0, 0};
  uint32_t has = 0, lit = 0;
  for (int e = f; e < f + n; ++e) {
    double lt = 0.0;
    const int i = A.perm[e];
    const double m = double(A.mass[i]);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      if (b >= nb) break;
      const double l = double(A.Lelem[int64_t(e) * nbp + b]);
      Lb[b] = __dadd_rn(Lb[b], l);
      lt = __dadd_rn(lt, l);
      // kappa and m are float32: their FP64 product is exact
      kmb[b] = __dadd_rn(kmb[b], __dmul_rn(double(A.kappa[int64_t(i) * nb + b]), m));
    }
    if (lt > 0.0) {  // else it adds zeros
#pragma unroll
      for (int a = 0; a < 3; ++a) cs[a] = __dadd_rn(cs[a], __dmul_rn(lt, A.pos64[3 * int64_t(e) + a]));
      cs[3] = __dadd_rn(cs[3], lt);
      if (e - f < 32) lit |= 1u << (e - f);
    }
  }
  // 1 / V: V = 2^-depth, so the product is exact
  const double iV = __longlong_as_double((long long)(1023 + A.depth[q]) << 52);
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    if (b < nbp) {
      const double al = b < nb ? kmb[b] * iV * inv_size2 : 0.0;
      A.alpha_leaf[q * nbp + b] = float(al);
      if (al > 0.0) has |= kMetaHasAlpha;
    }
    A.L64[q * 4 + b] = b < nb ? Lb[b] : 0.0;
    A.cs64[q * 4 + b] = cs[b];
  }
  if (cs[3] > 0.0) has |= kMetaHasL;
  A.flags[q] = has;
  A.lmask[q] = lit;
}

// The sums of an internal node from its halves'.
__device__ __forceinline__ void inner_sums(const TreeArgs& A, int64_t q) {
  const int64_t c = __ldcg(A.child + q);
  if (c < 0) return;
  const double2* L = reinterpret_cast<const double2*>(A.L64 + 4 * c);
  const double2* s = reinterpret_cast<const double2*>(A.cs64 + 4 * c);
  const uint32_t h0 = __ldcg(A.flags + c), h1 = __ldcg(A.flags + c + 1);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double2 l0 = __ldcg(L + i), l1 = __ldcg(L + 2 + i);
    const double2 s0 = __ldcg(s + i), s1 = __ldcg(s + 2 + i);
    __stcg(reinterpret_cast<double2*>(A.L64 + 4 * q) + i,
           make_double2(__dadd_rn(l0.x, l1.x), __dadd_rn(l0.y, l1.y)));
    __stcg(reinterpret_cast<double2*>(A.cs64 + 4 * q) + i,
           make_double2(__dadd_rn(s0.x, s1.x), __dadd_rn(s0.y, s1.y)));
  }
  // (a cell shines if a half does: luminosities are not negative)
  uint32_t has = (h0 | h1) & (kMetaHasAlpha | kMetaHasL);
  if (h0 & kMetaHasAlpha) has |= kMetaChild0Alpha;
  if (h1 & kMetaHasAlpha) has |= kMetaChild1Alpha;
  __stcg(A.flags + q, has);
}

// Every other bit triple of a 63-bit key from bit `shift` on: one axis's 21 bits.
__device__ __forceinline__ uint32_t compact3(uint64_t v, int shift) {
  v = (v >> shift) & 0x1249249249249249ull;
  v = (v ^ (v >> 2)) & 0x10c30c30c30c30c3ull;
  v = (v ^ (v >> 4)) & 0x100f00f00f00f00full;
  v = (v ^ (v >> 8)) & 0x1f0000ff0000ffull;
  v = (v ^ (v >> 16)) & 0x1f00000000ffffull;
  v = (v ^ (v >> 32)) & 0x1fffffull;
  return uint32_t(v);
}

// A node's record, centre and B from its sums: independent of other nodes.
__device__ __forceinline__ void finish_node(const TreeArgs& A, int64_t q) {
  const int nbp = A.nbp;
  const int d = A.depth[q], c = A.child[q];
  const uint64_t prefix = A.prefix[q];
  const uint32_t has = A.flags[q];
  const double cs3 = A.cs64[q * 4 + 3];
  double lo[3], cc[3], B2 = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = double(compact3(prefix, 2 - a)) * (1.0 / 2097152.0);
    const double ext = __longlong_as_double((long long)(1023 - splits_on_axis(d, a)) << 52);
    cc[a] = cs3 > 0.0 ? A.cs64[q * 4 + a] / cs3 : lo[a] + 0.5 * ext;
    // B: the farthest box corner from the centre of luminosity (Sec. 2.5.2),
    // the farther face on each axis
    const double d0 = __dsub_rn(lo[a], cc[a]), d1 = __dsub_rn(lo[a] + ext, cc[a]);
    B2 = __dadd_rn(B2, fmax(__dmul_rn(d0, d0), __dmul_rn(d1, d1)));
    A.c64[3 * q + a] = cc[a];
  }
  const double B = sqrt(B2);
  A.B64[q] = B;
  for (int b = 0; b < nbp; ++b) A.Lnode[q * nbp + b] = float(A.L64[q * 4 + b]);
  A.csrc[q] = make_float4(float(cc[0]), float(cc[1]), float(cc[2]), float(cs3));
  if (c >= 0) {
    A.lmask[q] = 0;
    for (int b = 0; b < nbp; ++b) A.alpha_leaf[q * nbp + b] = 0.0f;
  }
  NodeW w;
  w.lo[0] = float(lo[0]);
  w.lo[1] = float(lo[1]);
  w.lo[2] = float(lo[2]);
  w.B = float(B);
  w.child = c;
  w.aux = c < 0 ? A.first[q] : A.int_index[q];
  w.count = A.count[q];
  w.meta = uint32_t(d) | (uint32_t(d % 3) << kMetaAxisShift) | (c < 0 ? kMetaLeaf : 0u) | has;
  A.nodes[q] = w;
}

// Refused inputs, or a sort or topology that gave up at a barrier: the kernels
// that follow do nothing.  They would read what was not written, or spend the
// time of a build (and of one thread adding up a leaf of everything, when all
// positions are clamped to one corner: 1M elements 634 ms, now 0.45) on a refusal.
__device__ __forceinline__ bool build_stopped(const TreeArgs& A) {
  return __ldcg(A.status) != 0u;
}

__global__ void __launch_bounds__(kTreeThreads) k_build_tree(const __grid_constant__ TreeArgs A) {
  BuildState* S = A.S;
  const int blocks = gridDim.x, t = threadIdx.x;
  __shared__ int s_levels, s_lb, s_le, s_int, s_need;
  if (build_stopped(A)) return;
  int lb = 0, le = 1, level = 0, n_int = 0;
  int need = 0;
  if (blockIdx.x == 0) {
    if (t == 0) {
      A.prefix[0] = 0;
      A.depth[0] = 0;
      A.first[0] = 0;
      A.count[0] = int(A.N);
      A.parent[0] = -1;
      S->level_begin[0] = 0;
    }
    __syncthreads();
    // small levels, one after another
    while (le - lb <= kSmallLevel) {
      int done = 0;  // splits so far in this level
      for (int q0 = lb; q0 < le; q0 += kTreeThreads) {
        const int q = q0 + t;
        int m = -1, d = 0, f = 0, c = 0;
        if (q < le) {
          d = level;
          f = __ldcg(A.first + q);
          c = __ldcg(A.count + q);
        }
        if (le - lb <= 4 * kTreeThreads / 32) {  // few nodes, long searches: a warp each
          __shared__ int s_mid[4 * kTreeThreads / 32];
          for (int i = t >> 5; i < le - lb; i += kTreeThreads / 32) {
            const int at = split_at_warp(A, level, __ldcg(A.first + lb + i), __ldcg(A.count + lb + i));
            if ((t & 31) == 0) s_mid[i] = at;
          }
          __syncthreads();
          if (q < le) m = s_mid[t];
        } else if (q < le) {
          m = split_at(A, d, f, c);
        }
        int tile = 0;
        const int rank = done + tile_rank(m >= 0, tile);
        if (le + 2 * (done + tile) > A.cap) {
          need = le + 2 * (le - lb);
          break;
        }
        if (m >= 0) {
          emit_halves(A, q, le + 2 * rank, d, f, c, m);
          A.int_index[q] = n_int + rank;
        } else if (q < le) {
          A.child[q] = -1;
          A.int_index[q] = -1;
        }
        done += tile;
      }
      __syncthreads();  // the children are visible to this block
      if (need) break;
      if (t == 0) S->level_begin[level + 1] = le;
      n_int += done;
      lb = le;
      le += 2 * done;
      ++level;
      if (done == 0) break;
    }
    if (t == 0) {
      S->levels = level;
      S->n_internal = n_int;
      S->n_nodes = le;
      S->need = need;
      A.block_count[0] = lb;  // what the other blocks go on from
      A.block_count[1] = le;
    }
  }
  if (!grid_barrier(&S->bar, blocks, A.status, A.polls)) return;
  if (t == 0) {
    s_levels = __ldcg(&S->levels);
    s_int = __ldcg(&S->n_internal);
    s_need = __ldcg(&S->need);
    s_lb = __ldcg(A.block_count);
    s_le = __ldcg(A.block_count + 1);
  }
  __syncthreads();
  level = s_levels;
  n_int = s_int;
  need = s_need;
  lb = s_lb;
  le = s_le;
  if (need) return;
  if (!grid_barrier(&S->bar, blocks, A.status, A.polls)) return;  // block_count is free again
  // larger levels, all blocks
  while (le > lb) {
    const int per = (le - lb + blocks - 1) / blocks;
    const int c0 = min(le, lb + int(blockIdx.x) * per), c1 = min(le, c0 + per);
    int mine = 0;
    for (int q0 = c0; q0 < c1; q0 += kTreeThreads) {
      const int q = q0 + t;
      int m = -1;
      if (q < c1) {
        m = split_at(A, level, __ldcg(A.first + q), __ldcg(A.count + q));
        A.mid[q] = m;
      }
      mine += __syncthreads_count(m >= 0);
    }
    if (t == 0) __stcg(A.block_count + blockIdx.x, mine);
    if (!grid_barrier(&S->bar, blocks, A.status, A.polls)) return;
    int before = 0, all = 0;
    {
      __shared__ int s_before, s_all;
      if (t < 32) {
        for (int b = t; b < blocks; b += 32) {
          const int c = __ldcg(A.block_count + b);
          all += c;
          if (b < int(blockIdx.x)) before += c;
        }
        all = __reduce_add_sync(0xffffffffu, all);
        before = __reduce_add_sync(0xffffffffu, before);
        if (t == 0) {
          s_before = before;
          s_all = all;
        }
      }
      __syncthreads();
      before = s_before;
      all = s_all;
    }
    if (int64_t(le) + 2 * int64_t(all) > A.cap) {
      if (blockIdx.x == 0 && t == 0)
        S->need = int(min(int64_t(INT32_MAX), int64_t(le) + 2 * int64_t(all)));
      return;
    }
    for (int q0 = c0; q0 < c1; q0 += kTreeThreads) {
      const int q = q0 + t;
      const int m = q < c1 ? A.mid[q] : -1;
      int tile = 0;
      const int rank = before + tile_rank(m >= 0, tile);
      if (m >= 0) {
        emit_halves(A, q, le + 2 * rank, level, __ldcg(A.first + q), __ldcg(A.count + q), m);
        A.int_index[q] = n_int + rank;
      } else if (q < c1) {
        A.child[q] = -1;
        A.int_index[q] = -1;
      }
      before += tile;
    }
    if (blockIdx.x == 0 && t == 0) S->level_begin[level + 1] = le;
    n_int += all;
    lb = le;
    le += 2 * all;
    ++level;
    if (!grid_barrier(&S->bar, blocks, A.status, A.polls)) return;
    if (all == 0) break;
  }
  if (blockIdx.x == 0 && t == 0) {
    S->levels = level;
    S->n_internal = n_int;
    S->n_nodes = le;
  }
}

// The leaves' aggregates (the grid covers the nodes' arrays; how many there
// are is known on the device).
__global__ void __launch_bounds__(128) k_aggregate_leaves(const __grid_constant__ TreeArgs A) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (build_stopped(A) || A.S->need || q >= A.S->n_nodes || A.child[q] >= 0) return;
  const double size = A.S->size;
  leaf_sums(A, q, 1.0 / (size * size));
}

__global__ void __launch_bounds__(128) k_finish_nodes(const __grid_constant__ TreeArgs A) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (build_stopped(A) || A.S->need || q >= A.S->n_nodes) return;
  finish_node(A, q);
}

__global__ void __launch_bounds__(kTreeThreads, 2) k_sum_levels(const __grid_constant__ TreeArgs A) {
  BuildState* S = A.S;
  if (build_stopped(A) || S->need) return;
  const int blocks = gridDim.x, t = threadIdx.x;
  __shared__ int s_begin[kMaxLevels + 1];
  const int level = S->levels;
  for (int i = t; i < level; i += kTreeThreads) s_begin[i] = S->level_begin[i];
  if (t == 0) s_begin[level] = S->n_nodes;
  __syncthreads();
  const int64_t stride = int64_t(blocks) * kTreeThreads, at = int64_t(blockIdx.x) * kTreeThreads + t;
  bool together = false;  // whether the depth below was done by all blocks
  for (int d = level - 2; d >= 0; --d) {
    const int b0 = s_begin[d], b1 = s_begin[d + 1];
    const bool small = b1 - b0 <= kTreeThreads;
    if (together || (!small && d < level - 2)) {
      if (!grid_barrier(&S->bar, blocks, A.status, A.polls)) return;
    } else {
      __syncthreads();
    }
    together = !small;
    if (small) {
      if (blockIdx.x == 0 && t < b1 - b0) inner_sums(A, b0 + t);
    } else {
      for (int64_t q = b0 + at; q < b1; q += stride) inner_sums(A, q);
    }
  }
}

// The node arrays for `cap` nodes.
static int alloc_nodes(Tree* t, int64_t cap, cudaStream_t st) {
  const int nbp = t->nbp;
  T2_CHECK(dalloc(&t->prefix, 4 * cap, st));  // the topology arrays, in one piece
  t->depth = reinterpret_cast<int*>(t->prefix + cap);
  t->first = t->depth + cap;
  t->count = t->first + cap;
  t->child = t->count + cap;
  t->parent = t->child + cap;
  t->int_index = t->parent + cap;
  T2_CHECK(dalloc(&t->nodes, cap, st));
  T2_CHECK(dalloc(&t->Lnode, cap * nbp, st));
  T2_CHECK(dalloc(&t->csrc, cap, st));
  T2_CHECK(dalloc(&t->c64, 3 * cap, st));
  T2_CHECK(dalloc(&t->B64, cap, st));
  T2_CHECK(dalloc(&t->alpha_leaf, cap * nbp, st));
  T2_CHECK(dalloc(&t->lmask, cap, st));
  return TREVR2_OK;
}

static void free_nodes(Tree* t, cudaStream_t st) {
  dfree(t->prefix, st);
  t->depth = t->first = t->count = t->child = t->parent = t->int_index = nullptr;
  dfree(t->nodes, st);
  dfree(t->Lnode, st);
  dfree(t->csrc, st);
  dfree(t->c64, st);
  dfree(t->B64, st);
  dfree(t->alpha_leaf, st);
  dfree(t->lmask, st);
}

static void free_tree(Tree* t, cudaStream_t st) {
  dfree(t->keys, st);
  dfree(t->perm, st);
  dfree(t->inv, st);
  dfree(t->pos64, st);
  dfree(t->pos32, st);
  dfree(t->Lelem, st);
  dfree(t->km, st);
  dfree(t->mass, st);
  dfree(t->hn, st);
  free_nodes(t, st);
  dfree(t->dtau, st);
  dfree(t->nodes_refined, st);
  for (Table& tb : t->tables) free_table(&tb, st);
  t->tables.clear();
  if (t->scratch) cudaFreeAsync(t->scratch, st);
  t->scratch = nullptr;
  if (t->order_buf) cudaFreeAsync(t->order_buf, st);
  t->order_buf = nullptr;
  dfree(t->status, st);
  dfree(t->counter, st);
}

static inline unsigned blocks_for(int64_t n, int threads) {
  return unsigned((n + threads - 1) / threads);
}

// Everything up to the one read-back is enqueued without waiting: the inputs'
// check, the root cube, keys and sort run whatever the inputs hold (keys are
// clamped to the cube), the tree's kernels return at once where they were
// refused, and the host looks at the status and the sizes at the end.
static int build_impl(Tree* t, const double* pos, const float* mass, const float* kappa,
                      const float* lum, const float* h, const double* box_lo, double box_size,
                      cudaStream_t st) {
  const int64_t N = t->N;
  const int nb = t->nb, nbp = t->nbp;
  T2_CHECK(dalloc(&t->status, 2, st));  // status word, grid barrier of the tables' kernel
  T2_CHECK(dalloc(&t->counter, 1, st));
  T2_CUDA(cudaMemsetAsync(t->status, 0, sizeof(uint32_t), st));

  // 1. validation and root cube
  const int vblocks = int(std::min<int64_t>(std::max<int64_t>(blocks_for(N, 256), 1), 1024));
  DeviceTemp<double> partial(st);
  DeviceTemp<BuildState> state(st);
  T2_CHECK(dalloc(&partial.p, size_t(vblocks) * 6, st));
  T2_CHECK(dalloc(&state.p, 1, st));
  T2_CUDA(cudaMemsetAsync(state.p, 0, sizeof(BuildState), st));
  const bool explicit_box = box_lo && box_size > 0.0;
  const double lo[3] = {explicit_box ? box_lo[0] : 0.0, explicit_box ? box_lo[1] : 0.0,
                        explicit_box ? box_lo[2] : 0.0};
  k_validate<<<vblocks, 256, 0, st>>>(pos, mass, kappa, lum, h, N, nb, explicit_box, lo[0], lo[1],
                                      lo[2], box_size, partial.p, state.p, t->status);
  note_launch();

  // 2. keys and stable sort
  T2_CHECK(dalloc(&t->keys, N, st));
  T2_CHECK(dalloc(&t->perm, N, st));
  if (N > 0) {
    k_morton<<<blocks_for(N, 256), 256, 0, st>>>(pos, N, state.p, t->keys, t->perm);
    note_launch();
  }
  T2_CHECK(radix_sort_u64_i32(t->keys, t->perm, N, st, t->status));

  // 3. sorted element data
  T2_CHECK(dalloc(&t->inv, N, st));
  T2_CHECK(dalloc(&t->pos64, 3 * N, st));
  T2_CHECK(dalloc(&t->pos32, N, st));
  T2_CHECK(dalloc(&t->Lelem, N * nbp, st));
  T2_CHECK(dalloc(&t->km, N * nbp, st));
  T2_CHECK(dalloc(&t->hn, N, st));
  T2_CHECK(dalloc(&t->mass, N, st));
  if (N > 0) {
    k_gather_elements<<<blocks_for(N, 256), 256, 0, st>>>(pos, mass, kappa, lum, h, t->perm, N, nb,
                                                          nbp, state.p, t->inv, t->pos64, t->pos32,
                                                          t->Lelem, t->km, t->hn, t->mass);
    note_launch();
  }

  // 4. bisection and aggregates, into arrays sized for a tree of evenly filled
  // leaves; once more with larger ones when the tree has more nodes
  BuildState S;
  int64_t cap = std::min<int64_t>(std::max<int64_t>(1024, 4 * (N / std::max(t->bucket, 1)) + 64),
                                  INT32_MAX);
  for (;;) {
    T2_CHECK(alloc_nodes(t, cap, st));
    DeviceTemp<double> sums(st);
    DeviceTemp<int> ints(st);
    T2_CHECK(dalloc(&sums.p, 8 * cap, st));
    T2_CHECK(dalloc(&ints.p, 2 * cap + kMaxCoopBlocks, st));
    TreeArgs A;
    A.keys = t->keys;
    A.N = N;
    A.bucket = t->bucket;
    A.nb = nb;
    A.nbp = nbp;
    A.cap = int(cap);
    A.prefix = t->prefix;
    A.depth = t->depth;
    A.first = t->first;
    A.count = t->count;
    A.child = t->child;
    A.parent = t->parent;
    A.int_index = t->int_index;
    A.mid = ints.p;
    A.flags = reinterpret_cast<uint32_t*>(ints.p + cap);
    A.block_count = ints.p + 2 * cap;
    A.pos64 = t->pos64;
    A.Lelem = t->Lelem;
    A.perm = t->perm;
    A.kappa = kappa;
    A.mass = mass;
    A.L64 = sums.p;
    A.cs64 = sums.p + 4 * cap;
    A.Lnode = t->Lnode;
    A.csrc = t->csrc;
    A.c64 = t->c64;
    A.B64 = t->B64;
    A.alpha_leaf = t->alpha_leaf;
    A.lmask = t->lmask;
    A.nodes = t->nodes;
    A.S = state.p;
    A.status = t->status;
    A.polls = barrier_polls();
    int blocks = 0, blocks_inner = 0;
    T2_CHECK(coop_blocks(cap, 2 * kTreeThreads, 1, st, &blocks));
    T2_CHECK(coop_blocks(cap, kTreeThreads, 2, st, &blocks_inner));
    void* args[] = {&A};
    T2_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_build_tree),
                                        dim3(unsigned(blocks)), dim3(kTreeThreads), args, 0, st));
    note_launch();
    k_aggregate_leaves<<<blocks_for(cap, 128), 128, 0, st>>>(A);
    note_launch();
    T2_CUDA(cudaMemsetAsync(&state.p->bar, 0, sizeof(uint32_t), st));
    T2_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_sum_levels),
                                        dim3(unsigned(blocks_inner)), dim3(kTreeThreads), args, 0, st));
    note_launch();
    k_finish_nodes<<<blocks_for(cap, 128), 128, 0, st>>>(A);
    note_launch();
    uint32_t hstatus = 0;
    T2_CUDA(cudaMemcpyAsync(&S, state.p, sizeof(S), cudaMemcpyDeviceToHost, st));
    T2_CUDA(cudaMemcpyAsync(&hstatus, t->status, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    T2_CUDA(cudaStreamSynchronize(st));
    if (hstatus & kStatusBadInput) {
      set_error("trevr2_build: non-finite position, or negative/non-finite mass, kappa, lum or h");
      return TREVR2_EINVAL;
    }
    if (hstatus & kStatusOutsideBox) {
      set_error("trevr2_build: a position lies outside the given root cube");
      return TREVR2_EINVAL;
    }
    if (hstatus) {
      set_error("trevr2_build: a grid barrier gave up waiting (device status 0x%x)", hstatus);
      return TREVR2_ETIMEOUT;
    }
    if (S.need == 0) break;
    if (cap >= INT32_MAX) {
      set_error("trevr2_build: more than 2^31 nodes");
      return TREVR2_EUNSUPPORTED;
    }
    free_nodes(t, st);
    cap = std::min<int64_t>(std::max<int64_t>(2 * cap, S.need), INT32_MAX);
    T2_CUDA(cudaMemsetAsync(&state.p->bar, 0, sizeof(uint32_t), st));
    T2_CUDA(cudaMemsetAsync(&state.p->need, 0, sizeof(int), st));
  }
  for (int a = 0; a < 3; ++a) t->lo[a] = S.lo[a];
  t->size = S.size;
  t->n_nodes = S.n_nodes;
  t->max_depth = S.levels - 1;
  t->level_begin.assign(S.level_begin, S.level_begin + S.levels);
  t->level_begin.push_back(S.n_nodes);
  t->n_internal = S.n_internal;
  t->n_luminous = S.n_luminous;
  return TREVR2_OK;
}

}  // namespace trevr2

using namespace trevr2;

extern "C" {

const char* trevr2_last_error(void) { return g_err; }

int trevr2_debug_set(int what, int64_t value) {
  clear_error();
  switch (what) {
    case TREVR2_DEBUG_FAIL_ALLOC:
      if (value < -1) break;
      g_fail_alloc_after.store(value);
      return TREVR2_OK;
    case TREVR2_DEBUG_SOURCE_STACK:
      if (value < 0 || value > (int64_t(1) << 30)) break;
      g_source_stack_cap.store(int(value));
      return TREVR2_OK;
    case TREVR2_DEBUG_BARRIER_POLLS:
      if (value < 0 || value > int64_t(kBarrierSpins)) break;
      g_barrier_polls.store(value ? uint32_t(value) : kBarrierSpins);
      return TREVR2_OK;
    case TREVR2_DEBUG_CELL_CAP:  // (the buffers behind the list are 16-byte aligned)
      if (value < 0 || value > (1 << 20) || value % 32 != 0) break;
      g_cell_cap.store(value ? int(value) : INT_MAX);
      return TREVR2_OK;
    case TREVR2_DEBUG_TEAM_HITS:
      if (value < 0 || value > (1 << 20)) break;
      g_team_hits.store(value ? int(value) : INT_MAX);
      return TREVR2_OK;
    default:
      break;
  }
  set_error("trevr2_debug_set: unknown setting %d or value %lld out of range", what,
            static_cast<long long>(value));
  return TREVR2_EINVAL;
}

int trevr2_debug_pool_used(uint64_t* bytes) {
  clear_error();
  if (!bytes) {
    set_error("trevr2_debug_pool_used: bytes is NULL");
    return TREVR2_EINVAL;
  }
  T2_CUDA(cudaDeviceSynchronize());
  cudaMemPool_t pool = nullptr;
  T2_CHECK(library_pool(&pool));
  uint64_t used = 0;
  T2_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used));
  *bytes = uint64_t(used);
  return TREVR2_OK;
}

uint64_t trevr2_kernel_launches(void) { return g_launches.load(std::memory_order_relaxed); }

int trevr2_build(const double* pos, const float* mass, const float* kappa, const float* lum,
                 const float* h, int64_t N, int nb, const double* box_lo, double box_size,
                 int bucket, void* stream, trevr2_tree** out) {
  clear_error();
  if (!out) {
    set_error("trevr2_build: out is NULL");
    return TREVR2_EINVAL;
  }
  *out = nullptr;
  if (N < 0 || (N > 0 && (!pos || !mass || !kappa || !lum))) {
    set_error("trevr2_build: N < 0 or a NULL input array");
    return TREVR2_EINVAL;
  }
  if (N >= (int64_t(1) << 31)) {
    set_error("trevr2_build: N must be below 2^31");
    return TREVR2_EUNSUPPORTED;
  }
  if (nb < 1 || nb > TREVR2_MAX_BANDS) {
    set_error("trevr2_build: nb = %d outside [1, %d]", nb, TREVR2_MAX_BANDS);
    return nb < 1 ? TREVR2_EINVAL : TREVR2_EUNSUPPORTED;
  }
  if (bucket < 1 || bucket > 4096) {
    set_error("trevr2_build: bucket = %d outside [1, 4096]", bucket);
    return TREVR2_EINVAL;
  }
  if (box_lo && box_size > 0.0) {
    for (int a = 0; a < 3; ++a)
      if (!std::isfinite(box_lo[a])) {
        set_error("trevr2_build: non-finite box_lo");
        return TREVR2_EINVAL;
      }
    if (!std::isfinite(box_size)) {
      set_error("trevr2_build: non-finite box_size");
      return TREVR2_EINVAL;
    }
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Tree* t = new (std::nothrow) Tree();
  if (!t) {
    set_error("trevr2_build: host allocation failed");
    return TREVR2_ENOMEM;
  }
  t->N = N;
  t->nb = nb;
  t->nbp = nbp_of(nb);
  t->bucket = bucket;
  t->has_h = h != nullptr;
  t->last_stream = st;
  int rc;
  try {
    rc = build_impl(t, pos, mass, kappa, lum, h, box_lo, box_size, st);
  } catch (const std::bad_alloc&) {
    set_error("trevr2_build: host allocation failed");
    rc = TREVR2_ENOMEM;
  }
  if (rc != TREVR2_OK) {
    std::string msg = g_err;
    free_tree(t, st);
    delete t;
    set_error("%s", msg.c_str());
    return rc;
  }
  *out = reinterpret_cast<trevr2_tree*>(t);
  return TREVR2_OK;
}

int trevr2_free(trevr2_tree* tree) {
  clear_error();
  if (!tree) return TREVR2_OK;
  Tree* t = reinterpret_cast<Tree*>(tree);
  free_tree(t, t->last_stream);
  delete t;
  return TREVR2_OK;
}

int trevr2_tree_info_get(const trevr2_tree* tree, trevr2_tree_info* info) {
  clear_error();
  if (!tree || !info) {
    set_error("trevr2_tree_info_get: NULL argument");
    return TREVR2_EINVAL;
  }
  const Tree* t = reinterpret_cast<const Tree*>(tree);
  info->n_elements = t->N;
  info->n_nodes = t->n_nodes;
  info->n_internal = t->n_internal;
  info->n_leaves = t->n_nodes - t->n_internal;
  info->nb = t->nb;
  info->bucket = t->bucket;
  info->max_depth = t->max_depth;
  info->reserved = 0;
  for (int a = 0; a < 3; ++a) info->box_lo[a] = t->lo[a];
  info->box_size = t->size;
  return TREVR2_OK;
}

}  // extern "C"

namespace trevr2 {

// Export kernels: undo the normalisation and the band padding.
__global__ void k_export_bands(const float* src, int64_t n, int nb, int nbp, float scale, float* dst) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= n * nb) return;
  int64_t q = i / nb;
  int b = int(i % nb);
  dst[i] = src[q * nbp + b] * scale;
}

__global__ void k_export_centre(const double* c64, int64_t n, double lo0, double lo1, double lo2,
                                double size, double* dst) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= 3 * n) return;
  double lo = (i % 3 == 0) ? lo0 : ((i % 3 == 1) ? lo1 : lo2);
  dst[i] = lo + size * c64[i];
}

__global__ void k_export_scale(const double* src, int64_t n, double scale, double* dst) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) dst[i] = src[i] * scale;
}

}  // namespace trevr2

extern "C" int trevr2_tree_export(const trevr2_tree* tree, int field, void* dst, size_t bytes,
                                  void* stream) {
  clear_error();
  if (!tree || !dst) {
    set_error("trevr2_tree_export: NULL argument");
    return TREVR2_EINVAL;
  }
  const Tree* t = reinterpret_cast<const Tree*>(tree);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t N = t->N, n = t->n_nodes;
  const void* src = nullptr;
  size_t need = 0;
  switch (field) {
    case TREVR2_F_KEYS: src = t->keys; need = N * sizeof(uint64_t); break;
    case TREVR2_F_PERM: src = t->perm; need = N * sizeof(int); break;
    case TREVR2_F_PREFIX: src = t->prefix; need = n * sizeof(uint64_t); break;
    case TREVR2_F_DEPTH: src = t->depth; need = n * sizeof(int); break;
    case TREVR2_F_FIRST: src = t->first; need = n * sizeof(int); break;
    case TREVR2_F_COUNT: src = t->count; need = n * sizeof(int); break;
    case TREVR2_F_CHILD: src = t->child; need = n * sizeof(int); break;
    case TREVR2_F_PARENT: src = t->parent; need = n * sizeof(int); break;
    case TREVR2_F_LUM: need = n * t->nb * sizeof(float); break;
    case TREVR2_F_CENTRE: need = 3 * n * sizeof(double); break;
    case TREVR2_F_ALPHA_LEAF: need = n * t->nb * sizeof(float); break;
    case TREVR2_F_B: need = n * sizeof(double); break;
    default:
      set_error("trevr2_tree_export: unknown field %d", field);
      return TREVR2_EINVAL;
  }
  if (bytes < need) {
    set_error("trevr2_tree_export: destination holds %zu bytes, %zu needed", bytes, need);
    return TREVR2_EINVAL;
  }
  if (need == 0) return TREVR2_OK;
  if (src) {
    T2_CUDA(cudaMemcpyAsync(dst, src, need, cudaMemcpyDeviceToDevice, st));
  } else if (field == TREVR2_F_LUM) {
    k_export_bands<<<blocks_for(n * t->nb, 256), 256, 0, st>>>(t->Lnode, n, t->nb, t->nbp, 1.0f,
                                                                static_cast<float*>(dst)); note_launch();
  } else if (field == TREVR2_F_ALPHA_LEAF) {
    k_export_bands<<<blocks_for(n * t->nb, 256), 256, 0, st>>>(
        t->alpha_leaf, n, t->nb, t->nbp, float(1.0 / t->size), static_cast<float*>(dst)); note_launch();
  } else if (field == TREVR2_F_CENTRE) {
    k_export_centre<<<blocks_for(3 * n, 256), 256, 0, st>>>(t->c64, n, t->lo[0], t->lo[1],
                                                            t->lo[2], t->size,
                                                            static_cast<double*>(dst)); note_launch();
  } else if (field == TREVR2_F_B) {
    k_export_scale<<<blocks_for(n, 256), 256, 0, st>>>(t->B64, n, t->size,
                                                       static_cast<double*>(dst)); note_launch();
  }
  T2_CUDA(cudaGetLastError());
  return TREVR2_OK;
}

// ---------------------------------------------------------------------------
// Refinement tau_refine (Sec. 2.5.2; off by default): a cell whose optical
// depth varies by more than tau_refine inside it opens as well.  The
// variation is (largest - smallest bucket alpha among the leaves under the
// cell) times its longest side, the largest over the bands.  Opening is
// forced by a node copy whose B is so large that B > theta d holds for
// every d in the unit cube, so every walk (forward, per bucket, batched,
// adjoint) refines without any change to its code.
namespace trevr2 {

constexpr float kRefinedB = 1e18f;  // B^2 and the FP32 guard stay finite

// One depth of the tree, deepest first: the per-band range of the leaves'
// alpha under each node and the node's variation.
template <int NBP>
__global__ void k_tau_variation_level(int64_t lb, int64_t le, const NodeW* __restrict__ nodes,
                                      const float* __restrict__ alpha_leaf, float* amin,
                                      float* amax, float* __restrict__ dtau) {
  const int64_t q = lb + blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= le) return;
  const NodeW nd = nodes[q];
  float var = 0.0f;
#pragma unroll
  for (int b = 0; b < NBP; ++b) {
    float lo, hi;
    if (nd.meta & kMetaLeaf) {
      lo = hi = alpha_leaf[q * NBP + b];
    } else {
      const int64_t c = nd.child;
      lo = fminf(amin[c * NBP + b], amin[(c + 1) * NBP + b]);
      hi = fmaxf(amax[c * NBP + b], amax[(c + 1) * NBP + b]);
    }
    amin[q * NBP + b] = lo;
    amax[q * NBP + b] = hi;
    var = fmaxf(var, hi - lo);
  }
  // the longest side: the axis split least often, z, floor(depth / 3) times
  const int d = int(nd.meta & kMetaDepthMask);
  dtau[q] = var * ldexpf(1.0f, -splits_on_axis(d, 2));
}

__global__ void k_refine_nodes(int64_t n, const NodeW* __restrict__ nodes,
                               const float* __restrict__ dtau, float tau,
                               NodeW* __restrict__ out) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= n) return;
  NodeW nd = nodes[q];
  if (!(nd.meta & kMetaLeaf) && dtau[q] > tau) nd.B = kRefinedB;
  out[q] = nd;
}

}  // namespace trevr2

extern "C" int trevr2_set_tau_refine(trevr2_tree* tree, double tau_refine, void* stream) {
  clear_error();
  if (!tree) {
    set_error("trevr2_set_tau_refine: tree is NULL");
    return TREVR2_EINVAL;
  }
  if (!(tau_refine > 0.0)) {
    set_error("trevr2_set_tau_refine: tau_refine must be positive (infinity turns it off)");
    return TREVR2_EINVAL;
  }
  Tree* t = reinterpret_cast<Tree*>(tree);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (std::isinf(tau_refine)) {
    t->refine_on = false;
    t->tau_refine = tau_refine;
    return TREVR2_OK;
  }
  const int64_t n = t->n_nodes;
  if (!t->dtau) {
    // computed into temporaries and kept only when complete, so that a
    // failed call leaves the tree as it was
    DeviceTemp<float> dtau(st), range(st);
    T2_CHECK(dalloc(&dtau.p, size_t(n), st));
    T2_CHECK(dalloc(&range.p, size_t(n) * 2 * t->nbp, st));
    float* amin = range.p;
    float* amax = range.p + size_t(n) * t->nbp;
    for (int d = int(t->level_begin.size()) - 2; d >= 0; --d) {
      const int64_t lb = t->level_begin[d], le = t->level_begin[d + 1];
      if (le <= lb) continue;
      const unsigned g = blocks_for(le - lb, 256);
      switch (t->nbp) {
        case 1: k_tau_variation_level<1><<<g, 256, 0, st>>>(lb, le, t->nodes, t->alpha_leaf, amin, amax, dtau.p); break;
        case 2: k_tau_variation_level<2><<<g, 256, 0, st>>>(lb, le, t->nodes, t->alpha_leaf, amin, amax, dtau.p); break;
        default: k_tau_variation_level<4><<<g, 256, 0, st>>>(lb, le, t->nodes, t->alpha_leaf, amin, amax, dtau.p); break;
      }
      note_launch();
    }
    T2_CUDA(cudaGetLastError());
    t->dtau = dtau.p;
    dtau.p = nullptr;
  }
  if (!t->nodes_refined) T2_CHECK(dalloc(&t->nodes_refined, size_t(n), st));
  k_refine_nodes<<<blocks_for(n, 256), 256, 0, st>>>(n, t->nodes, t->dtau, float(tau_refine),
                                                      t->nodes_refined);
  note_launch();
  T2_CUDA(cudaGetLastError());
  t->refine_on = true;
  t->tau_refine = tau_refine;
  return TREVR2_OK;
}
