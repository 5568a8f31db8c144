// Internal declarations of the GB300 TREVR2 library (not part of the ABI).
//
// Coordinates: everything on the device lives in the normalised root cube
// [0,1)^3 (u = (x - lo)/size, computed in FP64).  Cell boxes are then exact
// dyadic numbers in FP32; absorption is stored per normalised length
// (alpha * size) and J is rescaled by 1/size^2 at the end.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "trevr2.h"

namespace trevr2 {

constexpr int kMaxDepth = 63;
constexpr int kKeyBits = 21;

// ---------------------------------------------------------------------------
// Node record read by the walk: one 32-byte load from the tree's arrays, which
// start on 256 bytes (load_node); copies in shared memory are 16-byte aligned.
struct __align__(16) NodeW {
  float lo[3];    // normalised lower corner (exact)
  float B;        // largest distance from the centre of luminosity to a corner
  int child;      // lower child, upper = child + 1; -1 for a leaf
  int aux;        // internal: row of the alpha table; leaf: first element (sorted)
  int count;      // elements under the node
  uint32_t meta;  // depth | flags
};
static_assert(sizeof(NodeW) == 32, "load_node reads a record at once, 32-byte aligned");
constexpr uint32_t kMetaDepthMask = 63u;
constexpr uint32_t kMetaLeaf = 1u << 8;
constexpr uint32_t kMetaHasL = 1u << 9;      // some luminosity below
constexpr uint32_t kMetaHasAlpha = 1u << 10; // some absorption below
constexpr int kMetaAxisShift = 12;            // split axis (depth mod 3) in bits 12-13
constexpr uint32_t kMetaChild0Alpha = 1u << 14;  // lower half has some absorption
constexpr uint32_t kMetaChild1Alpha = 1u << 15;  // upper half has some absorption

// Source found by the cut, binned to its beam: projected distance s along
// the beam, r/s, the geometric kernel g(r), and where its luminosity lives.
struct __align__(16) SrcEntry {
  float s;
  float rs;
  float w;
  int ref;  // node index, or sorted element index | kRefElement
};
constexpr int kRefElement = int(0x80000000u);

// Device status bits (OR-ed into the tree's status word).
constexpr uint32_t kStatusBadActive = 1u << 0;
constexpr uint32_t kStatusStackOverflow = 1u << 1;
constexpr uint32_t kStatusBadInput = 1u << 2;
constexpr uint32_t kStatusOutsideBox = 1u << 3;
constexpr uint32_t kStatusBarrier = 1u << 4;     // a grid barrier gave up waiting
constexpr uint32_t kStatusPPOverflow = 1u << 5;  // a p-p sphere held too many particles
constexpr uint32_t kStatusTables = 1u << 6;      // the barrier was the tables' kernel's

// Geometry of the transmission average for one cell shape and one beam pair:
// weights V1/V (= V2/V), V12/V and the chord through the centre of a cell of
// unit scale (d scales with the cell, the weights do not).
struct __align__(16) TransGeo {
  float w1;
  float w12;
  float d_unit;
  float pad;
};

struct Table {
  int nside = 0;
  // Whether a device status read after its kernel was free of kStatusTables.
  // Until then the kernel may have given up at a barrier; settle_tables drops
  // such a table, so that no later call takes it for a finished one.
  bool checked = false;
  bool linear = false;         // linear absorption average instead of Eq. transmissionavg
  float* alpha = nullptr;      // [n_internal][P][nbp] normalised absorption
  float4* dirs = nullptr;      // [npix] beam directions (xyz), w = pair index (int bits)
  double* dirs64 = nullptr;    // [npix][3]
  TransGeo* geo = nullptr;     // [3][P]
  // beams by direction for the cell-by-cell absorption (nside <= kCellNside),
  // built on first use: for every cell shape and square of a cube map of
  // directions, all beams in the order of the size from which on a cell there
  // can be crossed by them, and how many there are for each class of sizes
  float4* beam_inv = nullptr;     // [npix, by beam_slot] 1 / direction, w = pair (owns all three)
  uint8_t* beam_list = nullptr;   // [3][6 nf^2][npix rounded up to 16], nf = beam_map_side(nside)
  uint8_t* beam_count = nullptr;  // [3][6 nf^2][kConeClasses + 1]
  // complex source model (Sec. 2.7), built on first use with TREVR2_CSM
  float* csm_tau = nullptr;    // [n][npix][nbp] optical depth of each luminous cell's ray
  float* csm_d = nullptr;      // [n][npix] its length (normalised)
  int* csm_anti = nullptr;     // [npix] pixel of -n_k
};

// ---------------------------------------------------------------------------
struct Tree {
  int64_t N = 0;
  int nb = 0;
  int nbp = 0;     // bands padded to 1, 2 or 4
  int bucket = 12;
  double lo[3] = {0, 0, 0};
  double size = 1.0;
  int64_t n_nodes = 0;
  int64_t n_internal = 0;
  int max_depth = 0;
  int64_t n_luminous = 0;  // elements with some luminosity
  bool has_h = false;
  cudaStream_t last_stream = nullptr;

  // elements, sorted by key
  uint64_t* keys = nullptr;   // [N]
  int* perm = nullptr;        // [N] sorted -> caller index
  int* inv = nullptr;         // [N] caller index -> sorted
  double* pos64 = nullptr;    // [N][3] normalised
  float4* pos32 = nullptr;    // [N] normalised xyz, w = total luminosity
  float* Lelem = nullptr;     // [N][nbp]
  float* km = nullptr;        // [N][nbp] kappa * m (caller units)
  float* hn = nullptr;        // [N] element size / size
  float* mass = nullptr;      // [N] element mass (caller units)

  // nodes (breadth first)
  uint64_t* prefix = nullptr; // [n]
  int* depth = nullptr;       // [n]
  int* first = nullptr;       // [n]
  int* count = nullptr;       // [n]
  int* child = nullptr;       // [n]
  int* parent = nullptr;      // [n]
  int* int_index = nullptr;   // [n] row in the alpha table, -1 for leaves
  NodeW* nodes = nullptr;     // [n]
  float* Lnode = nullptr;     // [n][nbp]
  float4* csrc = nullptr;     // [n] centre of luminosity (normalised) xyz, w = total L
  double* c64 = nullptr;      // [n][3] normalised centre of luminosity
  double* B64 = nullptr;      // [n] normalised B
  float* alpha_leaf = nullptr;// [n][nbp] normalised bucket absorption (0 internal)
  uint32_t* lmask = nullptr;  // [n] leaves: which of their first 32 elements are luminous
  // refinement tau_refine (Sec. 2.5.2): node records with B raised where the
  // optical depth varies by more than tau_refine inside the cell
  float* dtau = nullptr;          // [n] optical-depth variation of each cell
  NodeW* nodes_refined = nullptr; // [n], kept until the tree is freed
  bool refine_on = false;
  double tau_refine = 0.0;
  std::vector<int64_t> level_begin;  // host: first node of each depth, plus end

  std::vector<Table> tables;  // cached per nside

  // walk buffers (grown on demand)
  void* scratch = nullptr;
  size_t scratch_bytes = 0;
  void* order_buf = nullptr;   // receivers in key order: keys + slots
  size_t order_bytes = 0;
  uint32_t* status = nullptr;             // device status word
  unsigned long long* counter = nullptr;  // device work counter
};

// ---------------------------------------------------------------------------
// Barrier of all blocks of one cooperative launch (so they are resident
// together): *bar counts arrivals, from 0 at the launch.  The wait ends after
// `polls` polls at the latest (barrier_polls()); then the barrier is marked as
// failed for good, `bits` go to *status, and every block gets false and returns.
constexpr uint32_t kBarrierSpins = 1u << 24;
constexpr uint32_t kBarrierFailed = 0x80000000u;

__device__ __forceinline__ bool grid_barrier(uint32_t* bar, uint32_t blocks, uint32_t* status,
                                             uint32_t polls, uint32_t bits = kStatusBarrier) {
  __shared__ uint32_t arrived_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t ok = 1;
    if (blocks > 1) {
      __threadfence();
      const uint32_t at = atomicAdd(bar, 1u);
      const uint32_t target = (at / blocks + 1u) * blocks;
      uint32_t seen = 0, spins = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
        if ((seen | at) & kBarrierFailed) ok = 0;
        if (ok && seen < target && ++spins == polls) {
          atomicOr(bar, kBarrierFailed);
          if (status) atomicOr(status, bits);
          ok = 0;
        }
      } while (ok && seen < target);
      __threadfence();
    }
    arrived_ok = ok;
  }
  __syncthreads();
  return arrived_ok != 0;
}

// ---------------------------------------------------------------------------
// Host helpers (errors, allocation).
void set_error(const char* fmt, ...);
void clear_error();  // first in every entry point (it also forgets the last one's pool)

int cuda_fail(cudaError_t e, const char* what);

// Counts kernels launched by this library (host side; see trevr2_kernel_launches).
void note_launch();
#define T2_CUDA(call)                                            \
  do {                                                           \
    cudaError_t e_ = (call);                                     \
    if (e_ != cudaSuccess) return ::trevr2::cuda_fail(e_, #call);\
  } while (0)
#define T2_CHECK(rc_expr)        \
  do {                           \
    int rc_ = (rc_expr);         \
    if (rc_ != TREVR2_OK) return rc_; \
  } while (0)

// Every device allocation of the library (stream ordered, freed with
// dfree / cudaFreeAsync).  `what` names it in the error message.  A failure
// requested with trevr2_debug_set(TREVR2_DEBUG_FAIL_ALLOC, n) happens here.
int device_alloc(void** p, size_t bytes, cudaStream_t st, const char* what);

template <class T>
int dalloc(T** p, size_t count, cudaStream_t st) {
  if (count == 0) count = 1;
  return device_alloc(reinterpret_cast<void**>(p), count * sizeof(T), st, "device allocation");
}

template <class T>
void dfree(T*& p, cudaStream_t st) {
  if (p) cudaFreeAsync(p, st);
  p = nullptr;
}

// A temporary device buffer freed (stream ordered) when it goes out of
// scope, so that every early error return releases it.
template <class T>
struct DeviceTemp {
  T* p = nullptr;
  cudaStream_t st;
  explicit DeviceTemp(cudaStream_t s) : st(s) {}
  ~DeviceTemp() { dfree(p, st); }
  DeviceTemp(const DeviceTemp&) = delete;
  DeviceTemp& operator=(const DeviceTemp&) = delete;
};

// Capacity of the source cut's traversal stack set by
// trevr2_debug_set(TREVR2_DEBUG_SOURCE_STACK, c); 0 when not set.
int debug_source_stack_cap();
// Polls of a grid barrier: kBarrierSpins, or what
// trevr2_debug_set(TREVR2_DEBUG_BARRIER_POLLS, n) allows.
uint32_t barrier_polls();
// Capacities lowered by TREVR2_DEBUG_CELL_CAP and TREVR2_DEBUG_TEAM_HITS
// (INT_MAX when not set).
int debug_cell_cap();
int debug_team_hits();

// Blocks of a cooperative launch on `st`: at most per_sm (the kernel's bound,
// so that they are resident together) per SM that the stream's work may use,
// fewer where the work would leave them idle at the barriers.
constexpr int kMaxCoopBlocks = 512;
int coop_blocks(int64_t work, int64_t per_block, int per_sm, cudaStream_t st, int* out);

// The receivers' slots in their elements' sorted order (keys: their sorted
// positions, N for an index outside [0, N)).
int order_receivers(const Tree* t, const int64_t* active, int64_t A, uint64_t* keys, int* slots,
                    cudaStream_t st);

// Exclusive scan of n int32 values in place; *d_total (device) gets the sum.
// ws: device, scan_ws_ints(n) ints.
size_t scan_ws_ints(int64_t n);
int scan_exclusive_i32(int* d, int64_t n, int* d_total, cudaStream_t st, int* ws);

// Stable LSD radix sort of keys below 2^key_bits with int32 payload (in place).
// ws (device, radix_ws_bytes(n) bytes) or NULL to allocate one stream ordered.
size_t radix_ws_bytes(int64_t n);
// A grid barrier that gives up sets kStatusBarrier in *status.
int radix_sort_u64_i32(uint64_t* keys, int* vals, int64_t n, cudaStream_t st, uint32_t* status,
                       int key_bits = 64, void* ws = nullptr);

// Alpha tables and beam directions for one nside and averaging (built and
// cached): Eq. transmissionavg, or with `linear` the volume-weighted linear
// average of the halves (Sec. 2.6's comparison scheme).
int ensure_table(Tree* t, int nside, cudaStream_t st, Table** out, bool linear = false);

// With the device status s of everything enqueued so far: drops the unchecked
// tables where their kernel gave up, else marks them as checked.
void settle_tables(Tree* t, uint32_t s, cudaStream_t st);

// For callers that keep a table's pointers or hand its values out without a
// read_status after them: reads the status if some table is unchecked
// (synchronises `st` then; not while it is being captured), settles the tables
// and returns ETIMEOUT when their kernel gave up.  Other status bits stay.
int check_tables(Tree* t, cudaStream_t st);
void free_table(Table* tb, cudaStream_t st);

// The finest beams whose absorption is summed cell by cell (their indices fit
// one byte: 192 beams at nside 4); finer ones are walked beam by beam.
constexpr int kCellNside = 4;
constexpr int kConeClasses = 32;
// 1 / n of a beam with a zero component: large enough to put any face not
// exactly at the origin beyond the root cube, small enough to stay finite.
constexpr float kFlatInv = 1e30f;
// Where the cell-by-cell walk keeps beam k in its tables (its own inverse): a
// look-up's beams are neighbours, k +- 1 in their ring or about 16 apart in the
// next at nside 4, and these fall into different 16-byte banks.
__host__ __device__ inline int beam_slot(int k) { return k ^ ((k >> 4) & 3); }
// Squares per cube face and axis: a square's half-diagonal is 0.18 / nside
// rad, a fifth of the spacing of the beams.
__host__ __device__ inline int beam_map_side(int nside) { return 8 * nside; }

// The beam look-up tables of one table's nside (built and cached).
int ensure_beam_map(Table* tb, cudaStream_t st);

inline int nbp_of(int nb) { return nb <= 1 ? 1 : (nb == 2 ? 2 : 4); }

// Extent of a cell at `depth` along axis a: 2^-(number of splits on a).
__host__ __device__ inline int splits_on_axis(int depth, int a) { return (depth + 2 - a) / 3; }

}  // namespace trevr2
