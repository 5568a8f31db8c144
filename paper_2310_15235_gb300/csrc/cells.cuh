// Absorption summed cell by cell (the walk's phase A for beams up to
// kCellNside), shared by the forward kernels.
//
// A receiver's cut holds about a thousand absorbing cells, and a beam crosses
// few of them; a cell is crossed by about three beams.  Walking every beam
// through the tree repeats each node's load and opening test once per beam
// that reaches it (8,700 stack pops a receiver on the clumpy 2M field, 18 of
// 32 lanes active) to find 2,800 crossings.  Here the cut is walked once, 32
// nodes a step, and its absorbing cells are listed; each cell then names the
// beams that can cross it by a look-up of its direction and angular radius,
// and only those (about 2.3 for each that does) are tested against its box.
// No lane walks anything: the (cell, beam) pairs are laid out evenly over the
// lanes.
//
// The crossings come in the order of the tree, not along the beams, so the
// optical depth is built from increments: a crossing adds alpha times its
// whole chord to the first source of its beam beyond it, and writes alpha
// (s - t0) to the sources inside it (each source of a beam lies in one cell);
// the sum of a beam's increments up to a source, plus that source's own, is
// its tau.  All sums run in a fixed order (lane and crossing order), so a
// receiver's J does not depend on the launch.
//
// What bounds it: L2 latency and instruction issue together (issue 53-60 % of
// cycles, 28 of 32 lanes active, 51k instructions a receiver of the 96^3 field,
// nside 4, against 84k beam by beam; the L1 is left about 50 KB and hits 17 %, so
// resident warps count: see kCellWarpsPerSM).  Measured against beam by beam, whole
// calls: 2M clumpy field, nside 4, theta 0.5, 3 bands 259 -> 200 ms; its
// per-bucket walk 45.2 -> 35.7 ms; 64^3, nside 2, 300 sources 6.6 -> 5.0 ms.
#pragma once

#include <algorithm>

#include "walk.cuh"

namespace trevr2 {

// Box extents by depth in shared memory: the longest side 2^-floor(depth / 3)
// (256 bytes, so that the walk kernels keep their blocks per SM), the others
// halved on the axes already split at this depth.  Every walk kernel fills
// the table before its first receiver.
__shared__ float g_ext_e[64];

__device__ __forceinline__ void init_ext_tab() {
  if (threadIdx.x < 64) g_ext_e[threadIdx.x] = __int_as_float((127 - int(threadIdx.x) / 3) << 23);
  __syncthreads();
}

// x, y, z extents (the values of node_ext), and w = the split axis's (z's).
__device__ __forceinline__ float4 ext_of(uint32_t meta) {
  const float e = g_ext_e[meta & kMetaDepthMask];
  const uint32_t r = (meta >> kMetaAxisShift) & 3u;
  return make_float4(r > 0u ? 0.5f * e : e, r > 1u ? 0.5f * e : e, e, e);
}

// A node record as one 32-byte load.
__device__ __forceinline__ NodeW load_node(const NodeW* p) {
  uint32_t r[8];
  asm("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "l"(p));
  NodeW n;
  n.lo[0] = __uint_as_float(r[0]);
  n.lo[1] = __uint_as_float(r[1]);
  n.lo[2] = __uint_as_float(r[2]);
  n.B = __uint_as_float(r[3]);
  n.child = int(r[4]);
  n.aux = int(r[5]);
  n.count = int(r[6]);
  n.meta = r[7];
  return n;
}

// 1 << s, 0 for s >= 32 (the shift clamps).
__device__ __forceinline__ unsigned bit_at(int s) {
  unsigned r;
  asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(s));
  return r;
}

// The cut seen from x, 32 nodes a step: the references of the sources with
// running index in [lo, lo + M) go to U[].ref as in phase_sources, and the
// absorbing cells with running index in [clo, clo + a.cell_cap) to cells[].
// Returns the numbers of sources and cells (warp-uniform).  A step takes the
// 32 top entries of the stack and puts the halves of the topmost back on top,
// so the stack stays ordered by depth and holds at most 32 (depth + 2)
// entries: by induction over the steps, at most 32 (d + 1) of depth d or less
// once deeper ones are there.
template <bool kBucket, bool kPP>
static __device__ int2 phase_cut(const WalkArgs& a, float3 x, int si, int lane, int* stk, int cap,
                                 SrcEntry* U, int lo, int* cells, int clo, float rpp) {
  int sp = 1;
  if (lane == 0) stk[0] = 0;
  __syncwarp();
  int emitted = 0, listed = 0;
  const unsigned lt = (1u << lane) - 1u;
  while (sp > 0) {
    const int k = min(32, sp);
    const int q = lane < k ? stk[sp - 1 - lane] : -1;
    sp -= k;
    bool push = false, cell = false, source = false, lit = false;
    int child = 0, first = 0, count = 0;
    __syncwarp();
    if (q >= 0) {
      const NodeW nd = load_node(a.nodes + q);
      if (nd.meta & (kMetaHasL | kMetaHasAlpha)) {
        const float4 e = ext_of(nd.meta);
        const bool opens = cell_opens_e<kBucket, kPP>(a, q, nd, make_float3(e.x, e.y, e.z), x, si, rpp);
        const bool leaf = (nd.meta & kMetaLeaf) != 0;
        const bool luminous = (nd.meta & kMetaHasL) != 0;
        push = opens && !leaf;
        cell = !push && (nd.meta & kMetaHasAlpha) != 0;
        source = !opens && luminous;
        lit = opens && leaf && luminous;
        child = nd.child;
        first = nd.aux;
        count = nd.count;
      }
    }
    {  // opened halves, the topmost node's on top
      const unsigned m = __ballot_sync(0xffffffffu, push);
      const int room = (cap - sp) >> 1, want = __popc(m);
      const int at = want - 1 - __popc(m & lt);
      if (push && at < room) {
        stk[sp + 2 * at] = child + 1;
        stk[sp + 2 * at + 1] = child;
      }
      if (want > room && lane == 0) atomicOr(a.status, kStatusStackOverflow);
      sp += 2 * min(want, room);
    }
    {  // absorbing cells
      const unsigned m = __ballot_sync(0xffffffffu, cell);
      const int idx = listed + __popc(m & lt) - clo;
      if (cell && unsigned(idx) < unsigned(a.cell_cap)) cells[idx] = q;
      listed += __popc(m);
    }
    {  // accepted luminous cells
      const unsigned m = __ballot_sync(0xffffffffu, source);
      const int idx = emitted + __popc(m & lt) - lo;
      if (source && unsigned(idx) < unsigned(a.M)) U[idx].ref = q;
      emitted += __popc(m);
    }
    // luminous elements of opened leaves
    if (__any_sync(0xffffffffu, lit)) {
      uint32_t bits = 0;
      if (!lit) {
        count = 0;
      } else {
        bits = a.lmask[q];
        bits &= ~bit_at(si - first);  // never the receiver itself
      }
      if (__any_sync(0xffffffffu, count > 32)) {  // leaves beyond the masks' 32 elements
        const int maxc = __reduce_max_sync(0xffffffffu, count);
        for (int e = 0; e < maxc; ++e) {
          const int sj = first + e;
          const bool em = e < count && a.pos32[sj].w > 0.0f && sj != si;
          const unsigned m = __ballot_sync(0xffffffffu, em);
          const int idx = emitted + __popc(m & lt) - lo;
          if (em && unsigned(idx) < unsigned(a.M)) U[idx].ref = sj | kRefElement;
          emitted += __popc(m);
        }
      } else {
        for (unsigned m; (m = __ballot_sync(0xffffffffu, bits != 0u)) != 0u; bits &= bits - 1u) {
          const int idx = emitted + __popc(m & lt) - lo;
          if (bits && unsigned(idx) < unsigned(a.M)) U[idx].ref = (first + __ffs(bits) - 1) | kRefElement;
          emitted += __popc(m);
        }
      }
    }
    __syncwarp();
  }
  return make_int2(emitted, listed);
}

// A warp's shared memory for the cells (ints), in the space of the cut's
// stack: 32 cells' boxes and the first 16 of each one's beams, 64 pending
// crossings, the distances of bin_cap sources.  Behind it the beams' bucket
// offsets [npix], their farthest distances [npix, by beam_slot] and 36 ints of
// scratch.
constexpr int kCellStage = 32 * 12;
constexpr int kCellHits = 64 * 4;

// Up to 32 crossings (t0, t1, row, beam), one per lane: their increments, to
// the sources [e0, e0 + m) of V.
// inside(j, alpha) is called for every source inside its crossing's cell.
template <int NBP, bool kInOrder, class Inside>
__device__ __forceinline__ void add_crossings(const WalkArgs& a, int lane, bool live, float4 h,
                                              const float4* binv, const float* ss, const int* off,
                                              int e0, int m, float s_before, float* T, float* own,
                                              bool first, Inside inside) {
  BandVec<NBP> add;
#pragma unroll
  for (int b = 0; b < NBP; ++b) add.v[b] = 0.0f;
  int key = -1;
  if (live) {
    const float t0 = h.x, t1 = h.y;
    const int row = __float_as_int(h.z), at = __float_as_int(h.w), k = beam_slot(at);
    const float* rp = row < 0 ? a.alpha_leaf + int64_t(-(row + 1)) * NBP
                              : a.alpha_tab + (int64_t(row) * a.P + __float_as_int(binv[at].w)) * NBP;
    add = load_bands<NBP>(rp);
    const int js = (k ? off[k - 1] : 0) - e0, je = min(off[k] - e0, m);
    int j = max(js, 0);
    for (int b = je; j < b;) {  // the first source of the beam at or beyond t0
      const int mid = (j + b) >> 1;
      if (ss[mid] < t0) j = mid + 1; else b = mid;
    }
    for (; j < je && ss[j] < t1; ++j) {  // sources inside the cell
      const float ds = ss[j] - t0;
      inside(j, add);
      BandVec<NBP> tk;
#pragma unroll
      for (int b = 0; b < NBP; ++b) tk.v[b] = add.v[b] * ds;
      if (!first) {
        const BandVec<NBP> was = load_bands<NBP>(own + j * NBP);
#pragma unroll
        for (int b = 0; b < NBP; ++b) tk.v[b] += was.v[b];
      }
      store_bands<NBP>(own + j * NBP, tk);
    }
    // (a crossing that ends before one of the beam's earlier sources has been
    // added to that one)
    if (j < je && !(js < 0 && t1 <= s_before)) key = j;
    const float len = t1 - t0;
#pragma unroll
    for (int b = 0; b < NBP; ++b) add.v[b] *= len;
  }
  // the first lane of those that meet the same source adds up their
  // increments in lane order, so that T is read and written once; kInOrder: one
  // after another onto T, so that the sum does not depend on how the crossings
  // fall into groups (k_walk_team's fall otherwise than k_walk's)
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  const bool lead = key >= 0 && (peers & ((1u << lane) - 1u)) == 0u;
  float* p = T + key * NBP;
  BandVec<NBP> old;
  if (lead) old = load_bands<NBP>(p);
  if constexpr (kInOrder) {
    if (lead) {
#pragma unroll
      for (int b = 0; b < NBP; ++b) old.v[b] += add.v[b];
    }
  }
  unsigned rest = lead ? peers & (peers - 1u) : 0u;
  while (__any_sync(0xffffffffu, rest != 0u)) {
    const int from = rest ? __ffs(rest) - 1 : lane;
#pragma unroll
    for (int b = 0; b < NBP; ++b) {
      const float v = __shfl_sync(0xffffffffu, add.v[b], from);
      if (rest) (kInOrder ? old : add).v[b] += v;
    }
    rest &= rest - 1u;
  }
  if (lead) {
    if constexpr (!kInOrder) {
#pragma unroll
      for (int b = 0; b < NBP; ++b) old.v[b] += add.v[b];
    }
    store_bands<NBP>(p, old);
  }
  __syncwarp();
}

// bin_sources for up to bin_cap sources: the records' (s, beam, index) are put
// in the order of their beams in shared memory, ranked there, and every record
// is moved once.  key: 2 bin_cap ints.
static __device__ int bin_sources_small(const WalkArgs& a, int lane, const SrcEntry* U, const int* Up,
                                        int n, SrcEntry* V, int* off, int* key) {
  const int npix = a.npix;
  float* ks = reinterpret_cast<float*>(key);
  uint32_t* kk = reinterpret_cast<uint32_t*>(key + a.bin_cap);
  for (int k = lane; k < npix; k += 32) off[k] = 0;
  __syncwarp();
  for (int e = lane; e < n; e += 32)
    if (const int k = Up[e]; k >= 0) atomicAdd(&off[k], 1);
  __syncwarp();
  // exclusive scan of the bucket sizes
  const int per = (npix + 31) / 32;
  const int b0 = min(lane * per, npix), b1 = min(b0 + per, npix);
  int sum = 0;
  for (int k = b0; k < b1; ++k) sum += off[k];
  const int incl = warp_incl_scan(sum, lane);
  int run = incl - sum;
  for (int k = b0; k < b1; ++k) {
    const int c = off[k];
    off[k] = run;
    run += c;
  }
  __syncwarp();
  for (int e = lane; e < n; e += 32) {
    const int k = Up[e];
    if (k < 0) continue;
    const int slot = atomicAdd(&off[k], 1);
    ks[slot] = U[e].s;
    kk[slot] = uint32_t(e) | (uint32_t(k) << 16);
  }
  __syncwarp();
  n = off[npix - 1];  // records binned
  // each record's rank in its bucket by (projected distance, index)
  for (int p = lane; p < n; p += 32) {
    const uint32_t me = kk[p];
    const int k = int(me >> 16), s0 = k ? off[k - 1] : 0, s1 = off[k];
    const float s = ks[p];
    int r = s0;
    for (int j = s0; j < s1; ++j) r += ks[j] < s || (ks[j] == s && kk[j] < me);
    V[r] = U[me & 0xffffu];
  }
  __syncwarp();
  return n;
}

// 32 cells of the cut, one per lane (q < 0: none): the (cell, beam) pairs that
// can cross, 32 at a time, each tested against its cell's box; push(hit, t0, t1,
// row, beam slot) is called by the whole warp for every 32 pairs.  The beams of
// a cell come from the look-up by its shape, the direction of its centre and
// the class of the cone about it that holds the box (sin^2 = H2 / D2; with x
// inside the sphere through the corners, every beam).  stage: kCellStage ints.
template <bool kPP, class Push>
__device__ __forceinline__ void cross_batch(const WalkArgs& a, float3 x, int lane, int q,
                                            int* stage, const float4* binv, const float* far,
                                            float rpp, Push push) {
  const unsigned lt = (1u << lane) - 1u;
  const int npix = a.npix, stride = (npix + 15) & ~15;
  const float nfh = 0.5f * float(a.beam_side);
  float4* box0 = reinterpret_cast<float4*>(stage);
  float4* box1 = box0 + 32;
  uint4* beams = reinterpret_cast<uint4*>(box1 + 32);
  const uint8_t* beams8 = reinterpret_cast<const uint8_t*>(beams);
  int count = 0, total;
  int start;
  {
    NodeW nd;
    if (q >= 0) nd = load_node(a.nodes + q);
    int sq = 0, row = 0;
    float lx = 0.0f, ly = 0.0f, lz = 0.0f, hx = 0.0f, hy = 0.0f, hz = 0.0f;
    if (q >= 0) {
      const float4 e = ext_of(nd.meta);
      lx = nd.lo[0] - x.x; hx = nd.lo[0] + e.x - x.x;
      ly = nd.lo[1] - x.y; hy = nd.lo[1] + e.y - x.y;
      lz = nd.lo[2] - x.z; hz = nd.lo[2] + e.z - x.z;
      row = (nd.meta & kMetaLeaf) ? -(q + 1) : nd.aux;
      const float cx = 0.5f * (lx + hx), cy = 0.5f * (ly + hy), cz = 0.5f * (lz + hz);
      const float D2 = cx * cx + cy * cy + cz * cz;
      const float H2 = 0.25f * (e.x * e.x + e.y * e.y + e.z * e.z);
      count = npix;
      if (D2 > H2) {
        // sqrt(1 - cos) by classes; the look-up's slack covers the approximations
        const float c2 = fmaxf(1e-12f, 1.0f - __fdividef(H2, D2));
        const float v = fmaxf(1e-12f, 1.0f - c2 * rsqrtf(c2));
        const int cls = int(v * rsqrtf(v) * float(kConeClasses) + 1.02f);
        if (cls <= kConeClasses) {
          const float ax = fabsf(cx), ay = fabsf(cy), az = fabsf(cz);
          const float vm = fmaxf(fmaxf(ax, ay), az);
          const bool mx = ax == vm, my = !mx && ay == vm;
          const float ca = mx ? cy : cx, cb = mx || my ? cz : cy, cm = mx ? cx : (my ? cy : cz);
          const float iv = __fdividef(nfh, vm);
          const int top = a.beam_side - 1;
          const int i = max(0, min(top, int(ca * iv + nfh))), j = max(0, min(top, int(cb * iv + nfh)));
          const int face = 6 * int((nd.meta >> kMetaAxisShift) & 3u) + (mx ? 0 : (my ? 2 : 4)) +
                           (cm < 0.0f ? 1 : 0);
          sq = (face * a.beam_side + i) * a.beam_side + j;
          count = a.beam_count[sq * (kConeClasses + 1) + cls];
        }
      }
    }
    const uint4 near16 = *reinterpret_cast<const uint4*>(a.beam_list + sq * stride);
    const int incl = warp_incl_scan(count, lane);
    start = incl - count;
    total = __shfl_sync(0xffffffffu, incl, 31);
    const unsigned some = __ballot_sync(0xffffffffu, count > 0);
    if (count > 0) {
      const int slot = __popc(some & lt);
      box0[slot] = make_float4(lx, ly, lz, hx);
      box1[slot] = make_float4(hy, hz, __int_as_float((sq << 13) | start), __int_as_float(row));
      beams[slot] = near16;
    } else {
      start = -1;  // owns no pair: stays negative below, which is no bit
    }
    __syncwarp();
  }
  int owners = -1;  // the last cell whose pairs start before this chunk
  for (int p = lane; p - lane < total; p += 32, start -= 32) {
    // a lane's pair belongs to the last cell that starts at or before it
    const unsigned begins = __reduce_or_sync(0xffffffffu, bit_at(start));
    const int slot = owners + __popc(begins & (2u * lt + 1u));
    owners += __popc(begins);
    const float4 b0 = box0[slot], b1 = box1[slot];
    const int meta = __float_as_int(b1.z), i = p - (meta & 0x1fff);
    const bool live = p < total;
    int k = beams8[16 * slot + min(i, 15)];
    if (live && i > 15) k = a.beam_list[(meta >> 13) * stride + i];
    k = live ? k : 0;
    const float4 iv = binv[k];
    const float ax = b0.x * iv.x, bx = b0.w * iv.x;
    const float ay = b0.y * iv.y, by = b1.x * iv.y;
    const float az = b0.z * iv.z, bz = b1.y * iv.z;
    float t0 = fmaxf(fmaxf(fminf(ax, bx), fminf(ay, by)), fmaxf(fminf(az, bz), 0.0f));
    const float t1 = fminf(fminf(fmaxf(ax, bx), fmaxf(ay, by)), fmaxf(az, bz));
    if constexpr (kPP) t0 = fmaxf(t0, rpp);  // cells absorb only beyond r_pp (Sec. 2.4)
    const bool hit = live && t0 < fminf(t1, far[k]);
    push(hit, t0, t1, __float_as_int(b1.w), k);
  }
  __syncwarp();
}

// tau of the n staged sources V (sorted by beam and distance) from the nc
// listed cells, into T[e][NBP]: set with `first`, added to what is there
// without.  own[e][NBP]: the depth of the cell that holds a source, up to it.
template <int NBP, bool kPP, bool kInOrder, class Inside>
__device__ __forceinline__ void absorb_cells(const WalkArgs& a, float3 x, int lane, int* region,
                             const float4* binv, const int* off, float* far, const SrcEntry* V,
                             float* T, float* own, int n, const int* cells, int nc, bool first,
                             float rpp, Inside inside) {
  const unsigned lt = (1u << lane) - 1u;
  const int npix = a.npix;
  int* stage = region;
  float4* hits = reinterpret_cast<float4*>(region + kCellStage);
  float* ss = reinterpret_cast<float*>(hits + kCellHits / 4);
  if (first) {
    BandVec<NBP> zero;
#pragma unroll
    for (int b = 0; b < NBP; ++b) zero.v[b] = 0.0f;
    for (int e = lane; e < n; e += 32) {
      store_bands<NBP>(T + e * NBP, zero);
      store_bands<NBP>(own + e * NBP, zero);
    }
  }
  for (int e0 = 0; e0 < n; e0 += a.bin_cap) {
    const int m = min(a.bin_cap, n - e0);
    float* Tw = T + e0 * NBP;
    const float s_before = e0 ? V[e0 - 1].s : 0.0f;
    __syncwarp();
    for (int e = lane; e < m; e += 32) ss[e] = V[e0 + e].s;
    __syncwarp();
    for (int k = lane; k < npix; k += 32) {
      const int s0 = max((k ? off[k - 1] : 0) - e0, 0), s1 = min(off[k] - e0, m);
      far[beam_slot(k)] = s1 > s0 ? ss[s1 - 1] : -1.0f;
    }
    int head = 0;  // crossings found; the last head % 32 are pending, in a ring of 64
    int q_next = lane < nc ? cells[lane] : -1;
    for (int c0 = 0; c0 < nc; c0 += 32) {
      const int q = q_next;
      q_next = c0 + 32 + lane < nc ? cells[c0 + 32 + lane] : -1;
      cross_batch<kPP>(a, x, lane, q, stage, binv, far, rpp, [&](bool hit, float t0, float t1, int row, int k) {
        const unsigned hm = __ballot_sync(0xffffffffu, hit);
        if (hit)
          hits[(head + __popc(hm & lt)) & 63] =
              make_float4(t0, t1, __int_as_float(row), __int_as_float(k));
        const int was = head;
        head += __popc(hm);
        __syncwarp();
        if ((head ^ was) & 32)
          add_crossings<NBP, kInOrder>(a, lane, true, hits[(was & 32) + lane], binv, ss, off, e0, m,
                                       s_before, Tw, own + e0 * NBP, first,
                                       [&](int j, const BandVec<NBP>& al) { inside(e0 + j, al); });
      });
    }
    if (head & 31)
      add_crossings<NBP, kInOrder>(a, lane, lane < (head & 31), hits[(head & 32) + lane], binv, ss,
                                   off, e0, m, s_before, Tw, own + e0 * NBP, first,
                                   [&](int j, const BandVec<NBP>& al) { inside(e0 + j, al); });
  }
  __syncwarp();
}

// The increments of all cells summed along each beam, a beam per lane.
template <int NBP>
__device__ __forceinline__ void sum_increments(int lane, int npix, const int* off, float* T,
                                               const float* own, int lanes = 32) {
  for (int k = lane; k < npix; k += lanes) {
    BandVec<NBP> run;
#pragma unroll
    for (int b = 0; b < NBP; ++b) run.v[b] = 0.0f;
    for (int j = k ? off[k - 1] : 0; j < off[k]; ++j) {
      const BandVec<NBP> t = load_bands<NBP>(T + j * NBP);
      BandVec<NBP> o = load_bands<NBP>(own + j * NBP);
#pragma unroll
      for (int b = 0; b < NBP; ++b) {
        run.v[b] += t.v[b];
        o.v[b] += run.v[b];
      }
      store_bands<NBP>(T + j * NBP, o);
    }
  }
}

constexpr int kCellCap = 2048;  // cells of a cut listed at once
// The same, or fewer with trevr2_debug_set(TREVR2_DEBUG_CELL_CAP, c).
inline int cell_list_cap() { return std::min(kCellCap, debug_cell_cap()); }

// A warp's part of a walk block's shared memory and of the walk buffers.
struct WarpMem {
  int* stk;          // traversal stacks / increments, boxes and crossings
  int* lstk;         // this lane's stack (beam by beam)
  int* off;          // [npix] ends of the beams' buckets, then scratch
  int* order;        // [npix] beams by distance (beam by beam)
  int* next_beam;
  NodeW* chain;      // the receiver's ancestors (beam by beam)
  float* far;        // [npix] the beams' farthest sources (cell by cell)
  const float4* binv;  // [npix] the block's copy of 1 / direction (cell by cell)
  SrcEntry* U;
  int* Up;
  SrcEntry* V;
  float* T;
  float* own;        // [M][4] depth inside the cell that holds a source (cell by cell)
  int* cells;
};

template <bool kCells>
__device__ __forceinline__ WarpMem warp_mem(const WalkArgs& a, int* smem, int64_t gw,
                                            SrcEntry* srcU, int* pixU, SrcEntry* srcV, float* srcT,
                                            int* cells) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  WarpMem w;
  w.binv = reinterpret_cast<const float4*>(smem);
  int* wsm = smem + (kCells ? 4 * a.npix : 0) + wib * a.warp_ints;
  w.stk = wsm;
  w.lstk = wsm + lane * 2 * (a.max_depth + 2);
  w.off = wsm + a.region_ints;
  w.order = w.off + a.npix;
  w.far = reinterpret_cast<float*>(w.off + a.npix);
  w.next_beam = w.off + 2 * a.npix + 32;  // after the beam order and its counts
  w.chain = reinterpret_cast<NodeW*>(w.off + 2 * a.npix + 36);
  w.U = srcU + gw * a.M;
  w.Up = pixU + gw * a.M;
  w.V = srcV + gw * a.M;
  w.T = srcT + gw * a.M * 4;
  w.cells = cells + gw * (a.cell_cap + 4 * a.M);
  w.own = reinterpret_cast<float*>(w.cells + a.cell_cap);
  return w;
}

// Fills a walk block's shared tables.
template <bool kCells>
__device__ __forceinline__ void init_block(const WalkArgs& a, int* smem) {
  if constexpr (kCells) {
    float4* binv = reinterpret_cast<float4*>(smem);
    for (int k = threadIdx.x; k < a.npix; k += blockDim.x) binv[k] = a.beam_inv[k];
  }
  init_ext_tab();
}

}  // namespace trevr2
