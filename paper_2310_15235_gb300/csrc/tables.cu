// Per-direction absorption tables (TREVR2, Sec. 2.6, Eq. transmissionavg).
//
// For every internal cell and every antipodal pair of HEALPix beams
// (N_ray/2 stored values per cell, Sec. 2.6), the two halves are combined by
// the volume-weighted transmission
//   T = [V1 e^{-d a1} + V2 e^{-d a2} + V12 e^{-d a1/2} e^{-d a2/2}] / V,
//   alpha = -ln(T) / d,
// with V12 the volume of points whose line along the beam crosses the shared
// face inside the cell, V1 = V2 = V/2 - V12/2, and d the chord through the
// centre of the shared face (the cell centre).  The through-ray term is the
// product of the two half-cell transmissions: the printed sum of the two
// exponentials exceeds 1 for a transparent cell and contradicts the paper's
// own worked example.  Leaves are isotropic (bucket absorption).  With
// TREVR2_LINEAR the halves are combined by their volume-weighted linear
// average instead (Sec. 2.6's comparison scheme): (alpha_1 + alpha_2) / 2,
// the same in every direction pair.
//
// Cell shapes repeat every three levels (cube split on x; 1:2:2 split on y;
// 1:1:2 split on z), so the weights depend only on (depth mod 3, beam pair)
// and the chord scales with 2^-(depth/3): they are computed once per nside in
// FP64.  The combination runs in FP32 as
//   m > 1:  ln T = -m + ln(sum_j w_j e^{-(x_j - m)})      (no underflow)
//   m <= 1: ln T = log1p(sum_j w_j expm1(-x_j)) if T > 1/2 (thin cells keep
//           their relative precision), else ln(sum_j w_j e^{-x_j}),
// where x_j are the exponents of the terms and m the smallest one with a
// nonzero weight — the same expression, evaluated stably.
#include <algorithm>

#include "healpix.cuh"
#include "internal.cuh"

namespace trevr2 {

__device__ __forceinline__ void table_dir(int nside, int npix, int k, double* dirs64, float4* dirs) {
  double v[3];
  hp_pix2vec(nside, k, v);
  for (int a = 0; a < 3; ++a) __stcg(dirs64 + 3 * k + a, v[a]);
  int pair = k < npix / 2 ? k : hp_vec2pix_f64(nside, -v[0], -v[1], -v[2]);
  __stcg(dirs + k, make_float4(float(v[0]), float(v[1]), float(v[2]), __int_as_float(pair)));
}

// Transmission geometry of one cell shape (unit scale) for one beam pair.
__device__ __forceinline__ TransGeo table_geo(int shape, const double n[3]) {
  double E[3] = {1.0, 1.0, 1.0};
  if (shape >= 1) E[0] = 0.5;
  if (shape >= 2) E[1] = 0.5;
  const int a = shape, b = (a + 1) % 3, c = (a + 2) % 3;
  const double V = E[0] * E[1] * E[2];
  double V12 = 0.0;
  if (n[a] != 0.0) {
    // depth u below the shared face: the rays through points at u that reach
    // the face inside it cover (Lb - u rb)(Lc - u rc); integrate to u_max.
    const double rb = fabs(n[b] / n[a]), rc = fabs(n[c] / n[a]);
    const double Lb = E[b], Lc = E[c];
    double u = 0.5 * E[a];
    if (rb > 0.0) u = fmin(u, Lb / rb);
    if (rc > 0.0) u = fmin(u, Lc / rc);
    V12 = 2.0 * (Lb * Lc * u - 0.5 * (Lb * rc + Lc * rb) * u * u + rb * rc * u * u * u / 3.0);
  }
  double d = INFINITY;
  for (int k = 0; k < 3; ++k)
    if (n[k] != 0.0) d = fmin(d, E[k] / fabs(n[k]));
  TransGeo g;
  g.w1 = float((0.5 * V - 0.5 * V12) / V);
  g.w12 = float(V12 / V);
  g.d_unit = float(d);
  g.pad = 0.0f;
  return g;
}

// The unit vector through point (a, b) of face f of the cube [-1, 1]^3:
// f / 2 is the face's axis, odd f its negative side, (a, b) the other two
// axes in increasing order.
__device__ __forceinline__ void cube_vec(int f, float a, float b, float v[3]) {
  const int m = f >> 1;
  const float r = 1.0f / sqrtf(1.0f + a * a + b * b), s = (f & 1) ? -r : r;
  v[0] = m == 0 ? s : a * r;
  v[1] = m == 1 ? s : (m == 0 ? a * r : b * r);
  v[2] = m == 2 ? s : b * r;
}

// One cell shape (depth mod 3) and one square of the direction map per warp.
// A cell whose centre lies in the square, with half-diagonal over distance at
// most rho, is held by the box about the square's own direction with the
// shape's half-extents at rho, each widened by the square's range on that axis
// (1e-4 covers the FP32 arithmetic here and in the walk): the beams that cross
// that box are the cell's candidates.  They only grow with rho, so a beam's
// place is the first class (rho up to sin of the cone half-angle acos(1 -
// (c / kConeClasses)^2)) that has it, and a class's candidates are the first
// ones of the list.
template <int kGroups>
__global__ void k_beam_map(int npix, int stride, int nf, const float4* __restrict__ dirs,
                           uint8_t* __restrict__ list, uint8_t* __restrict__ count,
                           float4* __restrict__ beam_inv) {
  if (blockIdx.x == 0 && threadIdx.x < npix) {
    const float4 n = dirs[threadIdx.x];
    beam_inv[beam_slot(threadIdx.x)] =
        make_float4(n.x != 0.0f ? 1.0f / n.x : kFlatInv, n.y != 0.0f ? 1.0f / n.y : kFlatInv,
                    n.z != 0.0f ? 1.0f / n.z : kFlatInv, n.w);
  }
  const int id = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (id >= 18 * nf * nf) return;
  const int shape = id / (6 * nf * nf), sq = id % (6 * nf * nf);
  const int f = sq / (nf * nf), i = (sq / nf) % nf, j = sq % nf;
  const float w = 2.0f / nf;
  float c[3], half[3], wide[3];
  cube_vec(f, -1.0f + (i + 0.5f) * w, -1.0f + (j + 0.5f) * w, c);
  const float norm = rsqrtf((shape >= 1 ? 0.25f : 1.0f) + (shape >= 2 ? 0.25f : 1.0f) + 1.0f);
  half[0] = shape >= 1 ? 0.5f * norm : norm;
  half[1] = shape >= 2 ? 0.5f * norm : norm;
  half[2] = norm;
  for (int a = 0; a < 3; ++a) wide[a] = 1e-4f;
  for (int q = 0; q < 4; ++q) {  // no square straddles an axis: the corners are extreme
    float v[3];
    cube_vec(f, -1.0f + (i + (q & 1)) * w, -1.0f + (j + (q >> 1)) * w, v);
    for (int a = 0; a < 3; ++a) wide[a] = fmaxf(wide[a], fabsf(v[a] - c[a]) + 1e-4f);
  }
  int first[kGroups];
#pragma unroll
  for (int g = 0; g < kGroups; ++g) {
    const int k = 32 * g + lane;
    first[g] = kConeClasses + 2;  // no beam
    if (k >= npix) continue;
    const float4 n4 = dirs[k];
    const float n[3] = {n4.x, n4.y, n4.z};
    // crossing times of the widened box: (c -+ (rho half + wide)) / n
    float mid[3], grow[3], base[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float inv = n[a] != 0.0f ? 1.0f / n[a] : kFlatInv;
      mid[a] = c[a] * inv;
      grow[a] = half[a] * fabsf(inv);
      base[a] = wide[a] * fabsf(inv);
    }
    int lo = 1, hi = kConeClasses + 1;  // hi: only as one of all beams
    while (lo < hi) {
      const int m = (lo + hi) >> 1;
      const float u = float(m) / float(kConeClasses), cr = 1.0f - u * u;
      const float rho = sqrtf(fmaxf(0.0f, 1.0f - cr * cr));
      float t0 = 0.0f, t1 = INFINITY;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float e = fmaf(rho, grow[a], base[a]);
        t0 = fmaxf(t0, mid[a] - e);
        t1 = fminf(t1, mid[a] + e);
      }
      if (t0 <= t1) hi = m; else lo = m + 1;
    }
    first[g] = lo;
  }
  uint8_t* out = list + size_t(id) * stride;
  uint8_t* cnt = count + size_t(id) * (kConeClasses + 1);
  if (lane == 0) cnt[0] = 0;
  int base = 0;
  for (int cls = 1; cls <= kConeClasses + 1; ++cls) {
#pragma unroll
    for (int g = 0; g < kGroups; ++g) {
      const unsigned m = __ballot_sync(0xffffffffu, first[g] == cls);
      if (first[g] == cls)
        out[base + __popc(m & ((1u << lane) - 1u))] = uint8_t(beam_slot(32 * g + lane));
      base += __popc(m);
    }
    if (lane == 0 && cls <= kConeClasses) cnt[cls] = uint8_t(base);
  }
  for (int k = npix + lane; k < stride; k += 32) out[k] = 0;
}

__device__ __forceinline__ float combine_alpha(float a1, float a2, float w1, float w12, float d) {
  const float x1 = d * a1, x2 = d * a2, x12 = 0.5f * (x1 + x2);
  float m = INFINITY;
  if (w1 > 0.0f) m = fminf(x1, x2);
  if (w12 > 0.0f) m = fminf(m, x12);
  float lnT;
  if (m > 1.0f) {
    float S = 0.0f;
    if (w1 > 0.0f) S += w1 * (expf(-(x1 - m)) + expf(-(x2 - m)));
    if (w12 > 0.0f) S += w12 * expf(-(x12 - m));
    lnT = -m + logf(S);
  } else {
    // sum_j w_j = 1, so T - 1 comes without T
    float e = 0.0f;
    if (w1 > 0.0f) e += w1 * (expm1f(-x1) + expm1f(-x2));
    if (w12 > 0.0f) e += w12 * expm1f(-x12);
    if (e > -0.5f) {
      lnT = log1pf(e);
    } else {
      float S = 0.0f;
      if (w1 > 0.0f) S += w1 * (expf(-x1) + expf(-x2));
      if (w12 > 0.0f) S += w12 * expf(-x12);
      lnT = logf(S);
    }
  }
  return fmaxf(0.0f, -lnT / d);
}

// One table in one cooperative launch: beam directions, then the transmission
// geometry, then the cells' absorption one depth at a time, deepest first
// (a thread per cell and beam pair), with grid barriers between; runs of small
// depths stay in block 0.  A launch per depth cost the small trees more than
// the depths' work.  Values another block wrote are read past the L1.
struct TableArgs {
  int nside, npix, P, nb, levels;
  bool linear;
  const NodeW* nodes;
  const int* int_index;
  const float* alpha_leaf;
  double* dirs64;
  float4* dirs;
  TransGeo* geo;
  float* tab;
  uint32_t* bar;
  uint32_t* status;
  uint32_t polls;
  int level_begin[kMaxDepth + 3];
};
constexpr int kTableThreads = 512;
constexpr int64_t kTableSmall = 4 * kTableThreads;  // items of a depth that block 0 does alone

template <int NBP>
__device__ __forceinline__ void alpha_item(const TableArgs& A, int q, int p) {
  const NodeW nd = A.nodes[q];
  if (nd.child < 0) return;
  const int P = A.P;
  const int depth = int(nd.meta & kMetaDepthMask);
  const float4 gv = __ldcg(reinterpret_cast<const float4*>(A.geo) + (depth % 3) * P + p);
  const float d = ldexpf(gv.z, -(depth / 3));
  float a1[NBP], a2[NBP];
  const int c = nd.child;
  const int i1 = A.int_index[c], i2 = A.int_index[c + 1];
#pragma unroll
  for (int b = 0; b < NBP; ++b) {
    a1[b] = i1 < 0 ? A.alpha_leaf[int64_t(c) * NBP + b] : __ldcg(A.tab + (int64_t(i1) * P + p) * NBP + b);
    a2[b] = i2 < 0 ? A.alpha_leaf[int64_t(c + 1) * NBP + b] : __ldcg(A.tab + (int64_t(i2) * P + p) * NBP + b);
  }
  float* out = A.tab + (int64_t(nd.aux) * P + p) * NBP;
#pragma unroll
  for (int b = 0; b < NBP; ++b) {
    float al = 0.0f;
    if (b < A.nb && (a1[b] > 0.0f || a2[b] > 0.0f))
      al = A.linear ? 0.5f * (a1[b] + a2[b]) : combine_alpha(a1[b], a2[b], gv.x, gv.y, d);
    __stcg(out + b, al);
  }
}

template <int NBP>
__global__ void __launch_bounds__(kTableThreads, 2) k_tables(const __grid_constant__ TableArgs A) {
  const int blocks = gridDim.x, t = threadIdx.x, P = A.P;
  const int64_t stride = int64_t(blocks) * kTableThreads, at = int64_t(blockIdx.x) * kTableThreads + t;
  for (int64_t k = at; k < A.npix; k += stride) table_dir(A.nside, A.npix, int(k), A.dirs64, A.dirs);
  if (!grid_barrier(A.bar, blocks, A.status, A.polls, kStatusBarrier | kStatusTables)) return;
  for (int64_t i = at; i < 3 * P; i += stride) {
    const int p = int(i % P);
    const double n[3] = {__ldcg(A.dirs64 + 3 * p), __ldcg(A.dirs64 + 3 * p + 1), __ldcg(A.dirs64 + 3 * p + 2)};
    const TransGeo g = table_geo(int(i / P), n);
    __stcg(reinterpret_cast<float4*>(A.geo) + i, make_float4(g.w1, g.w12, g.d_unit, g.pad));
  }
  bool together = true;  // whether all blocks did what the next depth needs
  for (int d = A.levels - 2; d >= 0; --d) {  // the deepest depth has leaves only
    const int b0 = A.level_begin[d], b1 = A.level_begin[d + 1];
    const int64_t items = int64_t(b1 - b0) * P;
    const bool small = items <= kTableSmall;
    if (together || !small) {
      if (!grid_barrier(A.bar, blocks, A.status, A.polls, kStatusBarrier | kStatusTables)) return;
    } else {
      __syncthreads();
    }
    together = !small;
    if (small) {
      if (blockIdx.x == 0)
        for (int i = t; i < int(items); i += kTableThreads)
          alpha_item<NBP>(A, b0 + int(unsigned(i) / unsigned(P)), int(unsigned(i) % unsigned(P)));
    } else if (items < (int64_t(1) << 31)) {
      for (unsigned i = unsigned(at); i < unsigned(items); i += unsigned(stride))
        alpha_item<NBP>(A, b0 + int(i / unsigned(P)), int(i % unsigned(P)));
    } else {
      for (int64_t i = at; i < items; i += stride) alpha_item<NBP>(A, b0 + int(i / P), int(i % P));
    }
  }
}

int ensure_beam_map(Table* tb, cudaStream_t st) {
  if (tb->beam_list) return TREVR2_OK;
  const int npix = 12 * tb->nside * tb->nside, stride = (npix + 15) & ~15;
  const int nf = beam_map_side(tb->nside);
  const size_t squares = size_t(18) * nf * nf, inv_bytes = size_t(npix) * sizeof(float4);
  DeviceTemp<uint8_t> map(st);  // inverses, lists, counts
  T2_CHECK(device_alloc(reinterpret_cast<void**>(&map.p),
                        inv_bytes + squares * (stride + kConeClasses + 1), st, "beam map"));
  uint8_t* list = map.p + inv_bytes;
  uint8_t* count = list + squares * stride;
  // beams in groups of a warp's lanes: up to 64 (nside 1, 2) or 192 of them
  const auto fn = npix <= 64 ? &k_beam_map<2> : &k_beam_map<6>;
  fn<<<unsigned((squares + 7) / 8), 256, 0, st>>>(npix, stride, nf, tb->dirs, list, count,
                                                  reinterpret_cast<float4*>(map.p));
  note_launch();
  T2_CUDA(cudaGetLastError());
  tb->beam_inv = reinterpret_cast<float4*>(map.p);
  tb->beam_list = list;
  tb->beam_count = count;
  map.p = nullptr;
  return TREVR2_OK;
}

void free_table(Table* tb, cudaStream_t st) {
  dfree(tb->alpha, st);
  dfree(tb->dirs, st);
  dfree(tb->dirs64, st);
  dfree(tb->geo, st);
  dfree(tb->beam_inv, st);
  dfree(tb->csm_tau, st);
  dfree(tb->csm_d, st);
  dfree(tb->csm_anti, st);
}

void settle_tables(Tree* t, uint32_t s, cudaStream_t st) {
  const bool gave_up = (s & kStatusTables) != 0;
  for (size_t i = 0; i < t->tables.size();) {
    Table& tb = t->tables[i];
    if (gave_up && !tb.checked) {
      free_table(&tb, st);
      t->tables.erase(t->tables.begin() + i);
    } else {
      tb.checked = true;
      ++i;
    }
  }
}

int check_tables(Tree* t, cudaStream_t st) {
  bool all = true;
  for (const Table& tb : t->tables) all = all && tb.checked;
  if (all) return TREVR2_OK;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  T2_CUDA(cudaStreamIsCapturing(st, &capture));
  if (capture != cudaStreamCaptureStatusNone) return TREVR2_OK;
  uint32_t s = 0;
  T2_CUDA(cudaMemcpyAsync(&s, t->status, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
  T2_CUDA(cudaStreamSynchronize(st));
  settle_tables(t, s, st);
  if (!(s & kStatusTables)) return TREVR2_OK;
  const uint32_t rest = s & ~(kStatusBarrier | kStatusTables);
  T2_CUDA(cudaMemcpyAsync(t->status, &rest, sizeof(uint32_t), cudaMemcpyHostToDevice, st));
  T2_CUDA(cudaStreamSynchronize(st));
  set_error("trevr2: a grid barrier of the absorption tables' kernel gave up waiting");
  return TREVR2_ETIMEOUT;
}

int ensure_table(Tree* t, int nside, cudaStream_t st, Table** out, bool linear) {
  for (Table& tb : t->tables)
    if (tb.nside == nside && tb.linear == linear) {
      *out = &tb;
      return TREVR2_OK;
    }
  const int npix = 12 * nside * nside, P = npix / 2;
  // built in temporaries and kept by the tree only when complete
  DeviceTemp<float4> dirs(st);
  DeviceTemp<double> dirs64(st);
  DeviceTemp<TransGeo> geo(st);
  DeviceTemp<float> alpha(st);
  T2_CHECK(dalloc(&dirs.p, npix, st));
  T2_CHECK(dalloc(&dirs64.p, 3 * size_t(npix), st));
  T2_CHECK(dalloc(&geo.p, 3 * size_t(P), st));
  T2_CHECK(dalloc(&alpha.p, size_t(std::max<int64_t>(t->n_internal, 1)) * P * t->nbp, st));
  Table tb;
  tb.nside = nside;
  tb.linear = linear;
  tb.dirs = dirs.p;
  tb.dirs64 = dirs64.p;
  tb.geo = geo.p;
  tb.alpha = alpha.p;
  TableArgs A;
  A.nside = nside;
  A.npix = npix;
  A.P = P;
  A.nb = t->nb;
  A.levels = t->max_depth + 1;
  A.linear = linear;
  A.nodes = t->nodes;
  A.int_index = t->int_index;
  A.alpha_leaf = t->alpha_leaf;
  A.dirs64 = tb.dirs64;
  A.dirs = tb.dirs;
  A.geo = tb.geo;
  A.tab = tb.alpha;
  A.bar = t->status + 1;
  A.status = t->status;
  A.polls = barrier_polls();
  int64_t widest = npix;
  for (int d = 0; d <= t->max_depth + 1; ++d) {
    A.level_begin[d] = int(t->level_begin[d]);
    if (d) widest = std::max(widest, (t->level_begin[d] - t->level_begin[d - 1]) * P);
  }
  int blocks = 0;
  T2_CHECK(coop_blocks(widest, 2 * kTableThreads, 2, st, &blocks));
  T2_CUDA(cudaMemsetAsync(A.bar, 0, sizeof(uint32_t), st));
  const void* fn = t->nbp == 1 ? reinterpret_cast<const void*>(&k_tables<1>)
                 : t->nbp == 2 ? reinterpret_cast<const void*>(&k_tables<2>)
                               : reinterpret_cast<const void*>(&k_tables<4>);
  void* args[] = {&A};
  T2_CUDA(cudaLaunchCooperativeKernel(fn, dim3(unsigned(blocks)), dim3(kTableThreads), args, 0, st));
  note_launch();
  T2_CUDA(cudaGetLastError());
  t->tables.push_back(tb);
  dirs.p = nullptr;
  dirs64.p = nullptr;
  geo.p = nullptr;
  alpha.p = nullptr;
  *out = &t->tables.back();
  return TREVR2_OK;
}

__global__ void k_export_alpha(const NodeW* __restrict__ nodes, const int* __restrict__ int_index,
                               const float* __restrict__ alpha_leaf, const float* __restrict__ tab,
                               int64_t n, int P, int nb, int nbp, float scale, float* __restrict__ dst) {
  int64_t idx = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (idx >= n * P * nb) return;
  int64_t q = idx / (int64_t(P) * nb);
  int rem = int(idx % (int64_t(P) * nb));
  int p = rem / nb, b = rem % nb;
  int iq = int_index[q];
  float a = iq < 0 ? alpha_leaf[q * nbp + b] : tab[(int64_t(iq) * P + p) * nbp + b];
  dst[idx] = a * scale;
}

__global__ void k_pix2vec(int nside, int npix, double* __restrict__ dst) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= npix) return;
  double v[3];
  hp_pix2vec(nside, k, v);
  for (int a = 0; a < 3; ++a) dst[3 * k + a] = v[a];
}

// The walk's pixel lookup: FP32 with a guard band, FP64 when inside it.
__global__ void k_vec2pix(int nside, const double* __restrict__ v, int64_t n, int32_t* __restrict__ pix) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  double x = v[3 * i], y = v[3 * i + 1], z = v[3 * i + 2];
  float fx = float(x), fy = float(y), fz = float(z);
  float r = sqrtf(fx * fx + fy * fy + fz * fz);
  int p = hp_vec2pix_f32(nside, fx, fy, fz, hp_guard(nside, r));
  if (p < 0) p = hp_vec2pix_f64(nside, x, y, z);
  pix[i] = p;
}

static bool valid_nside(int nside) {
  return nside >= 1 && nside <= TREVR2_MAX_NSIDE && (nside & (nside - 1)) == 0;
}

}  // namespace trevr2

using namespace trevr2;

extern "C" int trevr2_alpha_table(trevr2_tree* tree, int nside, float* dst, size_t bytes,
                                  void* stream) {
  clear_error();
  if (!tree || !dst) {
    set_error("trevr2_alpha_table: NULL argument");
    return TREVR2_EINVAL;
  }
  if (!valid_nside(nside)) {
    set_error("trevr2_alpha_table: nside %d is not a power of two in [1, %d]", nside, TREVR2_MAX_NSIDE);
    return TREVR2_EINVAL;
  }
  Tree* t = reinterpret_cast<Tree*>(tree);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  t->last_stream = st;
  const int P = 6 * nside * nside;
  const size_t need = size_t(t->n_nodes) * P * t->nb * sizeof(float);
  if (bytes < need) {
    set_error("trevr2_alpha_table: destination holds %zu bytes, %zu needed", bytes, need);
    return TREVR2_EINVAL;
  }
  Table* tb = nullptr;
  T2_CHECK(ensure_table(t, nside, st, &tb));
  T2_CHECK(check_tables(t, st));
  int64_t total = t->n_nodes * int64_t(P) * t->nb;
  if (total > 0)
    k_export_alpha<<<unsigned((total + 255) / 256), 256, 0, st>>>(
        t->nodes, t->int_index, t->alpha_leaf, tb->alpha, t->n_nodes, P, t->nb, t->nbp,
        float(1.0 / t->size), dst); note_launch();
  T2_CUDA(cudaGetLastError());
  return TREVR2_OK;
}

extern "C" int trevr2_healpix_pix2vec(int nside, double* dst, void* stream) {
  clear_error();
  if (!dst || !valid_nside(nside)) {
    set_error("trevr2_healpix_pix2vec: NULL destination or bad nside %d", nside);
    return TREVR2_EINVAL;
  }
  int npix = 12 * nside * nside;
  k_pix2vec<<<(npix + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(nside, npix, dst); note_launch();
  T2_CUDA(cudaGetLastError());
  return TREVR2_OK;
}

extern "C" int trevr2_healpix_vec2pix(int nside, const double* v, int64_t n, int32_t* pix, void* stream) {
  clear_error();
  if (n < 0 || (n > 0 && (!v || !pix)) || !valid_nside(nside)) {
    set_error("trevr2_healpix_vec2pix: bad arguments (nside %d, n %lld)", nside, (long long)n);
    return TREVR2_EINVAL;
  }
  if (n > 0)
    k_vec2pix<<<unsigned((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(nside, v, n, pix); note_launch();
  T2_CUDA(cudaGetLastError());
  return TREVR2_OK;
}
