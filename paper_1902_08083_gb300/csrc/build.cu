// Radiation-tree build on the GPU (Grond et al. 2019, Sec. 2.2 and 2.3):
// Morton keys -> stable radix sort (sort.cu) -> binary tree of Morton prefixes (topology.cu) ->
// source deposit -> bottom-up cell moments. The host synchronises once, when the cuts are known
// and so the number of cells, to allocate the cells and size the moment pass.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>

#include "morton.cuh"
#include "primitives.cuh"
#include "topology.cuh"
#include "trevr_internal.cuh"

namespace trevr {

// ------------------------------------------------------------------------------------
// Morton keys
// ------------------------------------------------------------------------------------
__global__ void keys_kernel(const float* __restrict__ xyz, const float* __restrict__ alpha,
                            const float* __restrict__ weight, int n, Domain32 D,
                            unsigned long long* __restrict__ keys, unsigned* __restrict__ vals,
                            int* status) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float x = xyz[i], y = xyz[(size_t)n + i], z = xyz[2 * (size_t)n + i];
  int bad = 0;
  unsigned long long k = 0;
  if (in_dom(x, D.lo[0], D.hi[0]) && in_dom(y, D.lo[1], D.hi[1]) && in_dom(z, D.lo[2], D.hi[2])) {
    k = (expand3(quantize(x, D.lo[0], D.scale)) << 2) |
        (expand3(quantize(y, D.lo[1], D.scale)) << 1) | expand3(quantize(z, D.lo[2], D.scale));
  } else {
    bad |= kStatusOutOfDomain;
  }
  float a = alpha[i];
  if (!(a >= 0.0f) || !isfinite(a)) bad |= kStatusInvalid;
  if (weight) {
    float wv = weight[i];
    if (!(wv > 0.0f) || !isfinite(wv)) bad |= kStatusInvalid;
  }
  if (bad) atomicOr(status, bad);
  keys[i] = k;
  vals[i] = (unsigned)i;
}

// ------------------------------------------------------------------------------------
// Sinks of a call in Morton order
// ------------------------------------------------------------------------------------
__global__ void sink_keys_kernel(const long long* __restrict__ sink_idx, int n, int n_gas,
                                 const int* __restrict__ rank,
                                 unsigned long long* __restrict__ keys, unsigned* __restrict__ vals) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const long long si = sink_idx[k];
  keys[k] = si >= 0 && si < n_gas ? (unsigned long long)rank[si] : (unsigned long long)n_gas;
  vals[k] = (unsigned)k;
}

namespace {
constexpr size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }
}

size_t sink_order_bytes(int n) {
  return 2 * align256((size_t)n * 8) + align256((size_t)n * 4) + align256(sort_work_words(n) * 4);
}

bool sink_order(const trevr_tree* t, const long long* sink_idx, int n, void* scratch,
                unsigned* order, cudaStream_t s) {
  unsigned char* p = static_cast<unsigned char*>(scratch);
  auto take = [&](size_t bytes) {
    void* q = p;
    p += align256(bytes);
    return q;
  };
  unsigned long long* keys = static_cast<unsigned long long*>(take((size_t)n * 8));
  SortScratch S;
  S.k2 = static_cast<unsigned long long*>(take((size_t)n * 8));
  S.v2 = static_cast<unsigned*>(take((size_t)n * 4));
  S.work = static_cast<unsigned*>(take(sort_work_words(n) * 4));
  S.size = (size_t)n;
  S.words = sort_work_words(n);
  const int n_gas = (int)t->n_gas;
  sink_keys_kernel<<<(n + 255) / 256, 256, 0, s>>>(sink_idx, n, n_gas, t->rank, keys, order);
  note_launch();
  int bits = 1;  // keys are ranks, and n_gas itself
  while (bits < 31 && (n_gas >> bits)) ++bits;
  return radix_sort(keys, order, n, bits, S, t->status, s);
}

// ------------------------------------------------------------------------------------
// Particle gather into Morton order
// ------------------------------------------------------------------------------------
// Sorted particles: position relative to the domain's lower corner (u = x - lo, one
// fp32 rounding; the frame of every fp32 decision, in which the cell planes are
// g * h), and alpha.
__global__ void gather_particles_kernel(const float* __restrict__ xyz,
                                        const float* __restrict__ alpha,
                                        const float* __restrict__ weight, int n, Domain32 D,
                                        const unsigned* __restrict__ order, float4* pos, float* w,
                                        int* perm, int* rank) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int o = (int)min(order[i], (unsigned)(n - 1));  // any number if the sort gave up
  pos[i] = make_float4(__fsub_rn(xyz[o], D.lo[0]), __fsub_rn(xyz[(size_t)n + o], D.lo[1]),
                       __fsub_rn(xyz[2 * (size_t)n + o], D.lo[2]), alpha[o]);
  w[i] = weight ? weight[o] : 1.0f;
  perm[i] = o;
  rank[o] = i;
}

// ------------------------------------------------------------------------------------
// Sources: leaf of each source (descend by the cut planes), sort, ranges
// ------------------------------------------------------------------------------------
__global__ void src_leaf_kernel(const float* __restrict__ xyz, const float* __restrict__ lum,
                                int n_src, Domain32 D, const int4* __restrict__ nT,
                                const int4* __restrict__ nglo, const int* __restrict__ nfirst,
                                unsigned long long* keys, unsigned* vals, int* status) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n_src) return;
  float x = xyz[s], y = xyz[(size_t)n_src + s], z = xyz[2 * (size_t)n_src + s];
  float L = lum[s];
  if (!(L >= 0.0f) || !isfinite(L)) atomicOr(status, kStatusInvalid);
  if (!(in_dom(x, D.lo[0], D.hi[0]) && in_dom(y, D.lo[1], D.hi[1]) &&
        in_dom(z, D.lo[2], D.hi[2]))) {
    atomicOr(status, kStatusOutOfDomain);
    keys[s] = 0;
    vals[s] = (unsigned)s;
    return;
  }
  int g[3] = {(int)quantize(x, D.lo[0], D.scale), (int)quantize(y, D.lo[1], D.scale),
              (int)quantize(z, D.lo[2], D.scale)};
  int X = kRoot;
  for (int it = 0; it < kMaxLevels; ++it) {
    int child = nT[X].x;
    if (child < 0) break;
    int a = nglo[X].w;
    int4 up = nglo[child + 1];
    int plane = a == 0 ? up.x : (a == 1 ? up.y : up.z);
    X = g[a] >= plane ? child + 1 : child;
  }
  keys[s] = (unsigned long long)nfirst[X];
  vals[s] = (unsigned)s;
}

// sources sorted by leaf, positions relative to the domain's lower corner
__global__ void gather_sources_kernel(const float* __restrict__ xyz, const float* __restrict__ lum,
                                      int n_src, int n_gas, Domain32 D,
                                      const unsigned* __restrict__ order,
                                      const unsigned long long* __restrict__ leaf_first,
                                      const int* __restrict__ leaf_of, float4* src, int* src_order,
                                      int* src_leaf) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n_src) return;
  const int o = (int)min(order[k], (unsigned)(n_src - 1));  // any number if the sort gave up
  src[k] = make_float4(__fsub_rn(xyz[o], D.lo[0]), __fsub_rn(xyz[(size_t)n_src + o], D.lo[1]),
                       __fsub_rn(xyz[2 * (size_t)n_src + o], D.lo[2]), lum[o]);
  src_order[k] = o;
  // the leaf that starts at that particle
  src_leaf[k] = leaf_of[min(leaf_first[k], (unsigned long long)(n_gas - 1))];
}

__device__ __forceinline__ int lower_bound_u64(const unsigned long long* a, int n,
                                               unsigned long long v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    int m = lo + ((hi - lo) >> 1);
    if (a[m] < v) lo = m + 1;
    else hi = m;
  }
  return lo;
}

__global__ void node_src_range_kernel(int n_cells_end, const int* __restrict__ nfirst,
                                      const int* __restrict__ ncount,
                                      const unsigned long long* __restrict__ src_keys, int n_src,
                                      int4* nT, unsigned* arrived) {
  int X = blockIdx.x * blockDim.x + threadIdx.x + kRoot;
  if (X >= n_cells_end) return;
  int a = lower_bound_u64(src_keys, n_src, (unsigned long long)nfirst[X]);
  int b = lower_bound_u64(src_keys, n_src, (unsigned long long)(nfirst[X] + ncount[X]));
  nT[X].z = a;
  nT[X].w = b - a;
  arrived[X] = 0;  // for the climb of the moments
}

// ------------------------------------------------------------------------------------
// Cell moments, bottom-up. FP64 sums; explicit round-to-nearest
// operations so that no multiply-add is contracted and the directional
// alpha_min/alpha_max follow the same operation order as their definition.
// ------------------------------------------------------------------------------------
struct __align__(16) Moments {
  double W, WA, L, LY[3], amin[3], amax[3];
};

struct MomentArrays {
  const int4* nT;
  const int4* nglo;
  const int4* nghi;
  const int* nfirst;
  const int* ncount;
  const float4* pos;
  const float* w;
  const float4* src;
  const int* levels;
  Moments* mom;
  double* nW;
  float4* nA;
  float4* nB;
  float4* nS;
  float* nl2;
  float4* nR;
  float4* nV;
  float h;
};

// a grid plane relative to the domain's lower corner: g * h, rounded once
__device__ __forceinline__ float rel_plane(float h, int g) { return __fmul_rn((float)g, h); }

// a cell's moments, which another block may have written in this launch
__device__ __forceinline__ Moments load_moments(const Moments* p) {
  static_assert(sizeof(Moments) == 6 * sizeof(double2), "six 16-byte loads");
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 a = __ldcg(q), b = __ldcg(q + 1), c = __ldcg(q + 2), d = __ldcg(q + 3),
                e = __ldcg(q + 4), f = __ldcg(q + 5);
  return Moments{a.x, a.y, b.x, {b.y, c.x, c.y}, {d.x, d.y, e.x}, {e.y, f.x, f.y}};
}

// the moments of one cell, from its particles and sources (a leaf) or from its two children
// (whose moments are complete)
__device__ __forceinline__ Moments cell_moments(const MomentArrays& A, int X) {
  const int4 t = A.nT[X];
  Moments m;
  if (t.x < 0) {
    double sw = 0.0, swa = 0.0;
    const int f = A.nfirst[X], c = A.ncount[X];
    for (int i = f; i < f + c; ++i) {
      double wi = (double)A.w[i];
      sw = __dadd_rn(sw, wi);
      swa = __dadd_rn(swa, __dmul_rn(wi, (double)A.pos[i].w));
    }
    double sl = 0.0, sy0 = 0.0, sy1 = 0.0, sy2 = 0.0;
    for (int s = t.z; s < t.z + t.w; ++s) {
      float4 y = A.src[s];
      double Lj = (double)y.w;
      sl = __dadd_rn(sl, Lj);
      sy0 = __dadd_rn(sy0, __dmul_rn(Lj, (double)y.x));
      sy1 = __dadd_rn(sy1, __dmul_rn(Lj, (double)y.y));
      sy2 = __dadd_rn(sy2, __dmul_rn(Lj, (double)y.z));
    }
    m.W = sw;
    m.WA = swa;
    m.L = sl;
    m.LY[0] = sy0;
    m.LY[1] = sy1;
    m.LY[2] = sy2;
    const double ab = __ddiv_rn(swa, sw);
#pragma unroll
    for (int d = 0; d < 3; ++d) m.amin[d] = m.amax[d] = ab;
    return m;
  }
  const int4 lX = A.nglo[X], hX = A.nghi[X], l2 = A.nglo[t.x + 1];
  const Moments m1 = load_moments(&A.mom[t.x]);
  const Moments m2 = load_moments(&A.mom[t.x + 1]);
  m.W = __dadd_rn(m1.W, m2.W);
  m.WA = __dadd_rn(m1.WA, m2.WA);
  m.L = __dadd_rn(m1.L, m2.L);
  const int a = lX.w;
  const int lo = a == 0 ? lX.x : (a == 1 ? lX.y : lX.z);
  const int hi = a == 0 ? hX.x : (a == 1 ? hX.y : hX.z);
  const int cut = a == 0 ? l2.x : (a == 1 ? l2.y : l2.z);
  const double w1 = (double)(cut - lo), w2 = (double)(hi - cut), Wd = (double)(hi - lo);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    m.LY[d] = __dadd_rn(m1.LY[d], m2.LY[d]);
    // across the cut: one child or the other
    m.amin[d] = fmin(m1.amin[d], m2.amin[d]);
    m.amax[d] = fmax(m1.amax[d], m2.amax[d]);
    if (d == a) {
      // the ray crosses both children: optical depths add, divide by the width
      m.amin[d] = __ddiv_rn(__dadd_rn(__dmul_rn(m1.amin[d], w1), __dmul_rn(m2.amin[d], w2)), Wd);
      m.amax[d] = __ddiv_rn(__dadd_rn(__dmul_rn(m1.amax[d], w1), __dmul_rn(m2.amax[d], w2)), Wd);
    }
  }
  return m;
}

// the walk records of one cell
__device__ __forceinline__ void cell_records(const MomentArrays& A, int X, const Moments& m) {
  A.nW[X] = m.W;
  const double amin = fmin(fmin(m.amin[0], m.amin[1]), m.amin[2]);
  const double amax = fmax(fmax(m.amax[0], m.amax[1]), m.amax[2]);
  const float abar = __double2float_rn(__ddiv_rn(m.WA, m.W));
  const float dal = __double2float_rn(__dsub_rn(amax, amin));
  const float Lf = __double2float_rn(m.L);
  const int4 gl = A.nglo[X], gh = A.nghi[X];
  const float blo[3] = {rel_plane(A.h, gl.x), rel_plane(A.h, gl.y), rel_plane(A.h, gl.z)};
  const float bhi[3] = {rel_plane(A.h, gh.x), rel_plane(A.h, gh.y), rel_plane(A.h, gh.z)};
  float c[3], l2 = 0.0f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    c[d] = m.L > 0.0 ? __double2float_rn(__ddiv_rn(m.LY[d], m.L)) : 0.0f;
    const float e = fmaxf(__fsub_rn(c[d], blo[d]), __fsub_rn(bhi[d], c[d]));
    l2 = __fadd_rn(l2, __fmul_rn(e, e));
  }
  A.nA[X] = make_float4(blo[0], blo[1], blo[2], abar);
  A.nB[X] = make_float4(bhi[0], bhi[1], bhi[2], dal);
  A.nS[X] = make_float4(c[0], c[1], c[2], Lf);
  A.nl2[X] = l2;
  const int child = A.nT[X].x, ax = gl.w;
  float plane = 0.0f;
  unsigned link = 3u, below = 0u;  // a leaf
  if (child >= 0) {
    const int4 u = A.nglo[child + 1];
    plane = rel_plane(A.h, ax == 0 ? u.x : (ax == 1 ? u.y : u.z));
    link = ((unsigned)child >> 1) << 2 | (unsigned)ax;  // children are the pair (2k, 2k + 1)
    below = (unsigned)child | (__double2float_rn(__ldcg(&A.mom[child].L)) > 0.0f ? 1u << 31 : 0u) |
            (__double2float_rn(__ldcg(&A.mom[child + 1].L)) > 0.0f ? 1u : 0u);
  }
  A.nV[2 * (size_t)X] = make_float4(blo[0], blo[1], blo[2], l2);
  A.nV[2 * (size_t)X + 1] = make_float4(bhi[0], bhi[1], bhi[2], __uint_as_float(below));
  A.nR[X] = make_float4(abar, dal, plane, __uint_as_float(link));
  if (X == kRoot) {  // entry 0: an empty leaf without light
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    A.nA[0] = A.nB[0] = A.nS[0] = A.nV[0] = A.nV[1] = zero;
    A.nR[0] = make_float4(0.0f, 0.0f, 0.0f, __uint_as_float(3u));
    A.nl2[0] = 0.0f;
    A.nW[0] = 0.0;
  }
}

// The moments of the levels up to the one that ends at `end`, whose lower levels are done: a
// thread per leaf, and per internal cell of that last level, then up while it is the second
// child to be done. No thread waits: the first to arrive at a cell ends there. The chain to the
// root is what this costs, so the records are another launch's.
__global__ void moments_climb_kernel(MomentArrays A, int last_begin, int end, unsigned* arrived) {
  int X = kRoot + blockIdx.x * blockDim.x + threadIdx.x;
  if (X >= end || (X < last_begin && A.nT[X].x >= 0)) return;
  while (true) {
    A.mom[X] = cell_moments(A, X);
    if (X == kRoot) return;
    const int up = A.nT[X].y;
    __threadfence();
    if (atomicAdd(&arrived[up], 1u) == 0) return;
    __threadfence();
    X = up;
  }
}

__global__ void records_kernel(MomentArrays A, int end) {
  const int X = kRoot + blockIdx.x * blockDim.x + threadIdx.x;
  if (X < end) cell_records(A, X, A.mom[X]);
}

__global__ void moments_level_kernel(MomentArrays A, int L) {
  const int begin = A.levels[2 * L], end = A.levels[2 * L + 1];
  for (int X = begin + blockIdx.x * blockDim.x + threadIdx.x; X < end;
       X += gridDim.x * blockDim.x) {
    const Moments m = cell_moments(A, X);
    A.mom[X] = m;
    cell_records(A, X, m);
  }
}

// ------------------------------------------------------------------------------------
// Host driver
// ------------------------------------------------------------------------------------
namespace {

// Arrays laid out one behind another, 256 bytes apart, in one block of the pool: a first pass
// over the layout adds up the sizes, a second hands out the addresses. A build made 35
// allocations and its tree's end 36 frees, about 100 us of host time, on the way of the next
// step's first launch.
struct Layout {
  char* base;
  size_t at;
  template <class T>
  void get(T*& p, size_t n) {
    p = base ? reinterpret_cast<T*>(base + at) : nullptr;
    at += ((n ? n : 1) * sizeof(T) + 255) & ~(size_t)255;
  }
};

template <class F>
void* allocate(const F& arrays, cudaStream_t s) {
  Layout sizes{nullptr, 0};
  arrays(sizes);
  void* p = nullptr;
  if (pool_malloc_async(&p, sizes.at, s) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  Layout places{static_cast<char*>(p), 0};
  arrays(places);
  return p;
}

inline int grid_for(long long n, int threads) { return (int)((n + threads - 1) / threads); }

}  // namespace

// Levels with up to so many cells in all are summed by one climbing launch; the levels below
// them, where a level fills the GPU, by a launch each. A build at 4096 / 2^18 / 2^20 / 2^22
// particles takes 285 / 455 / 693 / 1630 us with this line, 333 / 534 / 750 / 1678 with a launch
// for every level, 278 / 453 / 682 / 1696 with climbing only.
constexpr int kClimbCells = 131072;

int build_tree_impl(const float* gas_xyz, const float* alpha, const float* weight, long long n_gas_ll,
                    const float* src_xyz, const float* src_lum, long long n_src_ll,
                    const trevr_domain* dom, int bucket, cudaStream_t s, trevr_tree** out) {
  const int n = (int)n_gas_ll;
  const int ns = (int)n_src_ll;
  trevr_tree* t = new trevr_tree();
  std::memset(t, 0, sizeof(*t));
  cudaGetDevice(&t->device);
  t->n_gas = n;
  t->n_src = ns;
  t->bucket = bucket;
  for (int d = 0; d < 3; ++d) t->lo[d] = dom->lo[d];
  t->side = dom->side;
  {
    volatile float side = dom->side;  // fp32 on the host, as on the device
    t->h = side * (1.0f / 2097152.0f);
  }
  const int nmax = n > ns ? n : ns;
  unsigned *vals, *topo_scan, *svals;
  unsigned long long* skeys;
  SortScratch SS;
  SS.size = (size_t)nmax;
  // (not monotone: a smaller sort may have more tiles)
  SS.words = std::max(sort_work_words(n), sort_work_words(ns));
  TopoArrays TA;
  t->mem[0] = allocate(
      [&](Layout& a) {
        a.get(t->key, n);
        a.get(t->perm, n);
        a.get(t->rank, n);
        a.get(t->leaf_of, n);
        a.get(t->pos, n);
        a.get(t->w, n);
        a.get(t->src, ns);
        a.get(t->src_order, ns);
        a.get(t->src_leaf, ns);
        a.get(t->levels, 2 * kMaxLevels);
        a.get(t->d_stats, 9);  // and the status word
      },
      s);
  void* scratch = allocate(
      [&](Layout& a) {
        a.get(vals, n);
        a.get(SS.k2, SS.size);
        a.get(SS.v2, SS.size);
        a.get(SS.work, SS.words);
        a.get(TA.up, n);
        a.get(TA.range, n);
        a.get(TA.bit, n);
        a.get(TA.depth, n);
        a.get(TA.place, n);
        a.get(TA.list, n);
        a.get(TA.counts, topo_count_words(n));
        a.get(topo_scan, scan_scratch_words((int)topo_count_words(n)));
        a.get(skeys, ns);
        a.get(svals, ns);
      },
      s);
  void* sums = nullptr;  // the moments, later

  auto release = [&]() {  // the scratch blocks
    if (scratch) cudaFreeAsync(scratch, s);
    if (sums) cudaFreeAsync(sums, s);
    scratch = sums = nullptr;
  };
  auto fail = [&](int code) {
    release();
    for (void* p : t->mem)
      if (p) cudaFreeAsync(p, s);
    cudaStreamSynchronize(s);
    delete t;
    return code;
  };
  if (!t->mem[0] || !scratch) return fail(TREVR_ERR_OUT_OF_MEMORY);
  t->status = reinterpret_cast<int*>(t->d_stats + 8);
  cudaMemsetAsync(t->d_stats, 0, 9 * sizeof(unsigned long long), s);

  Domain32 D;
  for (int d = 0; d < 3; ++d) {
    volatile float lo = dom->lo[d], side = dom->side;
    D.lo[d] = lo;
    D.hi[d] = lo + side;
  }
  {
    volatile float side = dom->side;
    D.scale = 2097152.0f / side;
  }
  D.h = t->h;

  // 1. keys and sort
  keys_kernel<<<grid_for(n, 256), 256, 0, s>>>(gas_xyz, alpha, weight, n, D, t->key, vals,
                                                 t->status);
  note_launch();
  if (!radix_sort(t->key, vals, n, 63, SS, t->status, s)) return fail(TREVR_ERR_CUDA);
  gather_particles_kernel<<<grid_for(n, 256), 256, 0, s>>>(gas_xyz, alpha, weight, n, D, vals,
                                                            t->pos, t->w, t->perm, t->rank);
  note_launch();
  // 2. topology
  TA.n = n;
  TA.bucket = bucket;
  TA.key = t->key;
  TA.status = t->status;
  TA.leaf_of = t->leaf_of;
  TA.levels = t->levels;
  launch_cuts(TA, topo_scan, s);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return fail(cuda_to_error(err));
  int levels[2 * kMaxLevels];
  cudaMemcpyAsync(levels, t->levels, sizeof(levels), cudaMemcpyDeviceToHost, s);
  err = cudaStreamSynchronize(s);
  if (err != cudaSuccess) return fail(cuda_to_error(err));
  if (levels[1] <= levels[0]) return fail(TREVR_ERR_ITERATION_LIMIT);
  int max_depth = 0;
  for (int L = 0; L < kMaxLevels; ++L)
    if (levels[2 * L + 1] > levels[2 * L]) max_depth = L;
  const int end_cells = levels[2 * max_depth + 1];
  t->n_nodes = end_cells - kRoot;
  t->max_depth = max_depth;
  for (int l = 0; l < 2 * kMaxLevels; ++l) t->h_levels[l] = levels[l];

  const size_t ncell = (size_t)end_cells;
  Moments* mom;
  unsigned* arrived;
  t->mem[1] = allocate(
      [&](Layout& a) {
        a.get(t->nfirst, ncell);
        a.get(t->ncount, ncell);
        a.get(t->nglo, ncell);
        a.get(t->nghi, ncell);
        a.get(t->nT, ncell);
        a.get(t->ndepth, ncell);
        a.get(t->nD, ncell);
        a.get(t->nA, ncell);
        a.get(t->nB, ncell);
        a.get(t->nS, ncell);
        a.get(t->nl2, ncell);
        a.get(t->nR, ncell);
        a.get(t->nV, 2 * ncell);
        a.get(t->nW, ncell);
      },
      s);
  sums = allocate(
      [&](Layout& a) {
        a.get(mom, ncell);
        a.get(arrived, ncell);
      },
      s);
  if (!t->mem[1] || !sums) return fail(TREVR_ERR_OUT_OF_MEMORY);
  TA.nfirst = t->nfirst;
  TA.ncount = t->ncount;
  TA.nglo = t->nglo;
  TA.nghi = t->nghi;
  TA.nT = t->nT;
  TA.ndepth = t->ndepth;
  TA.nD = t->nD;
  launch_cells(TA, s);

  // 3. sources
  if (ns > 0) {
    src_leaf_kernel<<<grid_for(ns, 256), 256, 0, s>>>(src_xyz, src_lum, ns, D, t->nT, t->nglo,
                                                       t->nfirst, skeys, svals, t->status);
    note_launch();
    int bits = 1;  // keys are particle numbers
    while (bits < 31 && ((n - 1) >> bits)) ++bits;
    if (!radix_sort(skeys, svals, ns, bits, SS, t->status, s)) return fail(TREVR_ERR_CUDA);
    gather_sources_kernel<<<grid_for(ns, 256), 256, 0, s>>>(src_xyz, src_lum, ns, n, D, svals,
                                                             skeys, t->leaf_of, t->src,
                                                             t->src_order, t->src_leaf);
    note_launch();
  }
  node_src_range_kernel<<<grid_for(end_cells - kRoot, 256), 256, 0, s>>>(
      end_cells, t->nfirst, t->ncount, skeys, ns, t->nT, arrived);
  note_launch();
  // 4. moments, bottom-up
  MomentArrays MA;
  MA.nT = t->nT;
  MA.nglo = t->nglo;
  MA.nghi = t->nghi;
  MA.nfirst = t->nfirst;
  MA.ncount = t->ncount;
  MA.pos = t->pos;
  MA.w = t->w;
  MA.src = t->src;
  MA.levels = t->levels;
  MA.mom = mom;
  MA.nW = t->nW;
  MA.nA = t->nA;
  MA.nB = t->nB;
  MA.nS = t->nS;
  MA.nl2 = t->nl2;
  MA.nR = t->nR;
  MA.nV = t->nV;
  MA.h = t->h;
  int climb = 0;  // the lowest level of the climbing launch
  while (climb < max_depth && levels[2 * climb + 3] <= kClimbCells) ++climb;
  for (int L = max_depth; L > climb; --L) {
    int m = levels[2 * L + 1] - levels[2 * L];
    int blocks = grid_for(m, 128);
    if (blocks > 4096) blocks = 4096;
    moments_level_kernel<<<blocks, 128, 0, s>>>(MA, L);
    note_launch();
  }
  moments_climb_kernel<<<grid_for(levels[2 * climb + 1] - kRoot, 64), 64, 0, s>>>(
      MA, levels[2 * climb], levels[2 * climb + 1], arrived);
  records_kernel<<<grid_for(levels[2 * climb + 1] - kRoot, 128), 128, 0, s>>>(
      MA, levels[2 * climb + 1]);
  note_launch(2);
  release();
  int status = 0;
  cudaMemcpyAsync(&status, t->status, sizeof(int), cudaMemcpyDeviceToHost, s);
  err = cudaStreamSynchronize(s);
  if (err == cudaSuccess) err = cudaGetLastError();
  if (err != cudaSuccess) return fail(cuda_to_error(err));
  if (status) return fail(status_to_error(status));
  *out = t;
  return TREVR_OK;
}

}  // namespace trevr
