// Tree topology from the sorted Morton keys, without a pass per level.
//
// Every pair of neighbouring particles with different keys is a possible cut: the cell that it
// cuts holds the particles that share the key bits above the highest one in which the pair
// differs (the ranges of a binary radix tree, as Karras's parallel construction finds them).
// A cut is kept if its cell holds more than bucket particles. A cut's parent is the cut at
// either end of its range, the one of the lower bit, so each cut climbs to the root by itself:
// its depth, the path, and on each axis the nearest planes above it give its cell.
//   cut_kernel    range, bit and parent of every cut                      (one thread a pair)
//   depth_kernel  depth of the kept cuts, counted by depth in tiles of the particle order
//   a prefix sum over (depth, tile)
//   place_kernel  breadth-first place of each kept cut: by depth, then by particle order; and
//                 the levels' ranges of cells, which the host needs to allocate the cells
//   cell_kernel   the cell of each kept cut and its children that are leaves, whole records
// The children of the cut at place P are the cells 2 + 2 P and 3 + 2 P: the breadth-first
// numbering. Four launches and those of the prefix sum (one up to 16384 particles, three up to
// 2^24); a launch and two grid-wide barriers for each of ~20 levels took 266 us at 2^18
// particles and 141 us at 4096.
#include <cuda_runtime.h>
#include <stdint.h>

#include "morton.cuh"
#include "primitives.cuh"
#include "topology.cuh"
#include "trevr_internal.cuh"

namespace trevr {

namespace {

constexpr int kTile = 1024;      // particles per tile of the depth counts
constexpr int kTileThreads = 256;
constexpr int kDepths = 64;

__device__ __forceinline__ int axis_of(int bit) { return (62 - bit) % 3; }

// the plane of the cut at `key` (the first of the upper child): its bit is set there
__device__ __forceinline__ int plane_of(unsigned long long key, int bit) {
  const int shift = kGridBits - 1 - (62 - bit) / 3;
  return (int)((key_coord(key, axis_of(bit)) >> shift) << shift);
}

__device__ __forceinline__ int high_bit(unsigned long long a, unsigned long long b) {
  return 63 - __clzll((long long)(a ^ b));
}

__device__ __forceinline__ bool no_tree(const TopoArrays& A) {
  return *A.status & kStatusIterationLimit;  // the sort gave up: its keys are not in order
}

__global__ void cut_kernel(TopoArrays A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.n) return;
  const unsigned long long k = A.key[i], before = i > 0 ? A.key[i - 1] : k;
  if (k == before || no_tree(A)) {
    A.up[i] = kNoCut;
    return;
  }
  const int b = high_bit(before, k);
  const unsigned long long base = k >> (b + 1) << (b + 1), top = base | ((2ull << b) - 1ull);
  // the range [f, l) of the keys in [base, top]: steps of doubling length, then bisection
  unsigned w = 1;
  while (w < (unsigned)i && A.key[i - 1 - (int)w] >= base) w *= 2;
  int lo = w < (unsigned)i ? i - (int)w : 0, hi = i - 1;  // key[hi] >= base
  while (lo < hi) {
    const int m = lo + ((hi - lo) >> 1);
    if (A.key[m] >= base) hi = m;
    else lo = m + 1;
  }
  const int f = lo;
  w = 1;
  while (w < (unsigned)(A.n - i) && A.key[i + (int)w] <= top) w *= 2;
  lo = i + 1;
  hi = w < (unsigned)(A.n - i) ? i + (int)w : A.n;  // the first key above top is in [lo, hi]
  while (lo < hi) {
    const int m = lo + ((hi - lo) >> 1);
    if (A.key[m] > top) hi = m;
    else lo = m + 1;
  }
  const int l = lo;
  if (l - f <= A.bucket) {
    A.up[i] = kNoCut;
    return;
  }
  A.range[i] = make_int2(f, l);
  A.bit[i] = (unsigned char)b;
  const int bf = f > 0 ? high_bit(A.key[f - 1], A.key[f]) : 64;
  const int bl = l < A.n ? high_bit(A.key[l - 1], A.key[l]) : 64;
  // the upper child of the cut at f, or the lower child of the cut at l
  A.up[i] = bf == 64 && bl == 64 ? kRootCut : bf < bl ? 2 * f + 1 : 2 * l;
}

__global__ void __launch_bounds__(kTileThreads) depth_kernel(TopoArrays A, int tiles) {
  __shared__ unsigned count[kDepths];
  for (int d = threadIdx.x; d < kDepths; d += kTileThreads) count[d] = 0;
  __syncthreads();
  for (int r = 0; r < kTile / kTileThreads; ++r) {
    const int i = blockIdx.x * kTile + r * kTileThreads + threadIdx.x;
    if (i >= A.n) break;
    int u = A.up[i];
    if (u == kNoCut) continue;
    int d = 0;
    for (; u >= 0 && d < kDepths - 1; ++d) u = A.up[u >> 1];
    A.depth[i] = (unsigned char)d;
    atomicAdd(&count[d], 1u);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < kDepths; d += kTileThreads)
    A.counts[(size_t)d * tiles + blockIdx.x] = count[d];
  if (blockIdx.x == 0 && threadIdx.x == 0) A.counts[(size_t)kDepths * tiles] = 0;
}

__global__ void __launch_bounds__(kTileThreads) place_kernel(TopoArrays A, int tiles) {
  constexpr int kWarps = kTileThreads / 32, kItems = kTile / kTileThreads;
  __shared__ unsigned count[kWarps][kDepths];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int d = lane; d < kDepths; d += 32) count[warp][d] = 0;
  __syncwarp();
  if (blockIdx.x == 0 && threadIdx.x < kMaxLevels) {
    // the levels' cells: a thread each, from the cuts before and up to the depth above it
    const int d = (int)threadIdx.x - 1;
    int begin = kRoot, end = no_tree(A) ? kRoot : kRoot + 1;
    if (d >= 0) {
      begin = kRoot + 1 + 2 * (int)A.counts[(size_t)min(d, kDepths) * tiles];
      end = kRoot + 1 + 2 * (int)A.counts[(size_t)min(d + 1, kDepths) * tiles];
      if (begin == end) begin = end = 0;
    }
    A.levels[2 * threadIdx.x] = begin;
    A.levels[2 * threadIdx.x + 1] = end;
  }
  const int own = blockIdx.x * kTile + warp * 32 * kItems + lane;
  unsigned rank[kItems];
  int depth[kItems];
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int i = own + 32 * r;
    const bool kept = i < A.n && A.up[i] != kNoCut;
    depth[r] = kept ? A.depth[i] : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, depth[r]);
    const unsigned before = __popc(peers & ((1u << lane) - 1u));
    rank[r] = kept ? count[warp][depth[r]] + before : 0u;
    __syncwarp();
    if (kept && before == 0) count[warp][depth[r]] += __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x < kDepths) {
    unsigned s = A.counts[(size_t)threadIdx.x * tiles + blockIdx.x];
    for (int w = 0; w < kWarps; ++w) {
      const unsigned c = count[w][threadIdx.x];
      count[w][threadIdx.x] = s;
      s += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kItems; ++r)
    if (depth[r] >= 0) {
      const int p = (int)(count[warp][depth[r]] + rank[r]);
      A.place[own + 32 * r] = p;
      A.list[p] = own + 32 * r;
    }
}

// the cell that a cut's link `u` (2 * parent + side) names
__device__ __forceinline__ int cell_of(const TopoArrays& A, int u) {
  return u < 0 ? kRoot : 2 + 2 * A.place[u >> 1] + (u & 1);
}

__device__ __forceinline__ void write_cell(const TopoArrays& A, int X, int child, int parent,
                                           const int lo[3], const int hi[3], int axis, int first,
                                           int count, int depth, unsigned long long way) {
  A.nT[X] = make_int4(child, parent, 0, 0);
  A.nglo[X] = make_int4(lo[0], lo[1], lo[2], axis);
  A.nghi[X] = make_int4(hi[0], hi[1], hi[2], 0);
  A.nfirst[X] = first;
  A.ncount[X] = count;
  A.ndepth[X] = depth;
  A.nD[X] = way | 1ull << (63 - depth);
}

__global__ void cell_kernel(TopoArrays A, int tiles) {
  const int first_thread = blockIdx.x * blockDim.x + threadIdx.x;
  if (first_thread == 0) {  // the unused cell 0
    A.nT[0] = make_int4(-1, 0, 0, 0);
    A.nD[0] = 1ull << 63;
  }
  const int total = (int)A.counts[(size_t)kDepths * tiles];
  if (total == 0) {
    const int lo[3] = {0, 0, 0}, hi[3] = {kGridMax, kGridMax, kGridMax};
    if (first_thread == 0) write_cell(A, kRoot, -1, 0, lo, hi, -1, 0, A.n, 0, 0ull);
    for (int i = first_thread; i < A.n; i += gridDim.x * blockDim.x) A.leaf_of[i] = kRoot;
    return;
  }
  for (int p = first_thread; p < total; p += gridDim.x * blockDim.x) {
    const int i = A.list[p];
    int lo[3] = {0, 0, 0}, hi[3] = {kGridMax, kGridMax, kGridMax};
    unsigned long long way = 0;  // sides from the cell up, the deepest in bit 0
    unsigned seen = 0;
    int depth = 0;
    const int up = A.up[i];
    for (int u = up; u >= 0 && depth < kDepths - 1; ++depth) {
      const int q = u >> 1, b = A.bit[q], ax = axis_of(b);
      way |= (unsigned long long)(u & 1) << depth;
      const unsigned face = 1u << (2 * ax + (u & 1));
      if (!(seen & face)) {  // the nearest plane on this side
        seen |= face;
        const int g = plane_of(A.key[q], b);
#pragma unroll
        for (int d = 0; d < 3; ++d)
          if (d == ax) {
            if (u & 1) lo[d] = g;
            else hi[d] = g;
          }
      }
      u = A.up[q];
    }
    if (depth > 0) way <<= 64 - depth;
    const int b = A.bit[i], ax = axis_of(b), g = plane_of(A.key[i], b);
    const int2 range = A.range[i];
    const int X = cell_of(A, up), child = 2 + 2 * p;
    write_cell(A, X, child, up < 0 ? 0 : cell_of(A, A.up[up >> 1]), lo, hi, ax, range.x,
               range.y - range.x, depth, way);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int f = side ? i : range.x, n = (side ? range.y : i) - f;
      if (n > A.bucket && A.key[f] != A.key[f + n - 1]) continue;  // a cut of its own
      int clo[3] = {lo[0], lo[1], lo[2]}, chi[3] = {hi[0], hi[1], hi[2]};
#pragma unroll
      for (int d = 0; d < 3; ++d)
        if (d == ax) {
          if (side) clo[d] = g;
          else chi[d] = g;
        }
      write_cell(A, child + side, -1, X, clo, chi, -1, f, n, depth + 1,
                 way | (unsigned long long)side << (63 - depth));
      for (int j = f; j < f + n; ++j) A.leaf_of[j] = child + side;
    }
  }
}

int tiles_of(int n) { return (n + kTile - 1) / kTile; }

}  // namespace

size_t topo_count_words(int n) { return (size_t)kDepths * tiles_of(n) + 1; }

void launch_cuts(const TopoArrays& A, unsigned* scan_scratch, cudaStream_t s) {
  const int n = A.n, tiles = tiles_of(n);
  cut_kernel<<<(n + 255) / 256, 256, 0, s>>>(A);
  depth_kernel<<<tiles, kTileThreads, 0, s>>>(A, tiles);
  exclusive_scan_u32(A.counts, (int)topo_count_words(n), scan_scratch, s);
  place_kernel<<<tiles, kTileThreads, 0, s>>>(A, tiles);
  note_launch(3);
}

void launch_cells(const TopoArrays& A, cudaStream_t s) {
  const int blocks = A.n / 512 + 1;  // about one cut in six particles is kept
  cell_kernel<<<blocks < 4096 ? blocks : 4096, 128, 0, s>>>(A, tiles_of(A.n));
  note_launch();
}

}  // namespace trevr
