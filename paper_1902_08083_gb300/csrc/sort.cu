// Device-wide prefix sum, and the stable radix sort of (64-bit key, 32-bit value) pairs that
// orders particles along the Morton curve, sources by leaf and a call's sinks.
//
// The sort takes 8-bit digits from the least significant. Up to kSmallSort pairs are sorted by
// one block in one launch, the pairs in registers and shared memory throughout. Larger inputs
// take one launch that counts every digit of every pass, and one launch per pass: a tile of
// 2048 or 4096 pairs is ranked in shared memory, its digit counts are added up over the tiles
// before it by decoupled look-back (Merrill & Garland's single-pass scan, as Adinets &
// Merrill's one-sweep sort uses it), and its pairs are written in runs of equal digits. So a
// pass reads and writes each pair once (24 bytes) and nothing is counted twice.
#include <cuda_runtime.h>
#include <stdint.h>

#include "primitives.cuh"
#include "trevr_internal.cuh"

namespace trevr {

// ------------------------------------------------------------------------------------
// Device-wide exclusive scan (unsigned, in place)
// ------------------------------------------------------------------------------------
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__global__ void scan_tile_kernel(unsigned* data, int n, unsigned* tile_sums) {
  __shared__ unsigned smem[32];
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  unsigned v[kScanItems];
  unsigned s = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    v[j] = (base + j < n) ? data[base + j] : 0u;
    s += v[j];
  }
  unsigned total;
  unsigned off = block_exclusive_scan(s, smem, &total);
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    if (base + j < n) data[base + j] = off;
    off += v[j];
  }
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
}

__global__ void scan_add_kernel(unsigned* data, int n, const unsigned* tile_offsets) {
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  const unsigned o = tile_offsets[blockIdx.x];
#pragma unroll
  for (int j = 0; j < kScanItems; ++j)
    if (base + j < n) data[base + j] += o;
}

int scan_tiles(int n) { return (n + kScanTile - 1) / kScanTile; }

}  // namespace

// scratch must hold scan_scratch_words(n) unsigned
size_t scan_scratch_words(int n) {
  size_t w = 0;
  while (n > 1) {
    n = scan_tiles(n);
    w += (size_t)n;
  }
  return w + 1;
}

void exclusive_scan_u32(unsigned* data, int n, unsigned* scratch, cudaStream_t s) {
  if (n <= 0) return;
  int tiles = scan_tiles(n);
  scan_tile_kernel<<<tiles, kScanThreads, 0, s>>>(data, n, scratch);
  note_launch();
  if (tiles > 1) {
    exclusive_scan_u32(scratch, tiles, scratch + tiles, s);
    scan_add_kernel<<<tiles, kScanThreads, 0, s>>>(data, n, scratch);
    note_launch();
  }
}

// ------------------------------------------------------------------------------------
// Radix sort
// ------------------------------------------------------------------------------------
namespace {

// a tile's word of a digit: nothing yet (0), the tile's own count, or the count of this
// tile and all before it (at most 2^30 pairs)
constexpr unsigned kOwn = 0x40000000u, kAll = 0x80000000u;
constexpr int kPollLimit = 1 << 20;  // look-back polls of one digit before the pass gives up
constexpr int kWindow = 8;           // tiles that a look-back reads at a time
constexpr int kSmallThreads = 256, kSmallItems = kSmallSort / kSmallThreads;

__device__ __forceinline__ unsigned digit_of(unsigned long long k, int shift) {
  return (unsigned)(k >> shift) & 255u;
}

// Rank of each of a thread's ITEMS keys among the equal digits before it in its warp's run
// (item r of lane l is at r * 32 + l of the run); count[256] becomes the warp's totals. The
// lanes with a key's digit come from eight ballots, and one of them adds their number to the
// digit's count: no round waits for the one before (with __match_any_sync and a load and a
// store of the count in each round, a pass over 2^20 pairs took 22.6 us, most of it here).
template <int ITEMS>
__device__ __forceinline__ void rank_warp(const unsigned long long (&key)[ITEMS], int shift,
                                          unsigned* count, unsigned (&rank)[ITEMS]) {
  const unsigned lane = lane_id(), lt = (1u << lane) - 1u;
  unsigned peers[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const unsigned d = digit_of(key[r], shift);
    unsigned m = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const bool one = (d >> b) & 1u;
      const unsigned ones = __ballot_sync(0xffffffffu, one);
      m &= one ? ones : ~ones;
    }
    peers[r] = m;
  }
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    rank[r] = 0;
    if ((peers[r] & lt) == 0) rank[r] = atomicAdd(&count[digit_of(key[r], shift)], __popc(peers[r]));
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < ITEMS; ++r)
    rank[r] = __shfl_sync(0xffffffffu, rank[r], __ffs(peers[r]) - 1) + __popc(peers[r] & lt);
}

__global__ void __launch_bounds__(kSmallThreads) small_sort_kernel(unsigned long long* k,
                                                                   unsigned* v, int n,
                                                                   int passes) {
  constexpr int kWarps = kSmallThreads / 32;
  static_assert(kSmallThreads == 256, "one thread per digit");
  __shared__ unsigned long long stage[kSmallSort];
  __shared__ unsigned count[kWarps][256];
  __shared__ unsigned start[256];
  __shared__ unsigned smem[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int own = warp * 32 * kSmallItems + lane;
  unsigned long long key[kSmallItems];
  unsigned val[kSmallItems], rank[kSmallItems];
#pragma unroll
  for (int r = 0; r < kSmallItems; ++r) {
    const int i = own + 32 * r;
    key[r] = i < n ? k[i] : ~0ull;  // stays behind every pair: the sort is stable
    val[r] = i < n ? v[i] : 0u;
  }
  for (int p = 0; p < passes; ++p) {
    const int shift = 8 * p;
    for (int d = lane; d < 256; d += 32) count[warp][d] = 0;
    __syncwarp();
    rank_warp(key, shift, count[warp], rank);
    __syncthreads();
    unsigned total = 0, all;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const unsigned c = count[w][threadIdx.x];
      count[w][threadIdx.x] = total;
      total += c;
    }
    start[threadIdx.x] = block_exclusive_scan(total, smem, &all);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r) {
      const unsigned d = digit_of(key[r], shift);
      rank[r] += start[d] + count[warp][d];
      stage[rank[r]] = key[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r) key[r] = stage[own + 32 * r];
    __syncthreads();
    unsigned* vals = reinterpret_cast<unsigned*>(stage);
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r) vals[rank[r]] = val[r];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r) val[r] = vals[own + 32 * r];
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < kSmallItems; ++r) {
    const int i = own + 32 * r;
    if (i < n) {
      k[i] = key[r];
      v[i] = val[r];
    }
  }
}

constexpr int kCountItems = 4, kCountTile = 256 * kCountItems;

// counts[pass][digit] over all keys
__global__ void __launch_bounds__(256) digit_count_kernel(const unsigned long long* __restrict__ k,
                                                          int n, int passes, unsigned* counts) {
  __shared__ unsigned c[8][256];
  for (int i = threadIdx.x; i < 8 * 256; i += 256) (&c[0][0])[i] = 0;
  __syncthreads();
  for (int i0 = blockIdx.x * kCountTile; i0 < n; i0 += gridDim.x * kCountTile) {
    unsigned long long key[kCountItems];
#pragma unroll
    for (int r = 0; r < kCountItems; ++r) {
      const int i = i0 + 256 * r + (int)threadIdx.x;
      key[r] = i < n ? k[i] : 0ull;
    }
#pragma unroll
    for (int r = 0; r < kCountItems; ++r) {
      const int w0 = i0 + 256 * r + (int)(threadIdx.x & ~31u), in = min(32, n - w0);
      if (in <= 0) break;
      const bool own = (int)lane_id() < in;
      for (int p = 0; p < passes; ++p) {
        const unsigned d = digit_of(key[r], 8 * p);
        // clustered keys share their high digits: one add for a warp that agrees
        const unsigned d0 = __shfl_sync(0xffffffffu, d, 0);
        if (__all_sync(0xffffffffu, !own || d == d0)) {
          if (lane_id() == 0) atomicAdd(&c[p][d0], (unsigned)in);
        } else if (own) {
          atomicAdd(&c[p][d], 1u);
        }
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * 256; i += 256) {
    const unsigned v = (&c[0][0])[i];
    if (v) atomicAdd(&counts[i], v);
  }
}

// One pass: a tile of 256 ITEMS pairs per block, in the order of the blocks' tickets, so that
// the tiles before it are done or running. tiles_now holds this pass's words (zero at the
// start), tiles_next is cleared for the next pass.
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads, ITEMS > 8 ? 2 : 3) sort_pass_kernel(
    const unsigned long long* __restrict__ kin, const unsigned* __restrict__ vin,
    unsigned long long* __restrict__ kout, unsigned* __restrict__ vout, int n, int shift,
    const unsigned* __restrict__ counts, unsigned* ticket, unsigned* tiles_now,
    unsigned* __restrict__ tiles_next, int* status) {
  constexpr int kWarps = kSortThreads / 32, kTile = kSortThreads * ITEMS;
  static_assert(kSortThreads == 256, "one thread per digit");
  __shared__ unsigned long long stage[kTile];
  __shared__ unsigned count[kWarps][256];
  __shared__ unsigned start[256];   // first place of a digit in the tile
  __shared__ unsigned target[256];  // its first place in the output, less start
  __shared__ unsigned smem[32];
  __shared__ int s_tile, s_failed;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, d = threadIdx.x;
  if (threadIdx.x == 0) {
    s_tile = (int)atomicAdd(ticket, 1u);
    s_failed = 0;
  }
  for (int i = lane; i < 256; i += 32) count[warp][i] = 0;
  __syncthreads();
  const int tile = s_tile;
  const int base = tile * kTile, here = min(kTile, n - base);
  tiles_next[(size_t)tile * 256 + d] = 0;
  const int own = warp * 32 * ITEMS + lane;
  unsigned long long key[ITEMS];
  unsigned rank[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int i = own + 32 * r;
    key[r] = i < here ? kin[base + i] : ~0ull;  // behind every pair of the tile
  }
  rank_warp(key, shift, count[warp], rank);
  __syncthreads();
  unsigned total = 0, all;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const unsigned c = count[w][d];
    count[w][d] = total;
    total += c;
  }
  const unsigned off = block_exclusive_scan(total, smem, &all);
  if (d == 255) total -= (unsigned)(kTile - here);  // the filling is not counted
  volatile unsigned* words = tiles_now;
  unsigned before = 0;
  if (tile == 0) {
    words[d] = kAll | total;
  } else {
    words[(size_t)tile * 256 + d] = kOwn | total;
    int polls = 0;
    for (int t = tile - 1; t >= 0;) {
      unsigned w[kWindow];  // the words of the tiles t, t - 1, ... on their way together
#pragma unroll
      for (int q = 0; q < kWindow; ++q) w[q] = words[(size_t)max(t - q, 0) * 256 + d];
      bool all_found = false;
      int q = 0;
#pragma unroll
      for (int u = 0; u < kWindow; ++u) {
        if (q != u || all_found) continue;  // the word before was still empty, or the last
        if (w[u] & kAll) {
          before += w[u] & ~kAll;
          all_found = true;
        } else if (w[u] & kOwn) {
          before += w[u] & ~kOwn;
          ++q;
        }
      }
      if (all_found) break;
      t -= q;
      if (q == 0 && ++polls > kPollLimit) {
        s_failed = 1;
        break;
      }
    }
    words[(size_t)tile * 256 + d] = kAll | ((before + total) & ~kAll);
  }
  const unsigned first = block_exclusive_scan(counts[d], smem, &all);
  start[d] = off;
  target[d] = first + before - off;
  __syncthreads();
  if (s_failed) {
    if (threadIdx.x == 0) atomicOr(status, kStatusIterationLimit);
    return;
  }
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const unsigned g = digit_of(key[r], shift);
    rank[r] += start[g] + count[warp][g];
    stage[rank[r]] = key[r];
  }
  __syncthreads();
  unsigned to[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int j = threadIdx.x + kSortThreads * r;
    const unsigned long long k = stage[j];
    to[r] = j < here ? target[digit_of(k, shift)] + (unsigned)j : ~0u;
    if (to[r] < (unsigned)n) kout[to[r]] = k;
  }
  unsigned val[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int i = own + 32 * r;
    val[r] = i < here ? vin[base + i] : 0u;
  }
  __syncthreads();
  unsigned* vals = reinterpret_cast<unsigned*>(stage);
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) vals[rank[r]] = val[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r)
    if (to[r] < (unsigned)n) vout[to[r]] = vals[threadIdx.x + kSortThreads * r];
}

}  // namespace

// Pairs per tile: half the tile halves a block's ranking, and twice the tiles lengthen the
// look-back. 2048 / 4096 pairs take 97 / 112 us for 5000 keys of 63 bits, 131 / 147 for 2^18,
// 238 / 204 for 2^20 (the whole call of the allocation-free sort).
static int sort_tile(int n) { return n <= (1 << 18) ? kSortTile / 2 : kSortTile; }

size_t sort_work_words(int n) {
  if (n <= kSmallSort) return 1;
  return (size_t)kSortHead + 2 * 256 * (size_t)((n + sort_tile(n) - 1) / sort_tile(n));
}

bool radix_sort(unsigned long long* k, unsigned* v, int n, int bits, const SortScratch& S,
                int* status, cudaStream_t s) {
  if (n <= 1) return true;
  const int passes = (bits + 7) / 8;
  if (n <= kSmallSort) {
    small_sort_kernel<<<1, kSmallThreads, 0, s>>>(k, v, n, passes);
    note_launch();
    return true;
  }
  if (S.size < (size_t)n || S.words < sort_work_words(n)) return false;
  const int tile = sort_tile(n), tiles = (n + tile - 1) / tile;
  unsigned *counts = S.work, *tickets = S.work + 8 * 256;
  unsigned* words[2] = {S.work + kSortHead, S.work + kSortHead + 256 * (size_t)tiles};
  cudaMemsetAsync(S.work, 0, ((size_t)kSortHead + 256 * (size_t)tiles) * sizeof(unsigned), s);
  const int counters = (n + kCountTile - 1) / kCountTile, fill = 4 * sm_count();
  digit_count_kernel<<<counters < fill ? counters : fill, 256, 0, s>>>(k, n, passes, counts);
  note_launch();
  unsigned long long *ka = k, *kb = S.k2;
  unsigned *va = v, *vb = S.v2;
  for (int p = 0; p < passes; ++p) {
    const auto pass = tile == kSortTile ? sort_pass_kernel<kSortItems>
                                        : sort_pass_kernel<kSortItems / 2>;
    pass<<<tiles, kSortThreads, 0, s>>>(ka, va, kb, vb, n, 8 * p, counts + 256 * p, tickets + p,
                                        words[p & 1], words[(p & 1) ^ 1], status);
    note_launch();
    unsigned long long* tk = ka;
    ka = kb;
    kb = tk;
    unsigned* tv = va;
    va = vb;
    vb = tv;
  }
  if (ka != k) {
    cudaMemcpyAsync(k, ka, (size_t)n * sizeof(unsigned long long), cudaMemcpyDeviceToDevice, s);
    cudaMemcpyAsync(v, va, (size_t)n * sizeof(unsigned), cudaMemcpyDeviceToDevice, s);
  }
  return true;
}

}  // namespace trevr
