// Sink walk, reverse ray and flux sum (Grond et al. 2019, Sec. 2.2.1-2.2.3).
//
// Per sink (a gas particle at p in leaf S):
//   * source walk: a cell with L > 0 is merged into one pseudo-source at its
//     centre of luminosity when theta_open > l/r (Eq. openangle), tested as
//     l^2 < theta^2 r^2 in fp32; otherwise it is opened, and an opened leaf
//     gives its sources one by one;
//   * reverse ray to each pseudo-source: the segments are S, the pseudo-source's
//     cell C and the siblings of the cells on the two paths up to the children
//     of their lowest common ancestor A; each segment uses the cell's mean
//     absorption unless (alpha_max - alpha_min) * l > tau_ref (Eq. refcrit), in
//     which case its children are used instead;
//   * flux: sum of L exp(-tau) / (4 pi s^2) (Eq. simpint).
// The decisions (opening angle, refinement, "does the ray touch the cell") are
// evaluated with explicitly rounded fp32 operations in a fixed order. Positions,
// centres of luminosity and cell planes are stored relative to the domain's lower
// corner (planes g * h), so their fp32 rounding depends on the domain's size and not
// on its offset from the origin.
//
// GPU form (sinks in Morton order, so the lanes of a warp are neighbours in space). This
// file has variant 1 (walk_kernel), which clips every cell of a ray by itself: one lane per
// sink, a flat loop in which one iteration is a walk step or a cell clip, cells picked with
// selects from one per-lane list; a lane that finishes takes the next sink of its warp's
// chunk. The segment cells of a ray are known without following parent links: the sibling of
// a cell is its index XOR 1 (children are allocated in pairs) and the common ancestor's depth
// is the length of the common prefix of the sink's ancestor list and the walk path, kept as a
// 64-bit mask. Variants 2 and 3 are in cutwalk.cu.
#include <cuda_runtime.h>
#include <stdint.h>

#include "trevr_internal.cuh"
#include "walk_common.cuh"

namespace trevr {

namespace {

constexpr int kAnc = 0;     // offsets of the three parts of the per-lane list
constexpr int kPath = kDepth;
constexpr int kRef = 2 * kDepth;

// one slab of the clip: (lo - p) * (1/d), (hi - p) * (1/d), rounded after each step;
// along an axis the ray does not move on, the box is half-open [lo, hi), so a ray
// lying in the face between two cells belongs to the upper one only
__device__ __forceinline__ void slab(float lo, float hi, float p, float d, float inv, float& t0,
                                     float& t1, bool& miss) {
  if (d != 0.0f) {
    const float ta = __fmul_rn(__fsub_rn(lo, p), inv);
    const float tb = __fmul_rn(__fsub_rn(hi, p), inv);
    t0 = fmaxf(t0, fminf(ta, tb));
    t1 = fminf(t1, fmaxf(ta, tb));
  } else {
    miss = miss || p < lo || p >= hi;
  }
}

// gradient-carrying slab: remembers which axis sets t0 / t1
__device__ __forceinline__ void slab_g(int k, float lo, float hi, float p, float d, float inv,
                                       float& t0, float& t1, int& k0, int& k1, bool& miss) {
  if (d != 0.0f) {
    const float ta = __fmul_rn(__fsub_rn(lo, p), inv);
    const float tb = __fmul_rn(__fsub_rn(hi, p), inv);
    const float tn = fminf(ta, tb), tx = fmaxf(ta, tb);
    if (tn > t0) {
      t0 = tn;
      k0 = k;
    }
    if (tx < t1) {
      t1 = tx;
      k1 = k;
    }
  } else {
    miss = miss || p < lo || p >= hi;
  }
}

}  // namespace

// Per-lane lists, kept apart from the scalar state so that the state stays in
// registers: the ancestors of S | the depth-first path | cells to clip, and the
// walk stack (cell, depth).
struct Lists {
  int lst[3 * kDepth];
  int wstack[kDepth];
  int wdepth[kDepth];
};

// State of one lane: the sink it works on, its walk and its current ray.
// ADJ = false computes the flux. ADJ = true is the adjoint with the same
// decisions: every ray is traced twice, first for tau and d(tau)/dq, then, with
// the contribution f known, to scatter -g f l_X into each segment cell.
template <bool ADJ>
struct Lane {
  // sink
  int i;     // sorted position
  float gk;  // dLoss/dF of this sink (adjoint)
  float px, py, pz;
  int S, dS;
  unsigned long long on_path;  // bit d: path[d] is an ancestor of S
  int sp;                      // walk stack size
  CSum F;
  SinkCounters cnt;  // this sink's counters
  // ray
  bool in_ray;
  float dx, dy, dz, ix, iy, iz, len, s2, rayL;
  CSum tau;
  int C, dC, nSs, nb, b, rsp, boxes;
  // single sources of an opened leaf
  int j, j_end, leafC, dleaf;
  // adjoint
  int pass, src_j;
  float gq0, gq1, gq2, fcur;
  __device__ __forceinline__ void begin(const TreeView& T, int i_, float g, Lists& L_) {
    int* lst = L_.lst;
    int* wstack = L_.wstack;
    int* wdepth = L_.wdepth;
    i = i_;
    gk = g;
    const float4 p = T.pos[i];
    px = p.x;
    py = p.y;
    pz = p.z;
    S = T.leaf_of[i];
    dS = __ldg(&T.ndepth[S]);
    int u = S;
    for (int d = dS; d >= 0; --d) {
      lst[kAnc + d] = u;
      u = __ldg(&T.nT[u].y);
    }
    on_path = 0;
    wstack[0] = kRoot;
    wdepth[0] = 0;
    sp = 1;
    F = CSum();
    cnt = SinkCounters();
    in_ray = false;
    j = j_end = 0;
  }

  // One iteration. Returns false when the sink is finished.
  __device__ __forceinline__ bool step(const TreeView& T, const WalkParams& P, int stack_limit,
                                       int box_limit, int* status, const AdjointArgs& J,
                                       Lists& L_) {
    int* lst = L_.lst;
    int* wstack = L_.wstack;
    int* wdepth = L_.wdepth;
    if (in_ray) {
      const bool from_stack = rsp > 0;
      if (!from_stack && b >= nb) {
        finish_ray(J);
        return true;
      }
      // the next cell, by selects: refinement stack, else S, sink-side siblings,
      // C, pseudo-source-side siblings
      int off = kRef + rsp - 1;
      if (!from_stack) off = (b <= nSs) ? (kAnc + dS - b + 1) : (kPath + dC - (b - nSs - 2));
      const int v = lst[off];
      const int box = from_stack ? v : ((b == 0) ? S : ((b == nSs + 1) ? C : (v ^ 1)));
      rsp -= from_stack ? 1 : 0;
      b += from_stack ? 0 : 1;
      if (++boxes > box_limit) {
        atomicOr(status, kStatusIterationLimit);
        return false;
      }
      const float4 a = __ldg(&T.nA[box]);
      const float4 bb = __ldg(&T.nB[box]);
      const bool want_grad = ADJ && pass == 1 && src_j < 0;
      float t0 = 0.0f, t1 = 1.0f;
      bool miss = false;
      int k0 = -1, k1 = -1;
      if (want_grad) {
        slab_g(0, a.x, bb.x, px, dx, ix, t0, t1, k0, k1, miss);
        slab_g(1, a.y, bb.y, py, dy, iy, t0, t1, k0, k1, miss);
        slab_g(2, a.z, bb.z, pz, dz, iz, t0, t1, k0, k1, miss);
      } else {
        slab(a.x, bb.x, px, dx, ix, t0, t1, miss);
        slab(a.y, bb.y, py, dy, iy, t0, t1, miss);
        slab(a.z, bb.z, pz, dz, iz, t0, t1, miss);
      }
      const float l = (!miss && t1 > t0) ? __fmul_rn(__fsub_rn(t1, t0), len) : 0.0f;
      ++cnt.clip;
      if (!(l > 0.0f)) return true;
      if (P.tau_ref <= 0.0f || __fmul_rn(bb.w, l) > P.tau_ref) {
        const int child = __ldg(&T.nT[box].x);
        if (child >= 0) {
          if (rsp + 2 > stack_limit) {
            atomicOr(status, kStatusStackOverflow);
            return false;
          }
          ++cnt.ref;
          lst[kRef + rsp] = child + 1;
          lst[kRef + rsp + 1] = child;
          rsp += 2;
          return true;
        }
      }
      if (ADJ && pass == 2) {
        atomicAdd(&J.G[box], (double)(-gk * fcur * l));
        return true;
      }
      tau.add(a.w * l);
      if (want_grad) {
        // d l / d q: a slab parameter t = (b - p_k)/d_k moves as -t/d_k along q_k;
        // one clamped to 0 or 1 does not move
        const float w = (t1 - t0) / len;
        const float g0 = (k1 == 0 ? -t1 * ix : 0.0f) + (k0 == 0 ? t0 * ix : 0.0f);
        const float g1 = (k1 == 1 ? -t1 * iy : 0.0f) + (k0 == 1 ? t0 * iy : 0.0f);
        const float g2 = (k1 == 2 ? -t1 * iz : 0.0f) + (k0 == 2 ? t0 * iz : 0.0f);
        gq0 = fmaf(a.w, g0 * len + w * dx, gq0);
        gq1 = fmaf(a.w, g1 * len + w * dy, gq1);
        gq2 = fmaf(a.w, g2 * len + w * dz, gq2);
      }
      ++cnt.segs;
      return true;
    }

    // ---- walk step: find the next pseudo-source
    float qx, qy, qz, L;
    if (j < j_end) {
      const float4 y = __ldg(&T.src[j]);
      ++j;
      if (!(y.w > 0.0f)) return true;
      C = leafC;
      dC = dleaf;
      src_j = j - 1;
      qx = y.x;
      qy = y.y;
      qz = y.z;
      L = y.w;
    } else {
      if (sp == 0) return false;  // the sink is done
      --sp;
      const int X = wstack[sp];
      const int dX = wdepth[sp];
      lst[kPath + dX] = X;
      const unsigned long long bit = 1ull << dX;
      on_path = (dX <= dS && lst[kAnc + dX] == X) ? (on_path | bit) : (on_path & ~bit);
      const float4 s = __ldg(&T.nS[X]);
      if (!(s.w > 0.0f)) return true;
      ++cnt.visit;
      const float4 a = __ldg(&T.nA[X]);
      const float4 bb = __ldg(&T.nB[X]);
      const float ex = fmaxf(fmaxf(__fsub_rn(a.x, px), __fsub_rn(px, bb.x)), 0.0f);
      const float ey = fmaxf(fmaxf(__fsub_rn(a.y, py), __fsub_rn(py, bb.y)), 0.0f);
      const float ez = fmaxf(fmaxf(__fsub_rn(a.z, pz), __fsub_rn(pz, bb.z)), 0.0f);
      const float r2 =
          __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
      if (!(__ldg(&T.nl2[X]) < __fmul_rn(P.theta2, r2))) {
        const int4 t = __ldg(&T.nT[X]);
        if (t.x < 0) {
          j = t.z;
          j_end = t.z + t.w;
          leafC = X;
          dleaf = dX;
        } else {
          if (sp + 2 > stack_limit) {
            atomicOr(status, kStatusStackOverflow);
            return false;
          }
          wstack[sp] = t.x + 1;
          wdepth[sp] = dX + 1;
          wstack[sp + 1] = t.x;
          wdepth[sp + 1] = dX + 1;
          sp += 2;
        }
        return true;
      }
      C = X;
      dC = dX;
      src_j = -1;
      qx = s.x;
      qy = s.y;
      qz = s.z;
      L = s.w;
    }
    // ---- start the reverse ray from the sink to (q, L) in cell C
    dx = __fsub_rn(qx, px);
    dy = __fsub_rn(qy, py);
    dz = __fsub_rn(qz, pz);
    s2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
    if (s2 < P.smin2) return true;  // a source on top of the sink adds nothing
    len = __fsqrt_rn(s2);
    ix = dx != 0.0f ? __frcp_rn(dx) : 0.0f;
    iy = dy != 0.0f ? __frcp_rn(dy) : 0.0f;
    iz = dz != 0.0f ? __frcp_rn(dz) : 0.0f;
    rayL = L;
    tau = CSum();
    pass = 1;
    gq0 = gq1 = gq2 = 0.0f;
    b = 0;
    rsp = 0;
    boxes = 0;
    if (C == S) {
      nSs = 0;
      nb = 1;
    } else {
      // depth of the lowest common ancestor: the common prefix of path and anc
      const int mn = dC < dS ? dC : dS;
      const unsigned long long m = on_path & ((2ull << mn) - 1ull);  // mn <= 62
      const int dstar = __ffsll((long long)~m) - 2;
      nSs = dS - dstar - 1;  // siblings on the sink side
      nb = dS + dC - 2 * dstar;
    }
    in_ray = true;
    return true;
  }

  __device__ __forceinline__ void finish_ray(const AdjointArgs& J) {
    const float t = tau.get();
    const float f = rayL * expf(-t) / (kFourPi * s2);
    if (!ADJ) {
      F.add(f);
      ++cnt.rays;
      in_ray = false;
    } else if (pass == 1) {
      // second pass over the same cells, now that f is known
      fcur = f;
      pass = 2;
      b = 0;
      rsp = 0;
      boxes = 0;
    } else {
      const float gf = gk * fcur;
      if (src_j >= 0) {
        atomicAdd(&J.e[src_j], (double)(gf / rayL));
      } else {
        const float c = gf / rayL, inv_s2 = 2.0f / s2;
        atomicAdd(&J.a[C], (double)c);
        atomicAdd(&J.b[3 * C + 0], (double)(c * (-dx * inv_s2 - gq0)));
        atomicAdd(&J.b[3 * C + 1], (double)(c * (-dy * inv_s2 - gq1)));
        atomicAdd(&J.b[3 * C + 2], (double)(c * (-dz * inv_s2 - gq2)));
      }
      ++cnt.rays;
      in_ray = false;
    }
  }
};

// Runs the sinks [first, end) of a chunk with one warp: the lanes start on the
// first 32 and take the next unclaimed sink of the chunk when theirs is done.
// `map` turns a chunk position into (sorted position, output slot, dLoss/dF);
// positions it rejects are skipped. Every lane of the warp must call it.
template <bool ADJ, class Map>
__device__ __forceinline__ void run_chunk(const TreeView& T, const WalkParams& P, int first,
                                          int end, const Map& map, const SinkOut& out,
                                          int* status, const AdjointArgs& J, SinkCounters& tot) {
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt = (1u << lane) - 1u;
  const int stack_limit = P.stack_depth < kDepth ? P.stack_depth : kDepth;
  const int box_limit = 2 * T.n_nodes_cap + 4;
  Lane<ADJ> st;
  Lists lists;
  int next = first;     // next unclaimed chunk position (same value in every lane)
  bool active = false;  // this lane holds a sink
  int slot = -1;        // output slot of the lane's sink
  while (true) {
    // idle lanes claim the next positions of the chunk, in lane order
    const unsigned idle = __ballot_sync(0xffffffffu, !active);
    if (idle) {
      if (next >= end) {
        if (idle == 0xffffffffu) break;
      } else {
        const int pos = next + (int)__popc(idle & lt);
        if (!active && pos < end) {
          int i;
          float g;
          if (map(pos, i, slot, g)) {
            st.begin(T, i, g, lists);
            active = true;
          }
        }
        next += (int)__popc(idle);
        continue;  // a lane whose position was rejected claims again next round
      }
    }
    if (active && !st.step(T, P, stack_limit, box_limit, status, J, lists)) {
      active = false;
      if (!ADJ) {
        if (out.flux) out.flux[slot] = st.F.get();
        if (out.counters)
          reinterpret_cast<int4*>(out.counters)[slot] =
              make_int4(st.cnt.rays, st.cnt.segs, st.cnt.visit, st.cnt.ref);
      }
      tot.rays += st.cnt.rays;
      tot.segs += st.cnt.segs;
      tot.visit += st.cnt.visit;
      tot.ref += st.cnt.ref;
      tot.clip += st.cnt.clip;
    }
  }
}

template <bool ADJ>
__global__ void __launch_bounds__(128) walk_kernel(TreeView T, const long long* sink_idx,
                                                   int n_sink, int chunk, WalkParams P,
                                                   SinkOut out, unsigned long long* stats,
                                                   int* status, AdjointArgs J) {
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long first = warp * chunk;
  SinkCounters tot;
  if (first < n_sink) {
    const int end = (int)min((long long)n_sink, first + chunk);
    if (!ADJ && sink_idx) {  // sinks with an index out of range get zeros
      for (int k = (int)first + (int)(threadIdx.x & 31); k < end; k += 32) {
        const long long si = sink_idx[k];
        if (si < 0 || si >= T.n_gas) {
          if (out.flux) out.flux[k] = 0.0f;
          if (out.counters) reinterpret_cast<int4*>(out.counters)[k] = make_int4(0, 0, 0, 0);
        }
      }
    }
    PlainMap<ADJ> map{&T, sink_idx, J.grad_flux, status, P.order, n_sink};
    run_chunk<ADJ>(T, P, (int)first, end, map, out, status, J, tot);
  }
  if (stats) add_stats(tot, stats);
}

// Batched form: sorted positions of one tree, output in that tree's caller order.
struct TreeMap {
  const TreeView* T;
  __device__ __forceinline__ bool operator()(int k, int& i, int& slot, float& g) const {
    i = k;
    slot = T->perm[k];
    g = 0.0f;
    return true;
  }
};

// Many independent trees in one persistent launch. Work items are runs of
// `item` consecutive sinks (Morton order) of one tree; each warp takes the next
// item from a device counter, so warps that finish early keep pulling work from
// the boxes that are left. Per-sink arithmetic is the same as walk_kernel.
template <int BS>
__global__ void __launch_bounds__(BS) walk_batched_kernel(const TreeView* __restrict__ views,
                                                         float* const* __restrict__ flux_out,
                                                         const int2* __restrict__ items,
                                                         int n_items, int item,
                                                         unsigned* counter, WalkParams P,
                                                         unsigned long long* stats, int* status) {
  const unsigned lane = threadIdx.x & 31u;
  SinkCounters tot;
  while (true) {
    unsigned it = 0;
    if (lane == 0) it = atomicAdd(counter, 1u);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= (unsigned)n_items) break;
    const int2 w = items[it];
    const TreeView T = views[w.x];
    WalkParams Pt = P;  // the coincident-source cut (1e-12 side)^2 of this tree, in fp32
    const float smin = __fmul_rn(1e-12f, T.side);
    Pt.smin2 = __fmul_rn(smin, smin);
    SinkOut out{flux_out[w.x], nullptr, nullptr, nullptr, 0};
    TreeMap map{&T};
    run_chunk<false>(T, Pt, w.y, min(w.y + item, T.n_gas), map, out, status, AdjointArgs{}, tot);
  }
  if (stats) add_stats(tot, stats);
}

cudaError_t launch_walk_batched(const TreeView* views, float* const* flux_out, const int2* items,
                                int n_items, int item, unsigned* counter, const WalkParams& wp,
                                unsigned long long* stats, int* status, int block_size,
                                int n_sm, cudaStream_t s) {
  if (n_items <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  int per_sm = 1;
  if (wp.variant >= 2)
    return launch_cut_batched(views, flux_out, items, n_items, item, counter, wp, stats, status,
                              block_size, n_sm, s);
  if (block_size <= 64) {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, walk_batched_kernel<64>, 64, 0);
    walk_batched_kernel<64><<<n_sm * per_sm, 64, 0, s>>>(views, flux_out, items, n_items, item,
                                                         counter, wp, stats, status);
  } else if (block_size <= 128) {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, walk_batched_kernel<128>, 128, 0);
    walk_batched_kernel<128><<<n_sm * per_sm, 128, 0, s>>>(views, flux_out, items, n_items, item,
                                                           counter, wp, stats, status);
  } else {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, walk_batched_kernel<256>, 256, 0);
    walk_batched_kernel<256><<<n_sm * per_sm, 256, 0, s>>>(views, flux_out, items, n_items, item,
                                                           counter, wp, stats, status);
  }
  note_launch();
  return cudaGetLastError();
}

static int chunk_of(const WalkParams& wp) {
  return wp.sinks_per_warp > 0 ? wp.sinks_per_warp : kDefaultChunk;
}

cudaError_t launch_walk(const TreeView& T, const long long* sink_idx, int n_sink,
                        const WalkParams& wp, float* flux_out, int* counters,
                        unsigned long long* stats, int* status, int block_size,
                        cudaStream_t s) {
  if (n_sink <= 0) return cudaSuccess;
  (void)block_size;
  if (wp.variant >= 2)
    return launch_cut_walk(T, sink_idx, n_sink, wp, flux_out, counters, stats, status, s);
  const int chunk = chunk_of(wp);
  const long long warps = ((long long)n_sink + chunk - 1) / chunk;
  const int blocks = (int)((warps * 32 + 127) / 128);
  walk_kernel<false><<<blocks, 128, 0, s>>>(T, sink_idx, n_sink, chunk, wp,
                                            SinkOut{flux_out, counters, nullptr, nullptr, n_sink}, stats, status,
                                            AdjointArgs{});
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_walk_adjoint(const TreeView& T, const long long* sink_idx, int n_sink,
                                const WalkParams& wp, const AdjointArgs& J, int* status,
                                cudaStream_t s) {
  if (n_sink <= 0) return cudaSuccess;
  if (wp.variant >= 2) return launch_cut_adjoint(T, sink_idx, n_sink, wp, J, status, s);
  const int chunk = chunk_of(wp);
  const long long warps = ((long long)n_sink + chunk - 1) / chunk;
  const int blocks = (int)((warps * 32 + 127) / 128);
  walk_kernel<true><<<blocks, 128, 0, s>>>(T, sink_idx, n_sink, chunk, wp,
                                           SinkOut{nullptr, nullptr, nullptr, nullptr, n_sink}, nullptr, status, J);
  note_launch();
  return cudaGetLastError();
}

}  // namespace trevr
