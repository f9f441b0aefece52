// The flux walk of the warp variants (2 and 3): source walk, reverse rays and flux sum.
//
// The 32 lanes of a warp (32 consecutive sinks in Morton order) walk one depth-first
// stack in shared memory, with a mask of the lanes that still need each cell. A lane
// that accepts a cell, or reaches a source of an opened leaf, keeps that ray waiting; when a
// lane with a waiting ray gets another, the waiting rays of all lanes are traced together.
//
// Where a call has too few sinks to fill the GPU with a warp per 32, a block of several warps
// takes the same 32 sinks: each walks the source tree, and the takings (a cell accepted by some
// lanes, a source reached) are dealt out to the warps by what is taken, a hash of the cell's
// number or the source's. A sink's flux is summed in kSlots compensated parts, dealt out in the
// same way whether or not warps share a group: it depends neither on that nor on the other
// sinks of the group, and so not on the list that the sink stands in, or that list's order.
// Three kinds of sums keep this to rounding only. Bands and moments are summed by warp, without
// parts, and go by the number of warps, that is by how many sinks the call has (8 parts of each
// in local memory took 9.3 ms for three bands of 200003 sinks instead of 8.0, and 9.5 for the
// moments of 262144 instead of 7.5). The particle trace, whose rays are the longest, numbers
// the takings as the group comes to them, which spreads them more evenly.
//
// A ray is a list of pieces along [0, 1] (p + t d). All of them are cut from the clip of
// the common ancestor A of the sink's leaf S and the source's cell C: a cell's interval
// at its split plane, at t = (plane - p) * (1/d), gives the intervals of its children. On
// the same fp32 planes this is exactly the children's own slab clip, since boxes nest, the
// per-face t is monotone in the plane, and min and max are exact. So
//   * the two paths from A to C and to S are followed by cell records, one cut a level,
//     and only the siblings that the ray crosses become pieces (the C side in a
//     first-in-first-out list, in the ray's order; the S side on the stack above it);
//   * a piece that Eq. refcrit refines is cut in two: the nearer child goes on, the
//     farther one waits on the stack with the end of its interval. Pieces are taken in the
//     ray's order, so a piece begins where the one before it ended, and an entry is
//     (cell, end).
// Rounding can put a sink or a source an ulp outside its own cell. The siblings that then lie
// before the sink's path, or behind the source's, are set aside at the list's upper end and
// put into their place when the path is done. Cell 0 is an empty leaf: the entry (0, t) moves
// the ray on to t, where a sink is on the wrong side of A's own split plane.
//
// The adjoint (ADJ) follows the same pieces. Each has the axis of the plane it starts at, so
// that d(tau)/dq needs one term per boundary, t (abar behind - abar before) / d_k, and
// tau / s^2 d for the stretch of the ray; its segments are kept (cell, length) and replayed
// into the cells' sums once the ray's contribution f is known.
#include <cuda_runtime.h>
#include <stdint.h>

#include "trevr_internal.cuh"
#include "walk_common.cuh"

namespace trevr {

namespace {

// Pieces of a ray. From an ancestor A at depth ds to leaves at depth kDepth - 1 at most, either
// path has kDepth - 2 - ds siblings and its end. The C side waits whole, behind it the entry
// (0, t) and the S side but for the piece being walked; that one lies below depth ds + 1, and
// has one waiting child a level. While the list is made there are no waiting children, and the
// siblings set aside (at most one plane per axis lies within an ulp of a point; kSpare bounds
// them whatever the domain's planes are) take the upper end: they are siblings of the path, so
// the entries of both ends stay below kPieces together. The list is most of a thread's stack,
// which the driver sets aside for all threads that the GPU holds.
constexpr int kPieces = 3 * kDepth;
constexpr int kSpare = 20;
static_assert((kDepth - 1) + 1 + (kDepth - 2) + (kDepth - 3) <= kPieces,
              "the list holds every piece of a ray");
constexpr int kSegBuf = 64;  // segments of one ray kept for the adjoint's replay

constexpr int kSlots = 8;    // parts of a sink's flux; at most as many warps per group

// A warp's shared memory: the walk's stack, (cell, mask of the lanes that need it) and the
// place in a stack that holds dark cells too (stack_depth limits that one), and the queue of
// the particle trace.
template <bool SUB>
struct __align__(16) CutStack {
  float4 queue[SUB ? 64 : 1];
  int2 e[kDepth + 2];
  unsigned char place[kDepth + 2];
};

// A warp's share of a group's takings: those whose number & (parts - 1) is part. parts is a
// power of two, at most kSlots.
struct Share {
  int part, parts;
  __device__ __forceinline__ bool has(int number) const { return (number & (parts - 1)) == part; }
};

// The slot of a taking of cells, from the cell alone; a source's is its number. Against takings
// numbered as the group comes to them, the hash takes 6.4 instead of 6.9 ms for 100003 sinks
// and 9.2 instead of 9.5 for a background field of 32768 (more rays of a warp go to the same
// cells), but 13.7 instead of 13.0 for the particle trace of 8000, 33.9 instead of 33.2 of
// 65536. Numbered by lane, the rays that a warp traces together go to different cells: 12.6 ms
// for the background field, and 57.5 instead of 56.0 at 2^22 sinks.
__device__ __forceinline__ int cell_slot(int cell) {
  return (int)((unsigned)cell * 2654435761u >> 29);
}
static_assert(kSlots == 8, "the hash has three bits");

// Compensated sums of one lane's takings, one per slot.
struct Slots {
  float2 v[kSlots];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < kSlots; ++k) v[k] = make_float2(0.0f, 0.0f);
  }
  __device__ __forceinline__ void add(int k, float f) {
    CSum t;
    t.s = v[k].x;
    t.c = v[k].y;
    t.add(f);
    v[k] = make_float2(t.s, t.c);
  }
};

// s + c of a part joins the sum
__device__ __forceinline__ void join(CSum& sum, float2 part) {
  sum.add(part.x);
  sum.c = __fadd_rn(sum.c, part.y);
}

// ---------------------------------------------------------------------------
// Sub-bucket particle trace (Sec. 2.2.3, 3.1.3). The absorption below the bucket
// scale is the SPH field sum_j alpha_j w_j W(|x - x_j|, h_j), W(r, h) = w(r/h)/(pi h^3)
// the cubic spline of support 2h. Along a ray at impact parameter b from x_j, with s
// measured from the closest approach, the column over [s0, s1] is
// (Phi(x, s1/h) - Phi(x, s0/h)) / (pi h^2), x = b^2/h^2, where Phi(x, sigma) is the
// integral of w(sqrt(x + t^2)) over t in [0, sigma]: odd in sigma and constant beyond
// the support. Phi comes from the tree's pre-computed table (the paper's pre-computed
// kernel integral), bilinear in (x, sigma).
__device__ __forceinline__ float kint_phi(const float4* __restrict__ tab, float x, float sigma) {
  const float a = fminf(fabsf(sigma), 2.0f);
  const float fx = x * (0.25f * (float)kKintNX), fs = a * (0.5f * (float)kKintNS);
  const int i = min((int)fx, kKintNX - 1), j = min((int)fs, kKintNS - 1);
  const float u = fx - (float)i, v = fs - (float)j;
  const float4 c = __ldg(tab + (size_t)i * kKintNS + j);  // the cell's four corners
  const float p0 = fmaf(v, c.y - c.x, c.x);
  const float p1 = fmaf(v, c.w - c.z, c.z);
  const float p = fmaf(u, p1 - p0, p0);
  return sigma < 0.0f ? -p : p;
}

// Optical depth of lane src's chord p + t d, t in [t0, t1], through the particles
// listed for its leaf, the receiving particle (sorted index si) left out. The 32
// lanes of the warp test one neighbour each per round, with the next round's
// entries already loading; the neighbours that reach the chord are queued in shared
// memory, as (x, sigma_0, sigma_1, alpha w / (pi h^2)), and integrated 32 at a time:
// (Phi(x, sigma_1) - Phi(x, sigma_0)) times alpha w / (pi h^2), with x = b^2 / h^2 and
// sigma = s / h. Every lane must call it;
// all lanes return the sum.
__device__ __forceinline__ float sub_bucket_tau_warp(const TreeView& T, int src, int box, int si,
                                                     float px, float py, float pz, float dx,
                                                     float dy, float dz, float s2, float len,
                                                     float t0, float t1,
                                                     float4* __restrict__ queue) {
  const unsigned FULL = 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  box = __shfl_sync(FULL, box, src);
  si = __shfl_sync(FULL, si, src);
  px = __shfl_sync(FULL, px, src);
  py = __shfl_sync(FULL, py, src);
  pz = __shfl_sync(FULL, pz, src);
  dx = __shfl_sync(FULL, dx, src);
  dy = __shfl_sync(FULL, dy, src);
  dz = __shfl_sync(FULL, dz, src);
  s2 = __shfl_sync(FULL, s2, src);
  len = __shfl_sync(FULL, len, src);
  t0 = __shfl_sync(FULL, t0, src);
  t1 = __shfl_sync(FULL, t1, src);
  const float inv_s2 = 1.0f / s2;
  float part = 0.0f;
  int qn = 0;  // queued entries (warp-uniform)
  const unsigned k0 = __ldg(&T.nbr_first[box]), k1 = __ldg(&T.nbr_first[box + 1]);
  int2 nja = make_int2(-1, 0);  // the next round's entries
  float4 nq = make_float4(0.0f, 0.0f, 0.0f, 1.0f);
  if (k0 + lane < k1) {
    nja = __ldg(&T.nbr_ja[k0 + lane]);
    nq = __ldg(&T.nbr_sp[k0 + lane]);
  }
  for (unsigned base = k0; base < k1; base += 32u) {
    const unsigned k = base + lane;
    const int2 ja = nja;
    const float4 q = nq;
    if (k + 32u < k1) {
      nja = __ldg(&T.nbr_ja[k + 32u]);
      nq = __ldg(&T.nbr_sp[k + 32u]);
    }
    const float a = __int_as_float(ja.y);
    bool pass = false;
    float x = 0.0f, sa = 0.0f, sb = 0.0f;
    if (k < k1 && ja.x != si && a > 0.0f) {
      const float ux = q.x - px, uy = q.y - py, uz = q.z - pz;
      const float tc = (ux * dx + uy * dy + uz * dz) * inv_s2;
      const float ex = ux - tc * dx, ey = uy - tc * dy, ez = uz - tc * dz;
      const float b2 = ex * ex + ey * ey + ez * ez;
      const float ih = q.w;
      x = b2 * ih * ih;
      sa = ((t0 - tc) * len) * ih;
      sb = ((t1 - tc) * len) * ih;
      if (x < 4.0f) {  // the chord [sa, sb] must meet the support |sigma| < sqrt(4 - x)
        const float u22 = 4.0f - x;
        pass = (sb > 0.0f || sb * sb < u22) && (sa < 0.0f || sa * sa < u22);
      }
    }
    const unsigned m = __ballot_sync(FULL, pass);
    if (pass) {
      const float ih = q.w;
      queue[qn + __popc(m & ((1u << lane) - 1u))] =
          make_float4(x, sa, sb, a * (ih * ih * 0.318309886f));
    }
    qn += __popc(m);
    __syncwarp();
    if (qn >= 32) {
      const float4 g = queue[qn - 32 + (int)lane];
      part += g.w * (kint_phi(T.kint4, g.x, g.z) - kint_phi(T.kint4, g.x, g.y));
      qn -= 32;
      __syncwarp();
    }
  }
  if ((int)lane < qn) {
    const float4 g = queue[lane];
    part += g.w * (kint_phi(T.kint4, g.x, g.z) - kint_phi(T.kint4, g.x, g.y));
  }
  __syncwarp();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
  return part;
}

__device__ __forceinline__ unsigned cell_link(const float4& r) { return __float_as_uint(r.w); }
__device__ __forceinline__ bool is_leaf(unsigned link) { return (link & 3u) == 3u; }
__device__ __forceinline__ int lower_child(unsigned link) { return (int)((link >> 1) & ~1u); }

// A ray from the sink p: direction d, and 1/d per axis. Along an axis that the ray does not
// move on, 1/d is the largest float: (plane - p) * inv is then <= 0 for p >= plane and
// beyond 1 for p < plane, so the cuts give the half-open boxes [lo, hi) of that case.
struct Line {
  float px, py, pz, dx, dy, dz, ix, iy, iz, s2, len;
  __device__ __forceinline__ static float inverse(float d) {
    return d != 0.0f ? __frcp_rn(d) : 3.402823466e38f;
  }
  __device__ __forceinline__ void aim(float qx, float qy, float qz) {
    dx = __fsub_rn(qx, px);
    dy = __fsub_rn(qy, py);
    dz = __fsub_rn(qz, pz);
    s2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
    len = __fsqrt_rn(s2);
    ix = inverse(dx);
    iy = inverse(dy);
    iz = inverse(dz);
  }
  // where the ray crosses the split plane of r; forward: it goes to the upper child
  __device__ __forceinline__ float cross(const float4& r, bool& forward) const {
    const unsigned ax = cell_link(r) & 3u;
    const float p = ax == 0u ? px : (ax == 1u ? py : pz);
    const float i = ax == 0u ? ix : (ax == 1u ? iy : iz);
    forward = i > 0.0f;
    return __fmul_rn(__fsub_rn(r.z, p), i);
  }
  __device__ __forceinline__ void clip_axis(float lo, float hi, float p, float i, float& t0,
                                            float& t1) const {
    const float ta = __fmul_rn(__fsub_rn(lo, p), i), tb = __fmul_rn(__fsub_rn(hi, p), i);
    t0 = fmaxf(t0, fminf(ta, tb));
    t1 = fminf(t1, fmaxf(ta, tb));
  }
  __device__ __forceinline__ void clip(const float4& lo, const float4& hi, float& t0,
                                       float& t1) const {
    t0 = 0.0f;
    t1 = 1.0f;
    clip_axis(lo.x, hi.x, px, ix, t0, t1);
    clip_axis(lo.y, hi.y, py, iy, t0, t1);
    clip_axis(lo.z, hi.z, pz, iz, t0, t1);
  }
};

// Background sources (Sec. 2.2.4): the centre of luminosity of an accepted cell moved
// radially onto the sphere of radius P.bg_radius around the domain centre o (side / 2 in
// coordinates relative to the lower corner), in fp32 as d = c - o,
// s = sqrt((dx^2 + dy^2) + dz^2), q = o + d * (R / s); and the leaf that holds q (grid
// coordinates clamped to the grid), found by descending the cut planes from the root, with
// its path.
__device__ __forceinline__ void bg_end(const TreeView& T, const WalkParams& P, float& qx,
                                       float& qy, float& qz, int& Y, unsigned long long& way) {
  const float o = __fmul_rn(T.side, 0.5f);
  const float ddx = __fsub_rn(qx, o), ddy = __fsub_rn(qy, o), ddz = __fsub_rn(qz, o);
  const float sn = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(ddx, ddx), __fmul_rn(ddy, ddy)),
                                        __fmul_rn(ddz, ddz)));
  if (sn > 0.0f) {
    const float kk = __fdiv_rn(P.bg_radius, sn);
    qx = __fadd_rn(o, __fmul_rn(ddx, kk));
    qy = __fadd_rn(o, __fmul_rn(ddy, kk));
    qz = __fadd_rn(o, __fmul_rn(ddz, kk));
  }
  const float scale = __fdiv_rn(2097152.0f, T.side);
  const float q[3] = {qx, qy, qz};
  int g[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    float t = __fmul_rn(q[d], scale);
    if (!(t >= 0.0f)) t = 0.0f;
    const unsigned v = __float2uint_rz(t);
    g[d] = (int)(v > (unsigned)(kGridMax - 1) ? (unsigned)(kGridMax - 1) : v);
  }
  Y = kRoot;
  for (int it = 0; it < kDepth - 1; ++it) {
    const int ch = __ldg(&T.nT[Y].x);
    if (ch < 0) break;
    const int ax = __ldg(&T.nglo[Y].w);
    const int4 up = __ldg(&T.nglo[ch + 1]);
    const int gv = ax == 0 ? g[0] : (ax == 1 ? g[1] : g[2]);
    const int plane = ax == 0 ? up.x : (ax == 1 ? up.y : up.z);
    Y = gv >= plane ? ch + 1 : ch;
  }
  way = __ldg(&T.nD[Y]);
}

__device__ __forceinline__ int way_depth(unsigned long long way) {
  return 64 - __ffsll((long long)way);
}

// The sink of a lane: sorted index, dLoss/dF (adjoint), and the path of its leaf.
struct Sink {
  int i;
  float grad;
  unsigned long long way;
};

// The pieces of a lane's ray that wait: in [head, n_fifo) in the ray's order, in
// [n_fifo, n) as a stack that is taken first. axis: of the plane that a piece starts at
// (adjoint; 3 = none).
template <bool ADJ>
struct Pieces {
  int2 e[kPieces];  // (cell, end)
  unsigned char axis[ADJ ? kPieces : 1];
  __device__ __forceinline__ void put(int at, int cell, float end, unsigned ax) {
    e[at] = make_int2(cell, __float_as_int(end));
    if (ADJ) axis[at] = (unsigned char)ax;
  }
  __device__ __forceinline__ void move(int to, int from) {
    e[to] = e[from];
    if (ADJ) axis[to] = axis[from];
  }
};

// Sum of v over the lanes that asked (key >= 0) when they all name the same cell,
// else one atomic per lane. Every lane of the warp must call it.
__device__ __forceinline__ void warp_atomic_add(double* base, int key, float v) {
  const unsigned FULL = 0xffffffffu;
  const unsigned want = __ballot_sync(FULL, key >= 0);
  if (!want) return;
  const int k0 = __shfl_sync(FULL, key, __ffs(want) - 1);
  if (__all_sync(FULL, key < 0 || key == k0)) {
    float x = key >= 0 ? v : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&base[k0], (double)x);
  } else if (key >= 0) {
    atomicAdd(&base[key], (double)v);
  }
}

// The adjoint's segment terms scale * length into the cells' FP64 sums: the k-th from the
// end of every lane's list together, since neighbouring sinks' rays to one source share their
// last cells. Where 8 or more lanes name the same cell, they are summed in FP64 first. One
// atomic per lane and segment took 18 of the 50 ms of a backward pass at 2^20 sinks; this
// takes 6 (thresholds of 4 to 12 lanes and two more rounds of matching are within 1%).
__device__ __forceinline__ void add_segments(double* G, const int2* seg, int n, float scale) {
  const unsigned FULL = 0xffffffffu;
  const int most = __reduce_max_sync(FULL, n);
  for (int k = 1; k <= most; ++k) {
    int cell = -1;
    double v = 0.0;
    if (k <= n) {
      const int2 e = seg[n - k];
      cell = e.x;
      v = (double)(scale * __int_as_float(e.y));
    }
    const unsigned want = __ballot_sync(FULL, cell >= 0);
    const int c0 = __shfl_sync(FULL, cell, __ffs(want) - 1);
    const unsigned same = __ballot_sync(FULL, cell == c0);
    if (__popc(same) >= 8) {
      double x = cell == c0 ? v : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
      if ((int)(threadIdx.x & 31u) == __ffs(same) - 1) atomicAdd(&G[c0], x);
      if (cell == c0) cell = -1;
    }
    if (cell >= 0) atomicAdd(&G[cell], v);
  }
}

// One ray per lane that is `on`, from its sink to `ent` (a cell, or ~source); every lane of
// the warp must call it. The loop ends: a refined piece goes on at a child, whose number is
// larger than its parent's, and every entry of the list is taken once.
// STOP: a ray whose running optical depth passes P.tau_stop ends and adds nothing (Sec. 4);
// its segments and refinements are counted up to there.
// NB > 1: every band sums its own optical depth over the shared segments.
// SUB: a leaf whose own particles ask for refinement is integrated through them.
// TD: the top-down ray walk: A is the only piece, and Eq. refcrit alone splits it.
// ADJ: the terms of the adjoint instead of the flux. A ray with more segments than are kept
// is traced a second time.
template <bool ADJ, bool MOM, bool BG, bool STOP, int NB, bool SUB, bool CNT, bool TD>
__device__ __forceinline__ void cut_ray(const TreeView& T, const WalkParams& P, const float tref,
                                        const bool on, const int ent, const Sink& K, Line& ray,
                                        Pieces<ADJ>& W, const AdjointArgs& J, SinkCounters& cnt,
                                        const int slot, Slots& flux, CSum* F, Moments* mom,
                                        float4* queue) {
  const unsigned FULL = 0xffffffffu;
  float L = 0.0f;
  int C = kRoot;
  unsigned long long wayC = 0;
  bool traced = false;
  ray.s2 = ray.len = 1.0f;
  if (on) {
    float qx, qy, qz;
    if (ent < 0) {
      const float4 y = __ldg(&T.src[~ent]);
      qx = y.x;
      qy = y.y;
      qz = y.z;
      L = y.w;
      C = __ldg(&T.src_leaf[~ent]);
      wayC = __ldg(&T.nD[C]);
    } else {
      const float4 s = __ldg(&T.nS[ent]);
      qx = s.x;
      qy = s.y;
      qz = s.z;
      L = s.w;
      C = ent;
      if (BG) bg_end(T, P, qx, qy, qz, C, wayC);
      else wayC = __ldg(&T.nD[C]);
    }
    ray.aim(qx, qy, qz);
    traced = !(ray.s2 < P.smin2);  // a source on top of the sink adds nothing
  }
  KSum tau;
  KSum taub[NB];  // (NB > 1) optical depth of each band
  bool cut = false;
  // adjoint: the segments of the first pass, the gradient's boundary sums, and f
  int2 seg[ADJ ? kSegBuf : 1];
  int n_seg = 0;
  float gx = 0.0f, gy = 0.0f, gz = 0.0f, before = 0.0f, f = 0.0f;
  bool active = traced, again = false;
  do {
    int n_fifo = 0, n = 0, head = 0;
    int box = 0;
    unsigned ax = 3u;  // (ADJ) axis of the plane at t0
    float t0 = 0.0f, t1 = 0.0f;
    if (active) {
      const int dS = way_depth(K.way), dC = way_depth(wayC);
      const int ds = min(min(__clzll((long long)(K.way ^ wayC)), dS), dC);
      // A: down from the root along the shared path
      unsigned long long way = K.way;
      int cell = kRoot;
      float4 r = __ldg(&T.nR[kRoot]);
      for (int k = 0; k < ds; ++k) {
        cell = lower_child(cell_link(r)) + (int)(way >> 63);
        way <<= 1;
        r = __ldg(&T.nR[cell]);
      }
      float a, b;
      ray.clip(__ldg(&T.nV[2 * (size_t)cell]), __ldg(&T.nV[2 * (size_t)cell + 1]), a, b);
      if (TD || ds == dS || ds == dC) {  // one piece: A, or S = C
        if (CNT) ++cnt.clip;
        if (a < b) {
          box = cell;
          t0 = a;
          t1 = b;
        }
      } else {
        if (CNT) cnt.clip += dS + dC - 2 * ds;
        if (!(a < b)) a = b = 0.0f;  // the clip may be at infinity (1/d overflows)
        bool fwd;
        const float t = ray.cross(r, fwd);
        int up = (int)(way >> 63);
        const int child = lower_child(cell_link(r));
        const unsigned axA = cell_link(r) & 3u;
        const bool far_s = fwd == (up != 0);  // rounding only: the sink's child is the far one
        float aC = far_s ? a : fmaxf(a, t), bC = far_s ? fminf(b, t) : b;
        float aS = far_s ? fmaxf(a, t) : a, bS = far_s ? b : fminf(b, t);
        const float startC = aC, startS = aS;
        int aside = 0;
        if (aC < bC) {  // the C side, in the ray's order
          unsigned axC = far_s ? 3u : axA;
          int X = child + (up ^ 1);
          unsigned long long w = wayC << (ds + 1);
          for (int k = ds + 1; k < dC && aC < bC; ++k) {
            r = __ldg(&T.nR[X]);
            const float tc = ray.cross(r, fwd);
            const int u = (int)(w >> 63);
            w <<= 1;
            X = lower_child(cell_link(r)) + u;
            if (fwd == (u != 0)) {  // the sibling lies before the path
              const float e = fminf(bC, tc);
              if (aC < e) {
                W.put(n++, X ^ 1, e, axC);
                axC = cell_link(r) & 3u;
              }
              aC = fmaxf(aC, tc);
            } else {  // behind it: rounding only
              if (fmaxf(aC, tc) < bC && aside < kSpare)
                W.put(kPieces - ++aside, X ^ 1, bC, cell_link(r) & 3u);
              bC = fminf(bC, tc);
            }
          }
          if (aC < bC) W.put(n++, X, bC, axC);
          for (; aside > 0; --aside) W.move(n++, kPieces - aside);
        }
        n_fifo = n;
        if (aS < bS) {
          if (n_fifo > 0 && bS != startC) W.put(n++, 0, startC, 3u);
          unsigned axS = far_s ? axA : 3u;
          int X = child + up;
          way <<= 1;
          for (int k = ds + 1; k < dS && aS < bS; ++k) {
            r = __ldg(&T.nR[X]);
            const float tc = ray.cross(r, fwd);
            up = (int)(way >> 63);
            way <<= 1;
            X = lower_child(cell_link(r)) + up;
            if (fwd != (up != 0)) {  // the sibling lies behind the path
              if (fmaxf(aS, tc) < bS) W.put(n++, X ^ 1, bS, cell_link(r) & 3u);
              bS = fminf(bS, tc);
            } else {  // before it: rounding only
              const float e = fminf(bS, tc);
              if (aS < e && aside < kSpare) {
                W.put(kPieces - ++aside, X ^ 1, e, axS);
                axS = cell_link(r) & 3u;
              }
              aS = fmaxf(aS, tc);
            }
          }
          t0 = t1 = startS;
          if (aside > 0) {
            if (aS < bS) W.put(n++, X, bS, axS);
            for (; aside > 1; --aside) W.move(n++, kPieces - aside);
            box = W.e[kPieces - 1].x;
            t1 = __int_as_float(W.e[kPieces - 1].y);
          } else if (aS < bS) {
            box = X;
            t1 = bS;
          }
          if (ADJ) ax = far_s ? axA : 3u;
        } else if (n_fifo > 0) {
          t0 = t1 = startC;
        }
      }
    }
    while (__any_sync(FULL, active)) {
      bool need_sub = false;
      int sub_box = 0;
      float sub_t0 = 0.0f, sub_t1 = 0.0f;
      if (active) {
        const float4 r = __ldg(&T.nR[box]);
        const unsigned link = cell_link(r);
        const float l = __fmul_rn(__fsub_rn(t1, t0), ray.len);
        if (__fmul_rn(r.y, l) > tref && !is_leaf(link)) {
          bool fwd;
          const float t = ray.cross(r, fwd);
          const int near = lower_child(link) + (fwd ? 0 : 1);
          const bool hit_near = t > t0, hit_far = t < t1;
          if (CNT) {
            ++cnt.ref;
            cnt.clip += (int)hit_near + (int)hit_far;
          }
          if (hit_near && hit_far) {
            W.put(n++, near ^ 1, t1, link & 3u);
            t1 = t;
          }
          box = hit_near ? near : near ^ 1;
        } else {
          if (NB > 1) {
            const float4 ab = __ldg(&T.bA[box]);
            taub[0].add(__fmul_rn(ab.x, l));
            taub[1].add(__fmul_rn(ab.y, l));
            if (NB > 2) {
              taub[NB > 2 ? 2 : 0].add(__fmul_rn(ab.z, l));
              taub[NB > 2 ? 3 : 0].add(__fmul_rn(ab.w, l));
            }
          } else if (SUB && box != 0 && is_leaf(link) && l > 0.0f &&
                     __fmul_rn(__ldg(&T.dbk[box]), l) > tref) {
            // a bucket that still asks for refinement: its particles are traced by the
            // whole warp at the end of this step
            need_sub = true;
            sub_box = box;
            sub_t0 = t0;
            sub_t1 = t1;
            if (CNT) ++cnt.sub;
          } else if (!ADJ || !again) {
            tau.add(__fmul_rn(r.x, l));
          }
          if (CNT && box != 0 && l > 0.0f) ++cnt.segs;
          if (ADJ) {
            if (again) {
              if (l > 0.0f) atomicAdd(&J.G[box], (double)(-K.grad * f * l));
            } else {
              const float jump = (r.x - before) * t0;
              gx += ax == 0u ? jump : 0.0f;
              gy += ax == 1u ? jump : 0.0f;
              gz += ax == 2u ? jump : 0.0f;
              before = r.x;
              if (l > 0.0f && box != 0) {
                if (n_seg < kSegBuf) seg[n_seg] = make_int2(box, __float_as_int(l));
                ++n_seg;
              }
            }
          }
          t0 = t1;
          const bool stacked = n > n_fifo;
          active = stacked || head < n_fifo;
          if (STOP && tau.get() > P.tau_stop) {
            cut = true;
            active = false;
          }
          if (active) {
            const int at = stacked ? n - 1 : head;
            const int2 e = W.e[at];
            if (ADJ) ax = W.axis[at];
            n -= stacked ? 1 : 0;
            head += stacked ? 0 : 1;
            box = e.x;
            t1 = __int_as_float(e.y);
          }
        }
      }
      if (SUB) {
        // the leaves of this step that need the particle trace, one after another
        unsigned m = __ballot_sync(FULL, need_sub);
        while (m) {
          const int src = __ffs(m) - 1;
          m &= m - 1u;
          const float t = sub_bucket_tau_warp(T, src, sub_box, K.i, ray.px, ray.py, ray.pz, ray.dx,
                                              ray.dy, ray.dz, ray.s2, ray.len, sub_t0, sub_t1,
                                              queue);
          if ((int)(threadIdx.x & 31u) == src) tau.add(t);
        }
      }
    }
    if (ADJ && !again) {
      f = L * expf(-tau.get()) / (kFourPi * ray.s2);
      active = traced && n_seg > kSegBuf;  // too many segments to replay: trace the ray again
    }
    if (!ADJ) break;
    if (again) break;
    again = true;
  } while (__any_sync(FULL, active));
  if (ADJ) {
    // the segments' terms, then the pseudo-source's. The lanes mix single sources and
    // merged cells, so every lane takes part in every warp-wide sum, naming no key (-1) for
    // a term that is not its own.
    add_segments(J.G, seg, n_seg <= kSegBuf ? n_seg : 0, -K.grad * f);
    const bool single = traced && ent < 0, merged = traced && ent >= 0;
    const float c = traced ? K.grad * f / L : 0.0f;
    const float along = 2.0f / ray.s2 + tau.get() / ray.s2;
    // d(tau)/dq: the stretch of the ray, and its boundaries (none on a still axis)
    const float bx = gx != 0.0f ? ray.len * ray.ix * gx : 0.0f;
    const float by = gy != 0.0f ? ray.len * ray.iy * gy : 0.0f;
    const float bz = gz != 0.0f ? ray.len * ray.iz * gz : 0.0f;
    warp_atomic_add(J.e, single ? ~ent : -1, c);
    warp_atomic_add(J.a, merged ? C : -1, c);
    warp_atomic_add(J.b + 0, merged ? 3 * C : -1, c * (-ray.dx * along - bx));
    warp_atomic_add(J.b + 1, merged ? 3 * C : -1, c * (-ray.dy * along - by));
    warp_atomic_add(J.b + 2, merged ? 3 * C : -1, c * (-ray.dz * along - bz));
    return;
  }
  if (!traced) return;
  if (CNT) ++cnt.rays;
  if (STOP && cut) {
    if (CNT) ++cnt.cut;
    return;
  }
  if (NB > 1) {
    // the band luminosities of the source, or of the merged cell
    const float4 Lb = ent < 0 ? __ldg(&T.bLs[~ent]) : __ldg(&T.bLc[C]);
    const float den = kFourPi * ray.s2;
    F[0].add(Lb.x * expf(-taub[0].get()) / den);
    F[1].add(Lb.y * expf(-taub[1].get()) / den);
    if (NB > 2) {
      F[NB > 2 ? 2 : 0].add(Lb.z * expf(-taub[NB > 2 ? 2 : 0].get()) / den);
      F[NB > 2 ? 3 : 0].add(Lb.w * expf(-taub[NB > 2 ? 3 : 0].get()) / den);
    }
    return;
  }
  f = L * expf(-tau.get()) / (kFourPi * ray.s2);
  flux.add(slot, f);
  if (MOM) {
    const float il = 1.0f / ray.len;
    const float n0 = -ray.dx * il, n1 = -ray.dy * il, n2 = -ray.dz * il;
    mom->v[0].add(f * n0);
    mom->v[1].add(f * n1);
    mom->v[2].add(f * n2);
    mom->v[3].add(f * n0 * n0);
    mom->v[4].add(f * n1 * n1);
    mom->v[5].add(f * n2 * n2);
    mom->v[6].add(f * n0 * n1);
    mom->v[7].add(f * n0 * n2);
    mom->v[8].add(f * n1 * n2);
  }
}

// The walk of the 32 sinks of one warp (a lane holds the sorted position i if `has`);
// every lane of the warp must call it. MERGE: a ray waits until its lane gets
// another; without it (variant 2) the rays to a cell are traced as soon as it is accepted.
// A step of the walk is a chain of loads for all lanes, and below some 10^5 sinks that chain is
// what it takes. So a cell is two 16-byte loads that are on their way together (they were five
// in three arrays, one behind another), dark children are never pushed, and an opened leaf's
// sources are looked at 32 at a time: side by side, 7.35 -> 7.05 ms at 100003 sinks, 10.8 -> 9.6
// for a background field at 32768, 0.52 -> 0.48 for a step of 4096, 54.1 -> 53.2 at 2^22.
template <bool ADJ, bool MERGE, bool MOM, bool BG, bool STOP, int NB, bool SUB, bool CNT, bool TD>
__device__ __forceinline__ void cut_walk(const TreeView& T, const WalkParams& P, const bool has,
                                         const int i, const float grad, const Share share,
                                         CutStack<SUB>& ws, int* status, const AdjointArgs& J,
                                         SinkCounters& cnt, Slots& flux, CSum* F, Moments* mom) {
  const unsigned FULL = 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  const int stack_limit = P.stack_depth < kDepth ? P.stack_depth : kDepth;
  // tau_ref <= 0 refines every cell: any l * spread >= 0 passes
  const float tref = P.tau_ref <= 0.0f ? -1.0f : P.tau_ref;
  Pieces<ADJ> W;
  Line ray;
  ray.px = ray.py = ray.pz = 0.0f;
  Sink K{i, grad, 1ull << 63};
  if (has) {
    const float4 p = T.pos[i];
    ray.px = p.x;
    ray.py = p.y;
    ray.pz = p.z;
    K.way = __ldg(&T.nD[T.leaf_of[i]]);
  }
  const unsigned live = __ballot_sync(FULL, has);
  int sp = 0;
  if (live && __ldg(&T.nS[kRoot].w) > 0.0f) {
    if (lane == 0) {
      ws.e[0] = make_int2(kRoot, (int)live);
      ws.place[0] = 0;
    }
    sp = 1;
  }
  bool wait = false;      // this lane has a ray that waits to be traced, to w_ent
  int w_ent = 0;          // (a cell, or ~source)
  int j = 0, j_end = 0;   // sources of the opened leaf from j on are still to be looked at
  unsigned opened = 0;    // the lanes that opened it
  unsigned lit = 0, own = 0;  // of the 32 sources before j: those with light, this warp's of them
  int taken = 0, first = 0;   // (SUB) takings so far, and before the first of `lit`
  int w_slot = 0;             // the waiting ray's slot
  if (!ADJ && NB == 1) flux.clear();
  __syncwarp();
  while (true) {
    bool take = false, done = false;
    int ent = 0, turn = 0;
    if (own) {
      const int q = __ffs(own) - 1;
      own &= own - 1u;
      ent = ~(j - 32 + q);
      turn = SUB ? first + __popc(lit & ((1u << q) - 1u)) : j - 32 + q;
      take = (opened >> lane) & 1u;
    } else if (j < j_end) {
      const int mine = j + (int)lane;
      const bool light = mine < j_end && __ldg(&T.src[mine].w) > 0.0f;
      lit = __ballot_sync(FULL, light);
      first = taken;
      const int number = SUB ? first + __popc(lit & ((1u << lane) - 1u)) : mine;
      own = __ballot_sync(FULL, light && share.has(number));
      taken += __popc(lit);
      j += 32;
      continue;
    } else if (sp > 0) {
      --sp;
      const int2 top = ws.e[sp];
      const int X = top.x, place = ws.place[sp];
      __syncwarp();
      const float4 lo = __ldg(&T.nV[2 * (size_t)X]), hi = __ldg(&T.nV[2 * (size_t)X + 1]);
      const unsigned below = __float_as_uint(hi.w);
      bool open = false;
      if (((unsigned)top.y >> lane) & 1u) {
        if (CNT && share.part == 0) ++cnt.visit;
        const float ex = fmaxf(fmaxf(__fsub_rn(lo.x, ray.px), __fsub_rn(ray.px, hi.x)), 0.0f);
        const float ey = fmaxf(fmaxf(__fsub_rn(lo.y, ray.py), __fsub_rn(ray.py, hi.y)), 0.0f);
        const float ez = fmaxf(fmaxf(__fsub_rn(lo.z, ray.pz), __fsub_rn(ray.pz, hi.z)), 0.0f);
        const float r2 =
            __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
        take = lo.w < __fmul_rn(P.theta2, r2);
        open = !take;
      }
      ent = X;
      const unsigned openM = __ballot_sync(FULL, open);
      if (openM) {
        const int child = (int)(below & 0x7ffffffeu);
        if (child == 0) {
          const int4 t = __ldg(&T.nT[X]);
          j = t.z;
          j_end = t.z + t.w;
          opened = openM;
        } else if (place + 2 > stack_limit) {
          if (lane == 0) atomicOr(status, kStatusStackOverflow);
          sp = 0;
        } else {  // the children with light, the lower one on top
          if (below & 1u) {
            if (lane == 0) {
              ws.e[sp] = make_int2(child + 1, (int)openM);
              ws.place[sp] = (unsigned char)place;
            }
            ++sp;
          }
          if (below >> 31) {
            if (lane == 0) {
              ws.e[sp] = make_int2(child, (int)openM);
              ws.place[sp] = (unsigned char)(place + 1);
            }
            ++sp;
          }
          __syncwarp();
        }
      }
      if (!__any_sync(FULL, take)) continue;
      turn = SUB ? taken++ : cell_slot(X);
      if (!share.has(turn)) continue;
    } else {
      done = true;
    }
    if (__any_sync(FULL, wait && (done || take || !MERGE))) {
      cut_ray<ADJ, MOM, BG, STOP, NB, SUB, CNT, TD>(T, P, tref, wait, w_ent, K, ray, W, J, cnt,
                                                    w_slot, flux, F, mom, ws.queue);
      wait = false;
    }
    if (done) break;
    if (take) {
      wait = true;
      w_ent = ent;
      w_slot = turn & (kSlots - 1);
    }
  }
}

// Issue-bound where a call fills the GPU (86% of the issue slots at 2^20 sinks): the loop over
// a ray's pieces is ~60 instructions on one 16-byte record that L1 mostly has, and what bounds
// the walk is how many of them it runs. Clipping every base cell and refined child instead
// (~120 instructions on 44 bytes, 53 a ray where 35 are crossed) takes 124 ms a step at 2^22
// sinks and 2^14 clumped sources, the cut pieces take 60 (in turn, among other work; a rested
// GPU takes 118 and 52), and 22.3 and 6.7 ms at 100003 sinks, tau_ref = 0.01.
// Blocks of 128 per SM: 8 leave the plain walk its registers (54, no spills); when it took 57.3
// ms at 2^22 sinks and 8.4 at 100003, 12 and 16 blocks (40 and 32 registers) gave 58.9 and 55.9,
// but 9.5 and 10.1 at 100003, where a warp's own speed counts. The particle trace waits for L2
// and wants warps: 5 blocks (94 registers) take 33.0 ms at 2^16 sinks, 4 take 36.8 and 6, which
// spill, 36.1. The bands take 6 (8.95 ms for three at 200003 sinks, 9.2 at 8; 8.1 now).
constexpr int cut_blocks(bool SUB, int NB) { return SUB ? 5 : NB > 1 ? 6 : 8; }
// warps per group at most: the particle trace keeps 5 blocks of 4
constexpr int most_warps(bool SUB) { return SUB ? 4 : kSlots; }

// SHARED: the block's warps (a power of two, at most kSlots) share one group of 32 sinks.
template <bool SHARED, bool MERGE, bool MOM, bool BG, bool STOP, int NB, bool SUB, bool CNT,
          bool TD>
__global__ void __launch_bounds__(SHARED && !SUB ? 32 * kSlots : 128,
                                  SHARED && !SUB ? cut_blocks(SUB, NB) / 2 : cut_blocks(SUB, NB))
    cut_walk_kernel(TreeView T, const long long* sink_idx, int n_sink, WalkParams P, SinkOut out,
                    unsigned long long* stats, int* status) {
  // the warps' stacks, and after the walk the parts of the group's sums
  extern __shared__ float4 block_memory[];
  CutStack<SUB>* stacks = reinterpret_cast<CutStack<SUB>*>(block_memory);
  float2(*parts)[32] = reinterpret_cast<float2(*)[32]>(block_memory);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Share share = SHARED ? Share{warp, (int)(blockDim.x >> 5)} : Share{0, 1};
  const int k = SHARED ? blockIdx.x * 32 + lane : blockIdx.x * 128 + threadIdx.x;
  SinkCounters cnt;
  int i = 0, slot = 0;
  float g = 0.0f;
  bool has = false;
  if (k < n_sink) {
    PlainMap<false> map{&T, sink_idx, nullptr, status, P.order, n_sink};
    has = map(k, i, slot, g);
    if (!has && sink_idx && slot >= 0 && share.part == 0) {
      if (out.flux)
        for (int b = 0; b < (NB > 1 ? T.n_bands : 1); ++b)
          out.flux[(size_t)b * out.n_out + slot] = 0.0f;
      if (out.counters) reinterpret_cast<int4*>(out.counters)[slot] = make_int4(0, 0, 0, 0);
    }
  }
  Slots flux;
  CSum F[NB];
  Moments mom;
  if (__any_sync(0xffffffffu, has))
    cut_walk<false, MERGE, MOM, BG, STOP, NB, SUB, CNT, TD>(
        T, P, has, i, 0.0f, share, stacks[warp], status, AdjointArgs{}, cnt, flux, F,
        MOM ? &mom : nullptr);
  else if (NB == 1)
    flux.clear();
  if (CNT && stats) add_stats(cnt, stats);
  if (SHARED) __syncthreads();
  // the group's sums, in warp 0 (every warp of the block comes here)
  auto gather = [&](CSum& v) {
    parts[SHARED ? warp : 0][lane] = make_float2(v.s, v.c);
    __syncthreads();
    if (warp == 0)
      for (int w = 1; w < share.parts; ++w) join(v, parts[SHARED ? w : 0][lane]);
    __syncthreads();
  };
  if (NB == 1) {
    if (SHARED) {
#pragma unroll
      for (int q = 0; q < kSlots; ++q)
        if ((q & (share.parts - 1)) == share.part) parts[SHARED ? q : 0][lane] = flux.v[q];
      __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < kSlots; ++q) join(F[0], SHARED ? parts[SHARED ? q : 0][lane] : flux.v[q]);
    if (SHARED) __syncthreads();
  } else if (SHARED) {
#pragma unroll
    for (int b = 0; b < NB; ++b) gather(F[b]);
  }
  if (MOM && SHARED) {
#pragma unroll
    for (int q = 0; q < 9; ++q) gather(mom.v[q]);
  }
  if (CNT && SHARED && out.counters) {
    __shared__ int counted[3][32];
    if (warp == 0) counted[0][lane] = counted[1][lane] = counted[2][lane] = 0;
    __syncthreads();
    atomicAdd(&counted[0][lane], cnt.rays);
    atomicAdd(&counted[1][lane], cnt.segs);
    atomicAdd(&counted[2][lane], cnt.ref);
    __syncthreads();
    cnt.rays = counted[0][lane];
    cnt.segs = counted[1][lane];
    cnt.ref = counted[2][lane];
  }
  if (!has || warp >= (SHARED ? 1 : 4)) return;
  if (MOM) {
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (out.fvec) out.fvec[(size_t)q * out.n_out + slot] = mom.v[q].get();
#pragma unroll
    for (int q = 0; q < 6; ++q)
      if (out.press) out.press[(size_t)q * out.n_out + slot] = mom.v[3 + q].get();
  }
  if (NB > 1) {
    // band-major output: band b of sink slot at b * n_out + slot
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (out.flux && b < T.n_bands) out.flux[(size_t)b * out.n_out + slot] = F[b].get();
  } else if (out.flux) {
    out.flux[slot] = F[0].get();
  }
  if (out.counters)
    reinterpret_cast<int4*>(out.counters)[slot] = make_int4(cnt.rays, cnt.segs, cnt.visit, cnt.ref);
}

// Batched form: each work item is cut into groups of 32 consecutive sinks, one warp walk
// per group.
template <int BS, bool MERGE, bool CNT>
__global__ void __launch_bounds__(BS, 1024 / BS) cut_walk_batched_kernel(
    const TreeView* __restrict__ views, float* const* __restrict__ flux_out,
    const int2* __restrict__ items, int n_items, int item, unsigned* counter, WalkParams P,
    unsigned long long* stats, int* status) {
  __shared__ CutStack<false> stacks[BS / 32];
  CutStack<false>& ws = stacks[threadIdx.x >> 5];
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
    const int end = min(w.y + item, T.n_gas);
    for (int g0 = w.y; g0 < end; g0 += 32) {
      const int i = g0 + (int)lane;
      const bool has = i < end;
      Slots flux;
      CSum F;
      cut_walk<false, MERGE, false, false, false, 1, false, CNT, false>(
          T, Pt, has, i, 0.0f, Share{0, 1}, ws, status, AdjointArgs{}, tot, flux, &F, nullptr);
#pragma unroll
      for (int q = 0; q < kSlots; ++q) join(F, flux.v[q]);
      if (has) flux_out[w.x][T.perm[i]] = F.get();
    }
  }
  if (CNT && stats) add_stats(tot, stats);
}

// The adjoint walk; a sink with dLoss/dF = 0 is left out. Flux and gradients of 2^20 sinks
// and 1024 sources take 58.2 ms (121 when each cell was clipped and its bounding planes
// tracked), 25 of them the flux; 4 to 10 blocks per SM lie within 9%, 8 is the fastest.
template <bool SHARED, bool MERGE>
__global__ void __launch_bounds__(SHARED ? 32 * kSlots : 128, SHARED ? 4 : 8)
    cut_adjoint_kernel(TreeView T, const long long* sink_idx, int n_sink, WalkParams P, int* status,
                       AdjointArgs J) {
  extern __shared__ float4 block_memory[];
  CutStack<false>* stacks = reinterpret_cast<CutStack<false>*>(block_memory);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Share share = SHARED ? Share{warp, (int)(blockDim.x >> 5)} : Share{0, 1};
  const int k = SHARED ? blockIdx.x * 32 + lane : blockIdx.x * 128 + threadIdx.x;
  SinkCounters cnt;
  int i = 0, slot = 0;
  float g = 0.0f;
  bool has = false;
  if (k < n_sink) {
    PlainMap<true> map{&T, sink_idx, J.grad_flux, status, P.order, n_sink};
    has = map(k, i, slot, g);
  }
  Slots none;
  if (__any_sync(0xffffffffu, has))
    cut_walk<true, MERGE, false, false, false, 1, false, false, false>(
        T, P, has, i, g, share, stacks[warp], status, J, cnt, none, nullptr, nullptr);
}

// Warps per group of 32 sinks: doubled while the call then has at most 64 warps on each SM (152
// SMs where this was measured). At 32768 sinks of a background field 8 take 9.2 ms (1: 28.4,
// 2: 15.5, 4: 10.2); at 100003 sinks 2 take 6.37 (1: 7.27, 4: 6.25, 8: 6.82); at 65536 sinks with
// the particle trace 4 take 33.2 (1: 52.4, 2: 39.2); at 262144 sinks one warp takes 7.10 and 2
// take 7.18, 4 take 7.94, since every warp of a group walks the whole source tree.
int group_warps(int n_sink, int most) {
  const int groups = (n_sink + 31) / 32, fill = 64 * sm_count();
  int w = 1;
  while (w < most && 2 * w * groups <= fill) w *= 2;
  return w;
}

// Shared memory of a block, for the warps that it has: blocks of two warps with room for eight
// took 9.9 ms for 100003 sinks instead of 7.3, since what they hold is taken from L1.
template <bool SUB>
size_t block_bytes(int w) {
  const size_t stacks = (w > 1 ? w : 4) * sizeof(CutStack<SUB>);
  const size_t sums = kSlots * 32 * sizeof(float2);
  return w > 1 && stacks < sums ? sums : stacks;
}

template <bool MERGE, bool MOM, bool BG, bool STOP, int NB, bool SUB, bool TD>
cudaError_t launch(const TreeView& T, const long long* sink_idx, int n_sink, const WalkParams& wp,
                   const SinkOut& out, unsigned long long* stats, int* status, cudaStream_t s) {
  const int w = group_warps(n_sink, most_warps(SUB));
  const int grid = w > 1 ? (n_sink + 31) / 32 : (n_sink + 127) / 128;
  const int threads = w > 1 ? 32 * w : 128;
  auto go = [&](auto kernel, unsigned long long* st) {
    kernel<<<grid, threads, block_bytes<SUB>(w), s>>>(T, sink_idx, n_sink, wp, out, st, status);
  };
  if (!MOM && (out.counters || stats)) {
    if (w > 1) go(cut_walk_kernel<true, MERGE, MOM, BG, STOP, NB, SUB, !MOM, TD>, stats);
    else go(cut_walk_kernel<false, MERGE, MOM, BG, STOP, NB, SUB, !MOM, TD>, stats);
  } else {  // no counters asked for: the walk keeps none
    if (w > 1) go(cut_walk_kernel<true, MERGE, MOM, BG, STOP, NB, SUB, false, TD>, nullptr);
    else go(cut_walk_kernel<false, MERGE, MOM, BG, STOP, NB, SUB, false, TD>, nullptr);
  }
  note_launch();
  return cudaGetLastError();
}

template <int BS, bool MERGE, bool CNT>
void launch_batched(const TreeView* views, float* const* flux_out, const int2* items, int n_items,
                    int item, unsigned* counter, const WalkParams& wp, unsigned long long* stats,
                    int* status, int n_sm, cudaStream_t s) {
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cut_walk_batched_kernel<BS, MERGE, CNT>,
                                                BS, 0);
  cut_walk_batched_kernel<BS, MERGE, CNT><<<n_sm * per_sm, BS, 0, s>>>(
      views, flux_out, items, n_items, item, counter, wp, stats, status);
}

template <int BS>
void launch_batched(const TreeView* views, float* const* flux_out, const int2* items, int n_items,
                    int item, unsigned* counter, const WalkParams& wp, unsigned long long* stats,
                    int* status, int n_sm, cudaStream_t s) {
  auto go = [&](auto f) {
    f(views, flux_out, items, n_items, item, counter, wp, stats, status, n_sm, s);
  };
  if (wp.variant == 3)
    stats ? go(launch_batched<BS, true, true>) : go(launch_batched<BS, true, false>);
  else
    stats ? go(launch_batched<BS, false, true>) : go(launch_batched<BS, false, false>);
}

}  // namespace

cudaError_t launch_cut_batched(const TreeView* views, float* const* flux_out, const int2* items,
                               int n_items, int item, unsigned* counter, const WalkParams& wp,
                               unsigned long long* stats, int* status, int block_size, int n_sm,
                               cudaStream_t s) {
  if (block_size <= 64)
    launch_batched<64>(views, flux_out, items, n_items, item, counter, wp, stats, status, n_sm, s);
  else if (block_size <= 128)
    launch_batched<128>(views, flux_out, items, n_items, item, counter, wp, stats, status, n_sm,
                        s);
  else
    launch_batched<256>(views, flux_out, items, n_items, item, counter, wp, stats, status, n_sm,
                        s);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_cut_adjoint(const TreeView& T, const long long* sink_idx, int n_sink,
                               const WalkParams& wp, const AdjointArgs& J, int* status,
                               cudaStream_t s) {
  const int w = group_warps(n_sink, kSlots);
  const int grid = w > 1 ? (n_sink + 31) / 32 : (n_sink + 127) / 128;
  const int threads = w > 1 ? 32 * w : 128;
  auto go = [&](auto kernel) {
    kernel<<<grid, threads, block_bytes<false>(w), s>>>(T, sink_idx, n_sink, wp, status, J);
  };
  if (wp.variant == 3) {
    if (w > 1) go(cut_adjoint_kernel<true, true>);
    else go(cut_adjoint_kernel<false, true>);
  } else {
    if (w > 1) go(cut_adjoint_kernel<true, false>);
    else go(cut_adjoint_kernel<false, false>);
  }
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_walk_moments(const TreeView& T, const long long* sink_idx, int n_sink,
                                const WalkParams& wp, float* flux_out, float* fvec, float* press,
                                int* status, cudaStream_t s) {
  if (n_sink <= 0) return cudaSuccess;
  return launch<true, true, false, false, 1, false, false>(
      T, sink_idx, n_sink, wp, SinkOut{flux_out, nullptr, fvec, press, n_sink}, nullptr, status, s);
}

// Several bands: 2 band slots for 2 bands, 4 slots for 3 or 4 (an unused slot holds
// zeros and is not written). One band is the plain walk.
cudaError_t launch_walk_bands(const TreeView& T, const long long* sink_idx, int n_sink,
                              const WalkParams& wp, float* flux_out, int* counters,
                              unsigned long long* stats, int* status, cudaStream_t s) {
  if (n_sink <= 0) return cudaSuccess;
  const SinkOut o{flux_out, counters, nullptr, nullptr, n_sink};
  if (T.n_bands <= 2)
    return launch<true, false, false, false, 2, false, false>(T, sink_idx, n_sink, wp, o, stats,
                                                              status, s);
  return launch<true, false, false, false, 4, false, false>(T, sink_idx, n_sink, wp, o, stats,
                                                            status, s);
}

cudaError_t launch_cut_walk(const TreeView& T, const long long* sink_idx, int n_sink,
                            const WalkParams& wp, float* flux_out, int* counters,
                            unsigned long long* stats, int* status, cudaStream_t s) {
  const SinkOut o{flux_out, counters, nullptr, nullptr, n_sink};
  const bool bg = wp.bg_radius > 0.0f, stop = wp.tau_stop < INFINITY;
  if (wp.sub_bucket)
    return launch<true, false, false, false, 1, true, false>(T, sink_idx, n_sink, wp, o, stats,
                                                             status, s);
  if (bg && stop)
    return launch<true, false, true, true, 1, false, false>(T, sink_idx, n_sink, wp, o, stats,
                                                            status, s);
  if (bg)
    return launch<true, false, true, false, 1, false, false>(T, sink_idx, n_sink, wp, o, stats,
                                                             status, s);
  if (stop)
    return launch<true, false, false, true, 1, false, false>(T, sink_idx, n_sink, wp, o, stats,
                                                             status, s);
  if (wp.topdown)
    return launch<true, false, false, false, 1, false, true>(T, sink_idx, n_sink, wp, o, stats,
                                                             status, s);
  if (wp.variant == 3)
    return launch<true, false, false, false, 1, false, false>(T, sink_idx, n_sink, wp, o, stats,
                                                              status, s);
  return launch<false, false, false, false, 1, false, false>(T, sink_idx, n_sink, wp, o, stats,
                                                             status, s);
}

}  // namespace trevr
