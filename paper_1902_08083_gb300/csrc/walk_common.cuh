// What the walk translation units share: compensated sums, counters, output slots and the
// map from a call's sinks to sorted particles.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "trevr_internal.cuh"

namespace trevr {
namespace {

constexpr int kDepth = 64;  // > max cell depth (63): lists and stacks never overflow
constexpr float kFourPi = 12.566370614359172f;

// Neumaier-compensated fp32 sum.
struct CSum {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float x) {
    float t = __fadd_rn(s, x);
    if (fabsf(s) >= fabsf(x)) c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, t), x));
    else c = __fadd_rn(c, __fadd_rn(__fsub_rn(x, t), s));
    s = t;
  }
  __device__ __forceinline__ float get() const { return __fadd_rn(s, c); }
};

// Kahan-compensated fp32 running sum (branch-free), for the optical depth of one
// ray in the warp walks: c carries the low-order part that each addition loses,
// so the error of the sum stays within about 2 ulp of the total however many
// terms a refined ray has.
struct KSum {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float x) {
    const float y = __fsub_rn(x, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
  }
  __device__ __forceinline__ float get() const { return s; }
};

struct SinkCounters {
  int rays = 0, segs = 0, visit = 0, ref = 0, clip = 0, cut = 0, sub = 0;
};

// warp-reduce the counters and add them to the device totals (all lanes call it)
__device__ __forceinline__ void add_stats(const SinkCounters& c, unsigned long long* stats) {
  unsigned long long v[7] = {(unsigned long long)c.rays, (unsigned long long)c.segs,
                             (unsigned long long)c.visit, (unsigned long long)c.ref,
                             (unsigned long long)c.clip, (unsigned long long)c.cut,
                             (unsigned long long)c.sub};
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    unsigned long long x = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(&stats[q], x);
  }
}

// Where a finished sink's results go.
struct SinkOut {
  float* flux;    // flux per sink (caller order), or nullptr
  int* counters;  // 4 int per sink, or nullptr
  float* fvec;    // flux vector, 3 x n_sink (SoA), or nullptr
  float* press;   // second moment, 6 x n_sink (SoA: xx yy zz xy xz yz), or nullptr
  int n_out;      // n_sink (stride of the SoA blocks)
};

// Direction moments of the intensity at one sink: sum f n and sum f n n^T, n the
// unit vector from the pseudo-source to the sink (Eq. simpflux; Sec. 2.1).
struct Moments {
  CSum v[9];  // x y z | xx yy zz xy xz yz
};

// Sinks of a plain call: chunk position k is the k-th requested sink, or the one that
// `order` puts there.
template <bool ADJ>
struct PlainMap {
  const TreeView* T;
  const long long* sink_idx;
  const float* grad_flux;
  int* status;
  const unsigned* order;
  int n_sink;
  __device__ __forceinline__ bool operator()(int k, int& i, int& slot, float& g) const {
    if (sink_idx) {
      slot = order ? (int)order[k] : k;
      if ((unsigned)slot >= (unsigned)n_sink) {  // the order's sort gave up (status is set)
        slot = -1;
        return false;
      }
      const long long si = sink_idx[slot];
      if (si < 0 || si >= T->n_gas) {
        atomicOr(status, kStatusInvalid);
        return false;
      }
      i = T->rank[si];
    } else {
      i = k;
      slot = T->perm[k];
    }
    g = ADJ ? grad_flux[slot] : 0.0f;
    return !ADJ || g != 0.0f;  // the adjoint skips sinks with dLoss/dF = 0
  }
};

}  // namespace
}  // namespace trevr
