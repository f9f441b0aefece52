// Tree topology from sorted keys (topology.cu): its arrays and its launch.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "trevr_internal.cuh"

namespace trevr {

constexpr int kNoCut = -2, kRootCut = -1;

struct TopoArrays {
  int n;
  int bucket;
  const unsigned long long* key;
  const int* status;
  // per particle i, the cut between i - 1 and i
  int* up;               // 2 * parent cut + side (1 = upper child), kRootCut, or kNoCut
  int2* range;           // particles of the cut cell
  unsigned char* bit;    // key bit of the cut
  unsigned char* depth;  // of the cut cell
  int* place;            // breadth-first place of a kept cut
  int* list;             // the kept cut at a place
  unsigned* counts;      // topo_count_words(n): kept cuts by (depth, tile)
  // the tree
  int* nfirst;
  int* ncount;
  int4* nglo;  // w = split axis (-1 leaf)
  int4* nghi;
  int4* nT;    // x child, y parent, z src_first, w src_count
  int* ndepth;
  unsigned long long* nD;  // path from the root (TreeView::nD)
  int* leaf_of;
  int* levels;  // [kMaxLevels][2]
};

size_t topo_count_words(int n);
// The kept cuts, their places and the levels' cell ranges (an empty root level if the sort gave
// up). scan_scratch holds scan_scratch_words(topo_count_words(n)) words.
void launch_cuts(const TopoArrays& A, unsigned* scan_scratch, cudaStream_t s);
// The cells: the tree's arrays, which have to hold as many as the levels end at.
void launch_cells(const TopoArrays& A, cudaStream_t s);

}  // namespace trevr
