// Direct solves of the spatial problems (K + lam_q M) x = b by nested
// dissection of the grid, with the eliminated blocks kept as dense matrices
// (see nd.cu).
//
// The interior grid has n = 2^j - 1 nodes per direction.  A box of nodes is
// split by the middle plane of its longest direction (the separator) into two
// equal boxes, down to leaves of at most `leaf` nodes per direction; all boxes
// of one depth have the same size, so depth t holds 2^t boxes and box v of
// depth t has the children 2v and 2v+1.  The front of a box consists of its
// own nodes S (separator, or all nodes of a leaf) and its boundary B: the ring
// of grid nodes around the box, all of which belong to separators above it.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include <vector>

#include "common.cuh"
#include "kernels.h"

namespace st {

struct NdLevel {
  int d, n, depth;
  int sz[3];      // nodes of a box per direction
  int pieces[3];  // boxes per direction at this depth
  int split;      // direction of the separator, -1 for leaves
  signed char dims[48];  // directions of the splits above this depth
  int nodes;      // boxes: 2^depth
  int s;          // own nodes of a front
  int bmax;       // largest boundary of a front
  int ld;         // s + bmax
  int64_t idx;    // first front index (nodes x ld grid indices, own nodes first, -1 beyond the front)
  int64_t nb;     // first boundary count (one per box)
  int64_t u;      // first update value (nodes x bmax, per mode)
  int64_t g;      // forward matrices (nodes x s x bmax, per mode)
  int64_t h;      // backward matrices (nodes x ld x s, per mode)
};

struct NdPlan {
  int d = 0, n = 0;
  int64_t nrow = 0;
  std::vector<NdLevel> lv;   // depth 0 (the root) first
  int64_t nidx = 0, nnb = 0; // sizes of the index arrays
  int64_t ustride = 0;       // update values per mode
  int64_t mstride = 0;       // matrix elements per mode
  double solve_flops = 0.0;  // per mode
  double factor_flops = 0.0; // per mode
  int64_t work_elems = 0;    // elements of the factorisation workspace per mode
  int* idx = nullptr;        // device: front indices
  int* map = nullptr;        // device: per front position its place in each child's boundary (2 x nidx), or -1
  int* nb = nullptr;         // device: boundary counts
};

// Symbolic plan of the grid g with leaves of at most `leaf` nodes per direction
// (2^k - 1); device pointers are left null.
NdPlan nd_plan(const Geo& g, int leaf);
// Leaf size with the smallest estimated solve time for nmodes modes.
int nd_leaf(const Geo& g, int nmodes, size_t real_size);
// Fills the plan's device index arrays (allocated by the caller).
void launch_nd_index(const NdPlan& p, cudaStream_t s);
// Factorises K(c2) + lam_q M for every mode into mats (nmodes x mstride).  ws:
// nmodes x work_elems elements of scratch.  err[0] = 1 on a zero pivot.
template <typename R>
void launch_nd_factor(const NdPlan& p, const StencilCoef& sc, const double* c2, const cx<double>* lam,
                      int nmodes, cx<R>* mats, cx<R>* ws, int* err, cudaStream_t s);
// x_q = (K + lam_q M)^{-1} b_q for every active mode (vectors at q * vstride); u:
// nmodes x ustride scratch; x must not alias b.
template <typename R>
void launch_nd_solve(const NdPlan& p, const cx<R>* mats, const cx<R>* b, cx<R>* x, cx<R>* u, const CocgScal* scal,
                     int nmodes, int64_t vstride, cudaStream_t s);

}  // namespace st
