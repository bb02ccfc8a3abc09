// Nested dissection of the spatial problems (K + lam_q M) x = b (nd.h).
//
// Factorisation, boxes of one depth and all modes together, deepest first.
// The front of a box is the symmetric matrix on its nodes S (own) and B
// (boundary): the entries of K + lam M that involve an own node, plus the
// Schur complements of its two children.  Sweeping the own nodes out (blocks
// of kPb pivots, Gauss-Jordan on the whole front) turns it into
//   [ F_SS^{-1}                 . ]
//   [ -F_BS F_SS^{-1}   F_BB - F_BS F_SS^{-1} F_SB ],
// the last block being the child contribution of the box above.  With
// H = [F_SS^{-1} | -F_SS^{-1} F_SB] and G = F_BS F_SS^{-1} a solve is
//   up:   y_S = b_S - w_S,  u_B = w_B + G y_S      (w: the children's u)
//   down: x_S = H [y_S; x_B],
// one launch per depth and direction.  No pivoting: for Im lam != 0 the matrix
// -i (K + lam M) has the positive definite Hermitian part Im(lam) M, for real
// lam > 0 K + lam M is positive definite, and both properties pass to Schur
// complements, so every pivot block is non-singular.
//
// Why not a banded factor: a banded substitution is a chain of one dependent
// step per block of rows (508 exchanges between SMs for the 127^2 grid), while
// the depths here number about 2 log2 n in 2D, every depth is a batch of
// independent dense products that fills the device, and the factor is smaller
// (127^2: 1.2 M against 4.2 M elements per mode; 31^3: 18 M against 59 M).
// Whole component solves, banded (blocked over thread-block clusters up to
// band 128, row by row above) -> nested dissection, on GB300: 127^2 grid FP64,
// 5 modes 2.10 -> 0.43 ms; 15^3 FP64, 5 modes 13.6 -> 0.28 ms; 31^3 FP32, 17
// modes 114 -> 3.9 ms.  Set-up of the layered 2D medium n = 12 FP64 0.32 ->
// 0.15 s and of the 3D random medium n = 10 5.7 -> 0.8 s.  What bounds a solve: FP64, the
// FP64 pipe on grids with many modes, else launch and gather latency per
// depth; FP32, the latter, and HBM for 31^3.
#include <algorithm>
#include <cmath>

#include "nd.h"

namespace st {

namespace {

constexpr int kPb = 32;      // pivots per block of the factorisation
constexpr int kThreads = 256;

inline int64_t cdiv64(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Lower corner of box v.
__device__ __forceinline__ void box_lo(const NdLevel& L, int v, int lo[3]) {
  int p[3] = {0, 0, 0};
  for (int k = 0; k < L.depth; ++k) {
    const int bit = (v >> (L.depth - 1 - k)) & 1;
#pragma unroll
    for (int m = 0; m < 3; ++m)
      if (L.dims[k] == m) p[m] = 2 * p[m] + bit;
  }
#pragma unroll
  for (int m = 0; m < 3; ++m) lo[m] = p[m] * (L.sz[m] + 1);
}

// Grid points around and inside a box, clipped to the grid.
struct Hull {
  int lo[3], w[3];
};
__device__ __forceinline__ Hull box_hull(const NdLevel& L, const int lo[3]) {
  Hull e;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int a = k < L.d ? max(lo[k] - 1, 0) : 0;
    const int b = k < L.d ? min(lo[k] + L.sz[k] + 1, L.n) : 1;
    e.lo[k] = a;
    e.w[k] = b - a;
  }
  return e;
}

// Position of the grid point P in the boundary list of the box at lo (the
// hull's points in lexicographic order without the box's own), or -1.
__device__ __forceinline__ int ring_pos(const NdLevel& L, const int lo[3], const Hull& e, const int P[3]) {
  bool in = true, inside = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    in = in && P[k] >= e.lo[k] && P[k] < e.lo[k] + e.w[k];
    const int sz = k < L.d ? L.sz[k] : 1, l = k < L.d ? lo[k] : 0;
    inside = inside && P[k] >= l && P[k] < l + sz;
  }
  if (!in || inside) return -1;
  const int lex = ((P[2] - e.lo[2]) * e.w[1] + (P[1] - e.lo[1])) * e.w[0] + (P[0] - e.lo[0]);
  // points of the box that precede P
  const int s0 = L.sz[0], s1 = L.d > 1 ? L.sz[1] : 1, s2 = L.d > 2 ? L.sz[2] : 1;
  const int l1 = L.d > 1 ? lo[1] : 0, l2 = L.d > 2 ? lo[2] : 0;
  const int z = min(max(P[2] - l2, 0), s2);
  int before = z * s0 * s1;
  if (P[2] >= l2 && P[2] < l2 + s2) {
    const int y = min(max(P[1] - l1, 0), s1);
    before += y * s0;
    if (P[1] >= l1 && P[1] < l1 + s1) before += min(max(P[0] - lo[0], 0), s0);
  }
  return lex - before;
}

__device__ __forceinline__ int point_index(const NdLevel& L, const int P[3]) {
  return (P[2] * (L.d > 1 ? L.n : 0) + P[1]) * (L.d > 1 ? L.n : 0) + P[0];
}

// Front indices of every box of a depth: own nodes, then the boundary.
__global__ void k_nd_index(NdLevel L, int per, int* __restrict__ idx, int* __restrict__ nb) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)L.nodes * per) return;
  const int v = (int)(t / per), e = (int)(t - (int64_t)v * per);
  int lo[3];
  box_lo(L, v, lo);
  int* row = idx + L.idx + (int64_t)v * L.ld;
  if (e < L.s) {  // own node e: the box (leaf) or its middle plane, first direction fastest
    int w[3], P[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) w[k] = (k >= L.d || k == L.split) ? 1 : L.sz[k];
    P[0] = e % w[0];
    P[1] = (e / w[0]) % w[1];
    P[2] = e / (w[0] * w[1]);
#pragma unroll
    for (int k = 0; k < 3; ++k) P[k] = k < L.d ? lo[k] + (k == L.split ? (L.sz[k] - 1) / 2 : P[k]) : 0;
    row[e] = point_index(L, P);
    return;
  }
  const int r = e - L.s;  // hull point
  const Hull hu = box_hull(L, lo);
  const int vol = hu.w[0] * hu.w[1] * hu.w[2];
  const int own = L.sz[0] * (L.d > 1 ? L.sz[1] : 1) * (L.d > 2 ? L.sz[2] : 1);
  if (r == 0) nb[L.nb + v] = vol - own;
  if (r >= vol) return;
  const int P[3] = {hu.lo[0] + r % hu.w[0], hu.lo[1] + (r / hu.w[0]) % hu.w[1], hu.lo[2] + r / (hu.w[0] * hu.w[1])};
  const int pos = ring_pos(L, lo, hu, P);
  if (pos >= 0) row[L.s + pos] = point_index(L, P);
}

// Place of every front position in the boundary of each child (-1: not there).
__global__ void k_nd_map(NdLevel L, NdLevel C, const int* __restrict__ idx, int* __restrict__ map, int64_t nidx) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)L.nodes * L.ld) return;
  const int v = (int)(t / L.ld);
  const int g = idx[L.idx + t];
  int P[3] = {0, 0, 0};
  if (g >= 0) {
    P[0] = g % L.n;
    if (L.d > 1) P[1] = (g / L.n) % L.n;
    if (L.d > 2) P[2] = g / (L.n * L.n);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    int lo[3];
    box_lo(C, 2 * v + c, lo);
    map[c * nidx + L.idx + t] = g >= 0 ? ring_pos(C, lo, box_hull(C, lo), P) : -1;
  }
}

// ---------------------------------------------------------- factorisation
// Lower triangle of every front of a depth: original entries with an own node
// and the children's Schur complements.
template <int D, typename R>
__global__ void __launch_bounds__(kThreads)
    k_nd_assemble(NdLevel L, NdLevel C, bool leaf, const int* __restrict__ idx, const int* __restrict__ map,
                  int64_t nidx, StencilCoef sc, const double* __restrict__ c2, const cx<double>* __restrict__ lam,
                  const cx<R>* __restrict__ Fc, cx<R>* __restrict__ F) {
  const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int64_t fs = (int64_t)L.ld * L.ld;
  if (t >= L.nodes * fs) return;
  const int v = (int)(t / fs);
  const int e = (int)(t - (int64_t)v * fs);
  const int i = e / L.ld, j = e - i * L.ld;
  if (j > i) return;
  const int q = blockIdx.y;
  const int64_t row = L.idx + (int64_t)v * L.ld;
  const int a = idx[row + i], b = idx[row + j];
  cx<R> val = mk<R>(0, 0);
  if (a >= 0 && b >= 0) {
    if (j < L.s) {
      int A[3] = {a % L.n, 0, 0}, B[3] = {b % L.n, 0, 0};
      if (D > 1) {
        A[1] = (a / L.n) % L.n;
        B[1] = (b / L.n) % L.n;
      }
      if (D > 2) {
        A[2] = a / (L.n * L.n);
        B[2] = b / (L.n * L.n);
      }
      bool near = true;
      int st = 0, w3 = 1;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const int dl = B[k] - A[k];
        near = near && dl >= -1 && dl <= 1;
        st += (dl + 1) * w3;
        w3 *= 3;
      }
      if (near) {
        // c^2 over the cells that hold both nodes: cell A + e, e = 1 for a
        // neighbour above, 0 for one below, both otherwise
        double S = 0.0;
#pragma unroll
        for (int c = 0; c < (1 << D); ++c) {
          bool ok = true;
          int64_t cell = 0, str = 1;
#pragma unroll
          for (int k = 0; k < D; ++k) {
            const int ek = (c >> k) & 1, dl = B[k] - A[k];
            ok = ok && (dl == 0 || (dl == 1 && ek == 1) || (dl == -1 && ek == 0));
            cell += (int64_t)(A[k] + ek) * str;
            str *= L.n + 1;
          }
          if (ok) S += c2[cell];
        }
        const cx<double> l = lam[q];
        val = mk<R>((R)(S * sc.ke[st] + l.re * sc.mtot[st]), (R)(l.im * sc.mtot[st]));
      }
    }
    if (!leaf) {
      const int64_t cs = (int64_t)C.ld * C.ld;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int p = map[c * nidx + row + i], r = map[c * nidx + row + j];
        if (p < 0 || r < 0) continue;
        const cx<R>* M = Fc + ((int64_t)q * C.nodes + 2 * v + c) * cs;
        const int hi = C.s + max(p, r), lo = C.s + min(p, r);
        val = val + M[(int64_t)hi * C.ld + lo];
      }
    }
  }
  F[((int64_t)q * L.nodes + v) * fs + e] = val;
}

// Panels of one pivot block [k0, k0 + pb) of every front: C = the front's
// columns of the block (rows below from the lower triangle, rows above from
// its transpose; swept rows with the opposite sign, as Gauss-Jordan leaves
// them), T = C P with P the inverse of the pivot block.
constexpr int kPanelRows = 32;
template <typename R>
__global__ void __launch_bounds__(kThreads)
    k_nd_panel(NdLevel L, int k0, int pb, int chunks, const cx<R>* __restrict__ F, cx<R>* __restrict__ Cp,
               cx<R>* __restrict__ Tp, int* __restrict__ err) {
  __shared__ cx<R> P[kPb][kPb + 1];
  __shared__ cx<R> Cs[kPanelRows][kPb + 1];
  __shared__ cx<R> col[kPb];
  const int v = blockIdx.x / chunks, ch = blockIdx.x - v * chunks, q = blockIdx.y, tid = threadIdx.x;
  const int64_t f = (int64_t)q * L.nodes + v;
  const cx<R>* A = F + f * L.ld * L.ld;
  for (int e = tid; e < pb * pb; e += kThreads) {
    const int i = e / pb, j = e - i * pb;
    P[i][j] = A[(int64_t)(k0 + max(i, j)) * L.ld + k0 + min(i, j)];
  }
  const int r0 = ch * kPanelRows;
  for (int e = tid; e < kPanelRows * pb; e += kThreads) {
    int i, j;
    cx<R> c = mk<R>(0, 0);
    if (r0 >= k0) {  // consecutive threads over the columns of a row
      i = e / pb;
      j = e - i * pb;
    } else {  // over the rows of a column (read from the transpose)
      j = e / kPanelRows;
      i = e - j * kPanelRows;
    }
    const int r = r0 + i;
    if (r < L.ld) {
      if (r >= k0 + pb) c = A[(int64_t)r * L.ld + k0 + j];
      else if (r < k0) {
        c = A[(int64_t)(k0 + j) * L.ld + r];
        c = mk<R>(-c.re, -c.im);
      }
    }
    Cs[i][j] = c;
  }
  __syncthreads();
  // P := P^{-1}, unblocked Gauss-Jordan
  for (int k = 0; k < pb; ++k) {
    if (tid < pb) col[tid] = P[tid][k];
    __syncthreads();
    const cx<R> piv = col[k];
    const R den = piv.re * piv.re + piv.im * piv.im;
    if (!(den > R(0))) {
      if (tid == 0) atomicExch(err, 1);
    }
    const cx<R> inv = cdiv(mk<R>(R(1), R(0)), piv);
    if (tid < pb && tid != k) P[k][tid] = inv * P[k][tid];
    __syncthreads();
    for (int e = tid; e < pb * pb; e += kThreads) {
      const int i = e / pb, j = e - i * pb;
      if (i == k) continue;
      const cx<R> ci = col[i];
      if (j == k) {
        const cx<R> z = ci * inv;
        P[i][k] = mk<R>(-z.re, -z.im);
      } else {
        P[i][j] = fma_c(mk<R>(-ci.re, -ci.im), P[k][j], P[i][j]);
      }
    }
    __syncthreads();
    if (tid == 0) P[k][k] = inv;
    __syncthreads();
  }
  const int64_t pbase = f * L.ld * kPb;
  for (int e = tid; e < kPanelRows * pb; e += kThreads) {
    const int i = e / pb, j = e - i * pb, r = r0 + i;
    if (r >= L.ld) continue;
    cx<R> t;
    if (r >= k0 && r < k0 + pb) {
      t = P[r - k0][j];  // the pivot rows carry the inverse
    } else {
      t = mk<R>(0, 0);
      for (int k = 0; k < pb; ++k) t = fma_c(Cs[i][k], P[k][j], t);
    }
    Cp[pbase + (int64_t)r * kPb + j] = Cs[i][j];
    Tp[pbase + (int64_t)r * kPb + j] = t;
  }
}

// Gauss-Jordan update of the lower triangle with one pivot block:
//   A_ij -= s_j C_i . T_j  (s_j = -1 for a swept column j < k0, else 1),
//   A_ik = -T_i (pivot columns), A_kj = -T_j (pivot rows, swept columns),
//   A_kk = P.
// TS x TS tile per CTA of 256 threads, (TS/16)^2 entries per thread, both
// panels of the tile staged in shared memory pivot-major.
template <typename R, int TS>
__global__ void __launch_bounds__(kThreads)
    k_nd_update(NdLevel L, int k0, int pb, int tiles, cx<R>* __restrict__ F, const cx<R>* __restrict__ Cp,
                const cx<R>* __restrict__ Tp) {
  constexpr int NE = TS / 16, LDT = TS + 1;
  extern __shared__ __align__(16) unsigned char smem_nd[];
  cx<R>* Cs = reinterpret_cast<cx<R>*>(smem_nd);  // kPb x LDT
  cx<R>* Ts = Cs + kPb * LDT;
  const int ntri = tiles * (tiles + 1) / 2;
  const int v = blockIdx.x / ntri, e = blockIdx.x - v * ntri, q = blockIdx.y, tid = threadIdx.x;
  // tile pair (ti, tj), tj <= ti, from the triangular number
  int ti = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while ((ti + 1) * (ti + 2) / 2 <= e) ++ti;
  while (ti * (ti + 1) / 2 > e) --ti;
  const int tj = e - ti * (ti + 1) / 2;
  const int i0 = ti * TS, j0 = tj * TS;
  const int64_t f = (int64_t)q * L.nodes + v;
  cx<R>* A = F + f * L.ld * L.ld;
  const cx<R>* Cq = Cp + f * L.ld * kPb;
  const cx<R>* Tq = Tp + f * L.ld * kPb;
  for (int t = tid; t < TS * kPb; t += kThreads) {
    const int r = t / kPb, k = t - r * kPb;
    const bool kk = k < pb;
    Cs[k * LDT + r] = (kk && i0 + r < L.ld) ? Cq[(int64_t)(i0 + r) * kPb + k] : mk<R>(0, 0);
    Ts[k * LDT + r] = (kk && j0 + r < L.ld) ? Tq[(int64_t)(j0 + r) * kPb + k] : mk<R>(0, 0);
  }
  __syncthreads();
  const int tx = tid & 15, ty = tid >> 4;
  cx<R> acc[NE][NE];
#pragma unroll
  for (int a = 0; a < NE; ++a)
#pragma unroll
    for (int b = 0; b < NE; ++b) acc[a][b] = mk<R>(0, 0);
  for (int k = 0; k < pb; ++k) {
    cx<R> cc[NE], tt[NE];
#pragma unroll
    for (int a = 0; a < NE; ++a) cc[a] = Cs[k * LDT + ty + 16 * a];
#pragma unroll
    for (int b = 0; b < NE; ++b) tt[b] = Ts[k * LDT + tx + 16 * b];
#pragma unroll
    for (int a = 0; a < NE; ++a)
#pragma unroll
      for (int b = 0; b < NE; ++b) acc[a][b] = fma_c(cc[a], tt[b], acc[a][b]);
  }
#pragma unroll
  for (int a = 0; a < NE; ++a) {
    const int i = i0 + ty + 16 * a;
    if (i >= L.ld) continue;
#pragma unroll
    for (int b = 0; b < NE; ++b) {
      const int j = j0 + tx + 16 * b;
      if (j > i || j >= L.ld) continue;
      const bool pi = i >= k0 && i < k0 + pb, pj = j >= k0 && j < k0 + pb;
      cx<R>* d = A + (int64_t)i * L.ld + j;
      if (pj) {
        const cx<R> t = Tq[(int64_t)i * kPb + (j - k0)];
        *d = pi ? t : mk<R>(-t.re, -t.im);
      } else if (pi) {
        const cx<R> t = Tq[(int64_t)j * kPb + (i - k0)];
        *d = mk<R>(-t.re, -t.im);
      } else {
        const cx<R> o = *d;
        *d = j < k0 ? mk<R>(o.re + acc[a][b].re, o.im + acc[a][b].im)
                    : mk<R>(o.re - acc[a][b].re, o.im - acc[a][b].im);
      }
    }
  }
}

// Solve matrices of a depth from its swept fronts: G (own node k major,
// boundary fastest) and H (inputs [S; B] major, own node fastest).
template <typename R>
__global__ void __launch_bounds__(kThreads)
    k_nd_pack(NdLevel L, const cx<R>* __restrict__ F, cx<R>* __restrict__ mats, int64_t mstride) {
  const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int64_t per = (int64_t)L.ld * L.s;
  if (t >= L.nodes * per) return;
  const int v = (int)(t / per);
  const int e = (int)(t - (int64_t)v * per);
  const int k = e / L.s, i = e - k * L.s;  // input k, own node i
  const int q = blockIdx.y;
  const cx<R>* A = F + ((int64_t)q * L.nodes + v) * L.ld * L.ld;
  cx<R>* M = mats + (int64_t)q * mstride;
  const cx<R> x = A[(int64_t)max(k, i) * L.ld + min(k, i)];
  M[L.h + (int64_t)v * per + e] = x;  // F_SS^{-1}, then -F_BS F_SS^{-1} = (-F_SS^{-1} F_SB)^T
  if (k >= L.s) M[L.g + (int64_t)v * L.s * L.bmax + (int64_t)i * L.bmax + (k - L.s)] = mk<R>(-x.re, -x.im);
}

// ------------------------------------------------------------------ solve
// One depth of the upward (UP) or downward pass.  A task is 32 output rows of
// one front and mode, done by g warps: each takes every g-th input, a lane per
// row, so the matrix is read once, coalesced over the rows; the warps' sums
// meet in shared memory in a fixed order.  The inputs (own right-hand side
// minus the children's updates, and on the way down the boundary's solution)
// are gathered into shared memory by every task of the front.  AHEAD: launched
// with launch_overlapped, the first matrix entries are read while the depth
// before ends: a depth waits on dependent loads, and these leave the chain.  FP32
// components alone, three sweeps: 63^2 3 modes 256 -> 203 us, 31^2 5 modes
// 177 -> 149 us, 127^2 17 modes 1.25 -> 1.06 ms; FP64 (bound by its instructions)
// gained nothing.
template <typename R, bool UP, bool AHEAD>
__global__ void __launch_bounds__(512)
    k_nd_level(NdLevel L, int leaf, int64_t cu, int cbmax, int g, int chunks, int kmax, const int* __restrict__ idx,
               const int* __restrict__ map, int64_t nidx, const int* __restrict__ nbs,
               const cx<R>* __restrict__ mats, int64_t mstride, const cx<R>* b, cx<R>* x, cx<R>* u, int64_t ustride,
               const CocgScal* scal, int64_t vstride) {
  extern __shared__ __align__(16) unsigned char smem_nd[];
  const int q = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tp = (blockDim.x >> 5) / g;  // tasks per CTA
  const int tk = warp / g, wg = warp - tk * g;
  cx<R>* in = reinterpret_cast<cx<R>*>(smem_nd) + (size_t)tk * kmax;
  cx<R>* red = reinterpret_cast<cx<R>*>(smem_nd) + (size_t)tp * kmax + (size_t)warp * 32;
  const int64_t task = (int64_t)blockIdx.x * tp + tk;
  const bool live = task < (int64_t)L.nodes * chunks;
  const int v = live ? (int)(task / chunks) : 0;
  const int r = live ? (int)(task - (int64_t)v * chunks) * 32 + lane : 0;
  const int64_t row = L.idx + (int64_t)v * L.ld;
  const int nb = live ? nbs[L.nb + v] : 0;
  const cx<R>* bq = b + (int64_t)q * vstride;
  cx<R>* xq = x + (int64_t)q * vstride;
  cx<R>* uq = u + (int64_t)q * ustride;
  const int64_t c0 = cu + (int64_t)(2 * v) * cbmax, c1 = c0 + cbmax;  // the children's updates
  const int K = !live ? 0 : (UP ? L.s : L.s + nb);
  // this lane's row of the matrix, its first entries read while the kernel before ends
  const int rows = UP ? nb : L.s, ldm = UP ? L.bmax : L.s;
  const cx<R>* M = mats + (int64_t)q * mstride +
                   (UP ? L.g + (int64_t)v * L.s * L.bmax : L.h + (int64_t)v * L.ld * L.s) + r;
  const bool out = live && r < rows;
  cx<R> m[8];
  if constexpr (AHEAD) {
    if (out && wg + 7 * g < K) {
#pragma unroll
      for (int t = 0; t < 8; ++t) m[t] = M[(int64_t)(wg + t * g) * ldm];
    }
    grid_start();
  }
  if (scal != nullptr && !scal[q].active) return;
  for (int k = wg * 32 + lane; k < K; k += 32 * g) {
    cx<R> val;
    if (k < L.s) {
      val = bq[idx[row + k]];
      if (!leaf) {
        const int p0 = map[row + k], p1 = map[nidx + row + k];
        if (p0 >= 0) val = val - uq[c0 + p0];
        if (p1 >= 0) val = val - uq[c1 + p1];
      }
    } else {
      val = xq[idx[row + k]];
    }
    in[k] = val;
  }
  __syncthreads();
  cx<R> acc = mk<R>(0, 0);
  if (out) {
    cx<R> a2 = mk<R>(0, 0);
    int k = wg;
    for (; k + 7 * g < K; k += 8 * g) {
      if (!AHEAD || k != wg) {
#pragma unroll
        for (int t = 0; t < 8; ++t) m[t] = M[(int64_t)(k + t * g) * ldm];
      }
#pragma unroll
      for (int t = 0; t < 8; t += 2) {
        acc = fma_c(m[t], in[k + t * g], acc);
        a2 = fma_c(m[t + 1], in[k + (t + 1) * g], a2);
      }
    }
    // fewer than eight left: in FP32 their loads together as well (3D n = 10 62.5 ->
    // 59.0 ms, its component (6,4) 29.7 -> 26.1 ms); one by one in FP64, where the
    // extra instructions cost more (255^2, 3 modes 0.60 -> 0.63 ms)
    if constexpr (sizeof(R) == 4) {
      if (k < K) {
#pragma unroll
        for (int t = 0; t < 7; ++t)
          if (k + t * g < K) m[t] = M[(int64_t)(k + t * g) * ldm];
#pragma unroll
        for (int t = 0; t < 7; ++t)
          if (k + t * g < K) acc = fma_c(m[t], in[k + t * g], acc);
      }
    } else {
      for (; k < K; k += g) acc = fma_c(M[(int64_t)k * ldm], in[k], acc);
    }
    acc = acc + a2;
  }
  if (g > 1) {
    red[lane] = acc;
    __syncthreads();
    if (wg != 0) return;
    for (int w = 1; w < g; ++w) acc = acc + red[w * 32 + lane];
  }
  if (!out || wg != 0) return;
  if (UP) {
    if (!leaf) {
      const int p0 = map[row + L.s + r], p1 = map[nidx + row + L.s + r];
      if (p0 >= 0) acc = acc + uq[c0 + p0];
      if (p1 >= 0) acc = acc + uq[c1 + p1];
    }
    uq[L.u + (int64_t)v * L.bmax + r] = acc;
  } else {
    xq[idx[row + r]] = acc;
  }
}

template <typename R, bool UP>
void nd_level(const NdPlan& p, int t, const cx<R>* mats, const cx<R>* b, cx<R>* x, cx<R>* u, const CocgScal* scal,
              int nmodes, int64_t vstride, cudaStream_t s) {
  const NdLevel& L = p.lv[t];
  const bool leaf = t + 1 == (int)p.lv.size();
  const int rows = UP ? L.bmax : L.s, kmax = UP ? L.s : L.ld;
  const int chunks = (rows + 31) / 32;
  const int g = kmax > 384 ? 16 : (kmax > 96 ? 8 : (kmax > 48 ? 4 : (kmax > 24 ? 2 : 1)));
  const int threads = g > 8 ? 32 * g : 256, tp = threads / 32 / g;
  const int64_t tasks = (int64_t)L.nodes * chunks;
  const size_t smem = ((size_t)tp * kmax + threads) * sizeof(cx<R>);
  const int64_t cu = leaf ? 0 : p.lv[t + 1].u;
  const int cb = leaf ? 0 : p.lv[t + 1].bmax;
  const dim3 grid((unsigned)cdiv64(tasks, tp), nmodes);
  // FP32, at depths of at most one CTA of 256 threads an SM: 2D n = 8 (nine
  // components) 478 -> 397 us, and with the coarse solves of multigrid an ensemble
  // 12.9 -> 12.4 ms.  At every depth the early CTAs take room from other components:
  // the ensemble 13.3 ms, 2D n = 12 17.8 -> 18.2 ms; at up to two CTAs an SM the
  // ensemble 13.0 ms.
  const bool ahead = sizeof(R) == 4 && (int64_t)grid.x * grid.y * threads <= 152 * 256;
  auto kern = ahead ? k_nd_level<R, UP, sizeof(R) == 4> : k_nd_level<R, UP, false>;
  if (smem > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int lf = leaf ? 1 : 0;
  if (ahead)
    launch_overlapped(kern, grid, threads, smem, s, L, lf, cu, cb, g, chunks, kmax, p.idx, p.map, p.nidx, p.nb, mats,
                      p.mstride, b, x, u, p.ustride, scal, vstride);
  else
    kern<<<grid, threads, smem, s>>>(L, lf, cu, cb, g, chunks, kmax, p.idx, p.map, p.nidx, p.nb, mats, p.mstride, b, x,
                                     u, p.ustride, scal, vstride);
}

}  // namespace

NdPlan nd_plan(const Geo& g, int leaf) {
  NdPlan p;
  p.d = g.d;
  p.n = g.n;
  p.nrow = g.nnodes;
  NdLevel L{};
  L.d = g.d;
  L.n = g.n;
  for (int k = 0; k < 3; ++k) {
    L.sz[k] = k < g.d ? g.n : 1;
    L.pieces[k] = 1;
  }
  int64_t prev = 0, prev_pan = 0;
  for (int t = 0;; ++t) {
    L.depth = t;
    L.nodes = 1 << t;
    int big = 0;
    for (int k = 1; k < g.d; ++k)
      if (L.sz[k] >= L.sz[big]) big = k;
    const bool lf = L.sz[big] <= leaf;
    L.split = lf ? -1 : big;
    int64_t vol = 1, hull = 1, sep = 1;
    for (int k = 0; k < g.d; ++k) {
      vol *= L.sz[k];
      hull *= L.sz[k] + std::min(2, L.pieces[k] - 1);
      if (k != big) sep *= L.sz[k];
    }
    L.s = (int)(lf ? vol : sep);
    L.bmax = (int)(hull - vol);
    L.ld = L.s + L.bmax;
    L.idx = p.nidx;
    L.nb = p.nnb;
    L.u = p.ustride;
    L.g = p.mstride;
    L.h = L.g + (int64_t)L.nodes * L.s * L.bmax;
    p.nidx += (int64_t)L.nodes * L.ld;
    p.nnb += L.nodes;
    p.ustride += (int64_t)L.nodes * L.bmax;
    p.mstride = L.h + (int64_t)L.nodes * L.ld * L.s;
    p.solve_flops += 8.0 * L.nodes * ((double)L.s * L.s + 2.0 * L.s * L.bmax);
    p.factor_flops += 4.0 * L.nodes * (double)L.s * L.ld * L.ld;
    // fronts of two consecutive depths, and the two panels of either
    const int64_t fr = (int64_t)L.nodes * L.ld * L.ld, pan = 2 * (int64_t)L.nodes * L.ld * kPb;
    p.work_elems = std::max(p.work_elems, fr + prev + std::max(pan, prev_pan));
    prev = fr;
    prev_pan = pan;
    p.lv.push_back(L);
    if (lf) break;
    L.dims[t] = (signed char)big;
    L.sz[big] = (L.sz[big] - 1) / 2;
    L.pieces[big] *= 2;
  }
  return p;
}

int nd_leaf(const Geo& g, int nmodes, size_t real_size) {
  // estimated solve time: ~4 us per launch, and the matrices at the HBM rate
  // or their multiply-adds at the FP64 rate, whichever is longer
  int best = 3;
  double tbest = 1e300;
  for (int leaf = 3; leaf <= 63; leaf = 2 * leaf + 1) {
    const NdPlan p = nd_plan(g, leaf);
    if (p.lv.back().s > 256 && leaf > 3) break;
    const double launches = 2.0 * (double)p.lv.size() - 1.0;
    const double mem = (double)nmodes * p.solve_flops / 8.0 * 2.0 * (double)real_size / 5.0e12;
    const double alu = (double)nmodes * p.solve_flops / (real_size == 8 ? 1.1e12 : 4.0e13);
    const double t = launches * 4e-6 + std::max(mem, alu);
    if (t < tbest) {
      tbest = t;
      best = leaf;
    }
    if (leaf >= g.n) break;
  }
  return best;
}

void launch_nd_index(const NdPlan& p, cudaStream_t s) {
  cudaMemsetAsync(p.idx, 0xff, (size_t)p.nidx * sizeof(int), s);
  for (const NdLevel& L : p.lv) {
    int64_t hull = 1;
    for (int k = 0; k < p.d; ++k) hull *= L.sz[k] + std::min(2, L.pieces[k] - 1);
    const int per = L.s + (int)hull;
    k_nd_index<<<(unsigned)cdiv64((int64_t)L.nodes * per, kThreads), kThreads, 0, s>>>(L, per, p.idx, p.nb);
  }
  for (size_t t = 0; t + 1 < p.lv.size(); ++t)
    k_nd_map<<<(unsigned)cdiv64((int64_t)p.lv[t].nodes * p.lv[t].ld, kThreads), kThreads, 0, s>>>(
        p.lv[t], p.lv[t + 1], p.idx, p.map, p.nidx);
  note_launches(2 * (int)p.lv.size() - 1);
}

template <typename R>
void launch_nd_factor(const NdPlan& p, const StencilCoef& sc, const double* c2, const cx<double>* lam,
                      int nmodes, cx<R>* mats, cx<R>* ws, int* err, cudaStream_t s) {
  const int T = (int)p.lv.size();
  // workspace: the fronts of a depth alternate between its two ends, the panels in between
  const int64_t total = (int64_t)nmodes * p.work_elems;
  cx<R>* Fc = nullptr;
  int launched = 0;
  constexpr size_t sm64 = 2 * (size_t)kPb * 65 * sizeof(cx<R>), sm32 = 2 * (size_t)kPb * 33 * sizeof(cx<R>);
  cudaFuncSetAttribute(k_nd_update<R, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm64);
  for (int t = T - 1; t >= 0; --t) {
    const NdLevel& L = p.lv[t];
    const NdLevel& C = t + 1 < T ? p.lv[t + 1] : L;
    const int64_t fr = (int64_t)nmodes * L.nodes * L.ld * L.ld, pan = (int64_t)nmodes * L.nodes * L.ld * kPb;
    const bool low = ((T - 1 - t) & 1) == 0;
    cx<R>* F = low ? ws : ws + total - fr;
    cx<R>* Cp = low ? ws + fr : F - 2 * pan;
    cx<R>* Tp = Cp + pan;
    const dim3 ga((unsigned)cdiv64((int64_t)L.nodes * L.ld * L.ld, kThreads), nmodes);
    const bool leaf = t + 1 == T;
    if (p.d == 1)
      k_nd_assemble<1, R><<<ga, kThreads, 0, s>>>(L, C, leaf, p.idx, p.map, p.nidx, sc, c2, lam, Fc, F);
    else if (p.d == 2)
      k_nd_assemble<2, R><<<ga, kThreads, 0, s>>>(L, C, leaf, p.idx, p.map, p.nidx, sc, c2, lam, Fc, F);
    else
      k_nd_assemble<3, R><<<ga, kThreads, 0, s>>>(L, C, leaf, p.idx, p.map, p.nidx, sc, c2, lam, Fc, F);
    const int chunks = (L.ld + kPanelRows - 1) / kPanelRows;
    for (int k0 = 0; k0 < L.s; k0 += kPb) {
      const int pb = std::min(kPb, L.s - k0);
      k_nd_panel<R><<<dim3((unsigned)(L.nodes * chunks), nmodes), kThreads, 0, s>>>(L, k0, pb, chunks, F, Cp, Tp, err);
      if (L.ld > 96) {
        const int tiles = (L.ld + 63) / 64;
        k_nd_update<R, 64><<<dim3((unsigned)((int64_t)L.nodes * tiles * (tiles + 1) / 2), nmodes), kThreads, sm64, s>>>(
            L, k0, pb, tiles, F, Cp, Tp);
      } else {
        const int tiles = (L.ld + 31) / 32;
        k_nd_update<R, 32><<<dim3((unsigned)((int64_t)L.nodes * tiles * (tiles + 1) / 2), nmodes), kThreads, sm32, s>>>(
            L, k0, pb, tiles, F, Cp, Tp);
      }
      launched += 2;
    }
    k_nd_pack<R><<<dim3((unsigned)cdiv64((int64_t)L.nodes * L.ld * L.s, kThreads), nmodes), kThreads, 0, s>>>(
        L, F, mats, p.mstride);
    launched += 2;
    Fc = F;
  }
  note_launches(launched);
}

template <typename R>
void launch_nd_solve(const NdPlan& p, const cx<R>* mats, const cx<R>* b, cx<R>* x, cx<R>* u, const CocgScal* scal,
                     int nmodes, int64_t vstride, cudaStream_t s) {
  const int T = (int)p.lv.size();
  for (int t = T - 1; t >= 1; --t) nd_level<R, true>(p, t, mats, b, x, u, scal, nmodes, vstride, s);
  for (int t = 0; t < T; ++t) nd_level<R, false>(p, t, mats, b, x, u, scal, nmodes, vstride, s);
  note_launches(2 * T - 1);
}

#define ST_ND_INST(R)                                                                                              \
  template void launch_nd_factor<R>(const NdPlan&, const StencilCoef&, const double*,                              \
                                    const cx<double>*, int, cx<R>*, cx<R>*, int*, cudaStream_t);                   \
  template void launch_nd_solve<R>(const NdPlan&, const cx<R>*, const cx<R>*, cx<R>*, cx<R>*, const CocgScal*, int, \
                                   int64_t, cudaStream_t);
ST_ND_INST(double)
ST_ND_INST(float)
#undef ST_ND_INST

}  // namespace st
