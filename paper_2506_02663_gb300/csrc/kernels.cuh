// sm_103a kernels of libamr4.  Templated on the value type T (double / float) and the
// dimension D (2 / 3).  Every kernel works on padded patches (PatchDesc); physical ghost
// values are evaluated on the fly from Eqs. (velBCHomoDiri5th)/(Neumann5) whenever a stencil
// leaves the domain, so no kernel depends on physical ghost cells stored in memory.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "amr4_impl.h"

namespace amr4 {

// Eq. (velBCHomoDiri5th) and Eq. (Neumann5): [bc type][layer-1][m], m = 0..3 inward.
__constant__ double c_ghost[2][2][4] = {
    {{-77.0 / 12.0, 43.0 / 12.0, -17.0 / 12.0, 3.0 / 12.0},
     {-505.0 / 12.0, 335.0 / 12.0, -145.0 / 12.0, 27.0 / 12.0}},
    {{5.0 / 10.0, 9.0 / 10.0, -5.0 / 10.0, 1.0 / 10.0},
     {-75.0 / 10.0, 145.0 / 10.0, -75.0 / 10.0, 15.0 / 10.0}}};
// data coefficient: Dirichlet b (x face value), Neumann b (x h x outward derivative)
__constant__ double c_ghost_b[2][2] = {{5.0, 75.0 / 3.0}, {6.0 / 5.0, 6.0}};
__constant__ float c_ghost_f[2][2][4] = {
    {{-77.0f / 12.0f, 43.0f / 12.0f, -17.0f / 12.0f, 3.0f / 12.0f},
     {-505.0f / 12.0f, 335.0f / 12.0f, -145.0f / 12.0f, 27.0f / 12.0f}},
    {{5.0f / 10.0f, 9.0f / 10.0f, -5.0f / 10.0f, 1.0f / 10.0f},
     {-75.0f / 10.0f, 145.0f / 10.0f, -75.0f / 10.0f, 15.0f / 10.0f}}};
__constant__ float c_ghost_b_f[2][2] = {{5.0f, 75.0f / 3.0f}, {6.0f / 5.0f, 6.0f}};
// AMRCFI 1-D weights [pos][sub][a] for ratio r (r <= 4), set by the host
__constant__ double c_cfi[5 * 4 * 5];
__constant__ float c_cfi_f[5 * 4 * 5];

// Select the double or float copy of a precomputed constant (FP32 kernels never touch the
// FP64 pipe per cell; GB300's FP64 rate is a small fraction of its FP32 rate).
template <typename T>
__device__ __forceinline__ T pick(double d, float f);
template <>
__device__ __forceinline__ double pick<double>(double d, float) { return d; }
template <>
__device__ __forceinline__ float pick<float>(double, float f) { return f; }

template <typename T>
__device__ __forceinline__ T gcoef(int type, int layer, int m) {
  return pick<T>(c_ghost[type][layer][m], c_ghost_f[type][layer][m]);
}
template <typename T>
__device__ __forceinline__ T cfiw(int i) {
  return pick<T>(c_cfi[i], c_cfi_f[i]);
}

// Programmatic dependent launch: every kernel of the library is launched with programmatic
// stream serialisation, so its blocks may be scheduled while the previous kernel on the
// stream drains; each kernel therefore waits here, before touching any global data, until
// the grids it depends on have completed and their memory is visible.  Without the launch
// attribute the instruction returns at once.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr int BX = 32;
constexpr int BY = 8;

struct Cell {
  int c[3];  // local interior coordinates (may be -2..n+1)
};

__device__ __forceinline__ long long poff(const PatchDesc& p, int i, int j, int k) {
  return p.off + (long long)(i + NG) + (long long)(j + NG) * p.sy + (long long)(k + NG) * p.sz;
}

// Map a (blockIdx, threadIdx) to a cell of patch blockIdx.z; false when outside.
template <int D>
__device__ __forceinline__ bool thread_cell(const PatchDesc& p, int nby, int& i, int& j, int& k) {
  i = blockIdx.x * BX + threadIdx.x;
  const int by = (D == 3) ? (int)(blockIdx.y % nby) : (int)blockIdx.y;
  k = (D == 3) ? (int)(blockIdx.y / nby) : 0;
  j = by * BY + threadIdx.y;
  return i < p.n[0] && j < p.n[1] && k < p.n[2];
}

// Physical ghost value at local coordinates c (outside the domain along dimension d only).
template <typename T, int D>
__device__ T phys_ghost(const T* __restrict__ x, const PatchDesc& p, const LevelView& lv,
                        const T* __restrict__ bc, int ci, int cj, int ck, int d) {
  int c[3] = {ci, cj, ck};
  const int g = p.lo[d] + c[d];
  const int side = g < 0 ? 0 : 1;
  const int layer = side == 0 ? -g : g - lv.ndom[d] + 1;  // 1 or 2
  const int f = 2 * d + side;
  const int type = lv.bc[f];
  T v = T(0);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    int cc[3] = {c[0], c[1], c[2]};
    cc[d] = side == 0 ? (m - p.lo[d]) : (lv.ndom[d] - 1 - m - p.lo[d]);
    v += gcoef<T>(type, layer - 1, m) * x[poff(p, cc[0], cc[1], cc[2])];
  }
  if (bc != nullptr) {
    // transverse index over the domain face, lowest remaining dimension fastest
    long long t = 0, s = 1;
    for (int e = 0; e < D; ++e) {
      if (e == d) continue;
      t += (long long)(p.lo[e] + c[e]) * s;
      s *= lv.ndom[e];
    }
    const T gv = bc[lv.bc_off[f] + t];
    const T b = pick<T>(c_ghost_b[type][layer - 1], c_ghost_b_f[type][layer - 1]) *
                (type == 1 ? pick<T>(lv.hd, lv.hf) : T(1));
    v += b * gv;
  }
  return v;
}

// x at local coordinates (ci,cj,ck), evaluating physical ghosts on the fly.  ``ood`` is the
// single dimension that may leave the domain (-1: none checked).
template <typename T, int D>
__device__ __forceinline__ T read_nb(const T* __restrict__ x, const PatchDesc& p, const LevelView& lv,
                                     const T* __restrict__ bc, int ci, int cj, int ck, int d) {
  const int c[3] = {ci, cj, ck};
  const int g = p.lo[d] + c[d];
  if (g < 0 || g >= lv.ndom[d]) return phys_ghost<T, D>(x, p, lv, bc, ci, cj, ck, d);
  return x[poff(p, ci, cj, ck)];
}

// Homogeneous physical extension with corners: each out-of-domain dimension is expanded
// with the layer formula (Fig. 1(c): corner ghosts from already-extended values).
template <typename T, int D>
__device__ T read_ext(const T* __restrict__ x, const PatchDesc& p, const LevelView& lv, int ci, int cj, int ck) {
  const int c[3] = {ci, cj, ck};
  int idx[3][4];
  T w[3][4];
  int cnt[3] = {1, 1, 1};
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    idx[e][0] = c[e];
    w[e][0] = T(1);
    if (e >= D) continue;
    const int g = p.lo[e] + c[e];
    if (g < 0 || g >= lv.ndom[e]) {
      const int side = g < 0 ? 0 : 1;
      const int layer = side == 0 ? -g : g - lv.ndom[e] + 1;
      const int type = lv.bc[2 * e + side];
      cnt[e] = 4;
      for (int m = 0; m < 4; ++m) {
        idx[e][m] = side == 0 ? (m - p.lo[e]) : (lv.ndom[e] - 1 - m - p.lo[e]);
        w[e][m] = gcoef<T>(type, layer - 1, m);
      }
    }
  }
  T v = T(0);
  for (int a = 0; a < cnt[0]; ++a)
    for (int b = 0; b < cnt[1]; ++b)
      for (int q = 0; q < cnt[2]; ++q)
        v += w[0][a] * w[1][b] * w[2][q] * x[poff(p, idx[0][a], idx[1][b], idx[2][q])];
  return v;
}

// True Jacobi diagonal (x 12 h^2): -30 per dimension, plus the ghost-cell coefficients
// that fall back on the cell itself within two cells of a physical face (precomputed per
// face in LevelView::dcorr).
template <typename T, int D>
__device__ __forceinline__ T diag_sum(const LevelView& lv, const PatchDesc& p, const int c[3]) {
  T a = T(-30 * D);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int g = p.lo[d] + c[d];
    if (g == 0) a += pick<T>(lv.dcorr[2 * d][0], lv.dcorr_f[2 * d][0]);
    else if (g == 1) a += pick<T>(lv.dcorr[2 * d][1], lv.dcorr_f[2 * d][1]);
    if (g == lv.ndom[d] - 1) a += pick<T>(lv.dcorr[2 * d + 1][0], lv.dcorr_f[2 * d + 1][0]);
    else if (g == lv.ndom[d] - 2) a += pick<T>(lv.dcorr[2 * d + 1][1], lv.dcorr_f[2 * d + 1][1]);
  }
  return a;
}

// ------------------------------------------------------------------------ level operator
// MODE 0: out = alpha x + beta L x
// MODE 1: out = f - (alpha x + beta L x)
// MODE 2: out = x + omega (f - A x) / diag        (weighted Jacobi, Sec. 6.5)
// MODE 3: out = omega f / diag                    (first sweep from x = 0)
enum { OP_APPLY = 0, OP_RESID = 1, OP_JACOBI = 2, OP_JACOBI0 = 3 };

// 12 h^2 (L x) at one cell (TR = false), or 12 h^2 (L^T x) with the level operator's
// transpose (TR = true): the interior stencil is symmetric; outside the domain there is no
// row, so the transpose reads 0 there and instead gathers the ghost-formula coefficients of
// Eqs. (velBCHomoDiri5th)/(Neumann5) from the two rows that read the physical ghosts
// (ghost 1 is read by the face cell with weight 16 and the next cell with weight -1,
// ghost 2 by the face cell with weight -1).  Zero-CF semantics in both directions: stored
// CF ghost values are used as they are (zero in smoothing buffers).
template <typename T, int D, bool TR>
__device__ __forceinline__ T cell_Lx(const LevelView& lv, const PatchDesc& p, int i, int j, int k,
                                     const T* __restrict__ x, const T* __restrict__ bc) {
  const long long o = poff(p, i, j, k);
  const T xc = x[o];
  T s1 = T(0), s2 = T(0), extra = T(0);
  const int c[3] = {i, j, k};
  const long long st[3] = {1, p.sy, p.sz};
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int g = p.lo[d] + c[d];
    T m1, p1, m2, p2;
    if (g >= 2 && g <= lv.ndom[d] - 3) {
      m1 = x[o - st[d]];
      p1 = x[o + st[d]];
      m2 = x[o - 2 * st[d]];
      p2 = x[o + 2 * st[d]];
    } else if (!TR) {
      int cc[3] = {i, j, k};
      cc[d] = c[d] - 1; m1 = read_nb<T, D>(x, p, lv, bc, cc[0], cc[1], cc[2], d);
      cc[d] = c[d] + 1; p1 = read_nb<T, D>(x, p, lv, bc, cc[0], cc[1], cc[2], d);
      cc[d] = c[d] - 2; m2 = read_nb<T, D>(x, p, lv, bc, cc[0], cc[1], cc[2], d);
      cc[d] = c[d] + 2; p2 = read_nb<T, D>(x, p, lv, bc, cc[0], cc[1], cc[2], d);
    } else {
      m1 = (g - 1 >= 0) ? x[o - st[d]] : T(0);
      m2 = (g - 2 >= 0) ? x[o - 2 * st[d]] : T(0);
      p1 = (g + 1 < lv.ndom[d]) ? x[o + st[d]] : T(0);
      p2 = (g + 2 < lv.ndom[d]) ? x[o + 2 * st[d]] : T(0);
    }
    s1 += m1 + p1;
    s2 += m2 + p2;
    if (TR) {
      // low face: this cell is interior cell m = g of the rows' ghost formulas
      if (g <= 3 && p.lo[d] == 0) {
        const int t = lv.bc[2 * d];
        const long long o0 = o - (long long)c[d] * st[d];  // local index 0 along d
        const T w1 = T(16) * x[o0] - x[o0 + st[d]];
        const T w2 = -x[o0];
        extra += gcoef<T>(t, 0, g) * w1 + gcoef<T>(t, 1, g) * w2;
      }
      const int m = lv.ndom[d] - 1 - g;
      if (m <= 3 && p.lo[d] + p.n[d] == lv.ndom[d]) {
        const int t = lv.bc[2 * d + 1];
        const long long o0 = o + (long long)(p.n[d] - 1 - c[d]) * st[d];  // last cell along d
        const T w1 = T(16) * x[o0] - x[o0 - st[d]];
        const T w2 = -x[o0];
        extra += gcoef<T>(t, 0, m) * w1 + gcoef<T>(t, 1, m) * w2;
      }
    }
  }
  return (T(16) * s1 - s2 - T(30 * D) * xc) + extra;
}

template <typename T, int D, int MODE, bool TR = false>
__device__ __forceinline__ void cell_level_op(const LevelView& lv, const PatchDesc& p, int i, int j, int k,
                                              const T* __restrict__ x, const T* __restrict__ f,
                                              T* __restrict__ out, const T* __restrict__ bc, T alpha, T beta,
                                              T omega) {
  const long long o = poff(p, i, j, k);
  const T inv = pick<T>(lv.inv12h2, lv.inv12h2_f);
  const int c[3] = {i, j, k};
  if (MODE == OP_JACOBI0) {
    const T diag = alpha + beta * inv * diag_sum<T, D>(lv, p, c);
    out[o] = omega * f[o] / diag;
    return;
  }
  const T xc = x[o];
  const T ax = alpha * xc + beta * (cell_Lx<T, D, TR>(lv, p, i, j, k, x, bc) * inv);
  if (MODE == OP_APPLY) {
    out[o] = ax;
  } else if (MODE == OP_RESID) {
    out[o] = f[o] - ax;
  } else {
    const T diag = alpha + beta * inv * diag_sum<T, D>(lv, p, c);
    out[o] = xc + omega * (f[o] - ax) / diag;
  }
}

// distance class of global index g to the faces of an n-cell dimension: 0 interior, 1 and 2
// the first and second cell from the low face, 3 and 4 from the high face
__device__ __forceinline__ int face_class(int g, int n) {
  return g == 0 ? 1 : g == 1 ? 2 : g == n - 1 ? 3 : g == n - 2 ? 4 : 0;
}

// Jacobi factors omega / diag by distance class of the cell to the x, y [and z] faces
// (face_class; index x + 5 y [+ 25 z]), filled on the host (jacobi_factors).
template <typename T, int D>
struct JFac {
  T w[D == 3 ? 125 : 25];
};

// Sums of the first and of the second neighbours along one dimension of the cell at offset o,
// g <= 1 or g >= n - 2 (global index, n cells in the domain): a face cell reads the ghost
// layers 1 and 2, its neighbour layer 1.  Ghost values in read_nb's order of operations; both
// sums are commutative, so the low and the high side share one form.
template <typename T>
__device__ __forceinline__ void face_sums(const T* __restrict__ xb, int o, int st, int g, int n, int tlo, int thi, T& a1,
                                          T& a2) {
  const bool low = g < 2;
  const int q = low ? g : n - 1 - g;
  const int s = low ? st : -st;
  const int t = low ? tlo : thi;
  const int b = o - q * s;
  const T c0 = xb[b], c1 = xb[b + s], c2 = xb[b + 2 * s], c3 = xb[b + 3 * s];
  T g1 = T(0);
  g1 += gcoef<T>(t, 0, 0) * c0;
  g1 += gcoef<T>(t, 0, 1) * c1;
  g1 += gcoef<T>(t, 0, 2) * c2;
  g1 += gcoef<T>(t, 0, 3) * c3;
  if (q == 0) {
    T g2 = T(0);
    g2 += gcoef<T>(t, 1, 0) * c0;
    g2 += gcoef<T>(t, 1, 1) * c1;
    g2 += gcoef<T>(t, 1, 2) * c2;
    g2 += gcoef<T>(t, 1, 3) * c3;
    a1 = g1 + c1;
    a2 = g2 + c2;
  } else {
    a1 = c0 + c2;
    a2 = g1 + c3;
  }
}

// neighbour sums along one dimension, class 0: two cells or more from both faces
template <typename T>
__device__ __forceinline__ void line_sums(const T* __restrict__ xb, int o, int st, bool inner, int g, int n, int tlo,
                                          int thi, T& a1, T& a2) {
  if (inner) {
    a1 = xb[o - st] + xb[o + st];
    a2 = xb[o - 2 * st] + xb[o + 2 * st];
  } else {
    face_sums<T>(xb, o, st, g, n, tlo, thi, a1, a2);
  }
}

// The transposed operator's sums along one dimension (cell_Lx with TR): zero outside the domain,
// and in the four cells next to a face ``ex`` gathers the ghost coefficients of the two rows
// that read the ghosts.  i: patch-local index, n: domain, [plo, plo + pn): the patch.
template <typename T>
__device__ __forceinline__ void trans_sums(const T* __restrict__ xb, int o, int st, int i, int n, int plo, int pn, int tlo,
                                           int thi, T& a1, T& a2, T& ex) {
  const int g = plo + i;
  const T m1 = g >= 1 ? xb[o - st] : T(0), p1 = g + 1 < n ? xb[o + st] : T(0);
  const T m2 = g >= 2 ? xb[o - 2 * st] : T(0), p2 = g + 2 < n ? xb[o + 2 * st] : T(0);
  a1 = m1 + p1;
  a2 = m2 + p2;
  if (g <= 3 && plo == 0) {
    const int f = o - i * st;
    const T w1 = T(16) * xb[f] - xb[f + st], w2 = -xb[f];
    ex += gcoef<T>(tlo, 0, g) * w1 + gcoef<T>(tlo, 1, g) * w2;
  }
  const int m = n - 1 - g;
  if (m <= 3 && plo + pn == n) {
    const int f = o + (pn - 1 - i) * st;
    const T w1 = T(16) * xb[f] - xb[f - st], w2 = -xb[f];
    ex += gcoef<T>(thi, 0, m) * w1 + gcoef<T>(thi, 1, m) * w2;
  }
}

// f - A x (or f - A^T x) coefficients and sums of one cell near a face, 2-D, homogeneous data
template <typename T, int MODE, bool TR>
__device__ __forceinline__ void edge_op2d(const LevelView& lv, const PatchDesc& p, int i, int j, const T* __restrict__ x,
                                          const T* __restrict__ f, T* __restrict__ out, T alpha, T beta,
                                          const JFac<T, 2>& jf) {
  const int sy = (int)p.sy, o = (j + NG) * sy + i + NG;
  const int gx = p.lo[0] + i, gy = p.lo[1] + j;
  const int cx = face_class(gx, lv.ndom[0]), cy = face_class(gy, lv.ndom[1]);
  if (MODE == OP_JACOBI0) {
    out[p.off + o] = jf.w[cx + 5 * cy] * f[p.off + o];
    return;
  }
  const T* __restrict__ xb = x + p.off;
  const T xc = xb[o];
  T fk = T(0);
  if (MODE != OP_APPLY) fk = f[p.off + o];
  T x1, x2, y1, y2, ex = T(0);
  if (TR) {
    trans_sums<T>(xb, o, 1, i, lv.ndom[0], p.lo[0], p.n[0], lv.bc[0], lv.bc[1], x1, x2, ex);
    trans_sums<T>(xb, o, sy, j, lv.ndom[1], p.lo[1], p.n[1], lv.bc[2], lv.bc[3], y1, y2, ex);
  } else {
    line_sums<T>(xb, o, 1, cx == 0, gx, lv.ndom[0], lv.bc[0], lv.bc[1], x1, x2);
    line_sums<T>(xb, o, sy, cy == 0, gy, lv.ndom[1], lv.bc[2], lv.bc[3], y1, y2);
  }
  const T s1 = x1 + y1, s2 = x2 + y2;
  const T inv = pick<T>(lv.inv12h2, lv.inv12h2_f);
  const T ax = alpha * xc + beta * (((T(16) * s1 - s2 - T(60) * xc) + ex) * inv);
  if (MODE == OP_APPLY) out[p.off + o] = ax;
  else if (MODE == OP_RESID) out[p.off + o] = fk - ax;
  else out[p.off + o] = xc + jf.w[cx + 5 * cy] * (fk - ax);
}

template <typename T, int D, int MODE, bool TR = false>
__global__ void __launch_bounds__(BX* BY) k_level_op(LevelView lv, int nby, const T* __restrict__ x,
                                                     const T* __restrict__ f, T* __restrict__ out,
                                                     const T* __restrict__ bc, T alpha, T beta, T omega,
                                                     const unsigned char* __restrict__ vmask) {
  pdl_wait();
  const PatchDesc p = lv.patches[blockIdx.z];
  int i, j, k;
  if (!thread_cell<D>(p, nby, i, j, k)) return;
  if (vmask != nullptr && vmask[poff(p, i, j, k)] == 0) return;
  cell_level_op<T, D, MODE, TR>(lv, p, i, j, k, x, f, out, bc, alpha, beta, omega);
}

// 2-D level operator, tiled: each thread computes ROWS (1, 2 or 4; chosen per grid by the
// autotuner) consecutive cells of one column with 32-bit patch-local offsets and reuses the
// column loads.  A thread whose cells (plus the two-cell stencil reach) lie inside the
// domain and the patch takes the fast path with the constant interior diagonal (omega /
// diag precomputed); the others run the generic per-cell code.  Both paths sum the
// stencil in the same order as cell_Lx.
template <typename T, int MODE, bool TR, int ROWS>
__device__ __forceinline__ void level_op2d_tiled_body(const LevelView& lv, int pz, const T* __restrict__ x,
                                                      const T* __restrict__ f, T* __restrict__ out,
                                                      const T* __restrict__ bc, T alpha, T beta, T omega,
                                                      T omega_over_diag, const unsigned char* __restrict__ vmask,
                                                      const JFac<T, 2>& jf) {
  const PatchDesc p = lv.patches[pz];
  const int i = blockIdx.x * BX + threadIdx.x;
  const int j0 = (blockIdx.y * BY + threadIdx.y) * ROWS;
  // per thread: its column strip and the two-cell reach inside the patch and the domain
  // (the transpose also gathers ghost coefficients at distance 2 and 3 from a physical face)
  const bool full = i < p.n[0] && j0 + ROWS <= p.n[1];
  constexpr int M = TR ? 4 : 2;
  const int g0 = p.lo[0] + i, g1 = p.lo[1] + j0;
  const bool inside = g0 >= M && g0 <= lv.ndom[0] - 1 - M && g1 >= M && g1 + ROWS - 1 <= lv.ndom[1] - 1 - M;
  if (!(full && inside)) {
    if (i >= p.n[0]) return;
    for (int r = 0; r < ROWS; ++r) {
      const int j = j0 + r;
      if (j >= p.n[1]) return;
      if (vmask != nullptr && vmask[poff(p, i, j, 0)] == 0) continue;
      if (bc != nullptr)
        cell_level_op<T, 2, MODE, TR>(lv, p, i, j, 0, x, f, out, bc, alpha, beta, omega);
      else edge_op2d<T, MODE, TR>(lv, p, i, j, x, f, out, alpha, beta, jf);
    }
    return;
  }
  const T* __restrict__ xb = x + p.off;
  const int sy = (int)p.sy;
  const int o = (j0 + NG) * sy + (i + NG);
  const T inv = pick<T>(lv.inv12h2, lv.inv12h2_f);
  if (MODE == OP_JACOBI0) {
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
      if (vmask == nullptr || vmask[p.off + o + r * sy]) out[p.off + o + r * sy] = omega_over_diag * f[p.off + o + r * sy];
    return;
  }
  T col[ROWS + 4];
#pragma unroll
  for (int q = 0; q < ROWS + 4; ++q) col[q] = xb[o + (q - 2) * sy];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int orr = o + r * sy;
    if (vmask != nullptr && !vmask[p.off + orr]) continue;
    const T xc = col[r + 2];
    const T s1 = (xb[orr - 1] + xb[orr + 1]) + (col[r + 1] + col[r + 3]);
    const T s2 = (xb[orr - 2] + xb[orr + 2]) + (col[r] + col[r + 4]);
    const long long og = p.off + orr;
    if constexpr (sizeof(T) == 8) {
      // FP64: alpha x + beta L x = kc0 x + kc1 s1 - kc2 s2, three multiply-adds after the sums
      // (FP64 arithmetic, not memory, bounds these passes on this part)
      const T kc2 = beta * inv, kc1 = T(16) * kc2, kc0 = alpha - T(60) * kc2;
      if (MODE == OP_APPLY) {
        out[og] = kc0 * xc + (kc1 * s1 - kc2 * s2);
      } else {
        const T res = fma(kc2, s2, fma(-kc1, s1, fma(-kc0, xc, f[og])));
        if (MODE == OP_RESID) out[og] = res;
        else out[og] = fma(omega_over_diag, res, xc);
      }
    } else {
      const T lap = (T(16) * s1 - s2 - T(60) * xc) + T(0);
      const T ax = alpha * xc + beta * (lap * inv);
      if (MODE == OP_APPLY) out[og] = ax;
      else if (MODE == OP_RESID) out[og] = f[og] - ax;
      else out[og] = xc + omega_over_diag * (f[og] - ax);
    }
  }
}

template <typename T, int MODE, bool TR, int ROWS>
__global__ void __launch_bounds__(BX* BY) k_level_op2d_tiled(LevelView lv, const T* __restrict__ x,
                                                             const T* __restrict__ f, T* __restrict__ out,
                                                             const T* __restrict__ bc, T alpha, T beta, T omega,
                                                             T omega_over_diag, const unsigned char* __restrict__ vmask,
                                                             const __grid_constant__ JFac<T, 2> jf) {
  pdl_wait();
  level_op2d_tiled_body<T, MODE, TR, ROWS>(lv, blockIdx.z, x, f, out, bc, alpha, beta, omega, omega_over_diag, vmask, jf);
}

// ------------------------------------------------------------------------ z-chunked 3-D marching operator
// Level operator on a single-patch 3-D level whose x and y extents are multiples of the
// 32 x 8R tile (R = 2 or 4 rows per thread, chosen per grid by the tile autotuner).  Block b
// marches up z through chunk b / ntiles of tile column b % ntiles; the host sizes the chunks
// so that the grid fits one wave, and since neighbouring tiles carry consecutive block
// indices they march side by side and a tile's halo rows come from L2 where the neighbour
// has just brought them in.  Thread (tx, ty) owns the columns (i0 + tx, j0 + ty + 8 r),
// r < R: x at planes k-2..k+2 of each sits in registers, the plane k with its two-cell halo
// in shared memory (double-buffered, one barrier per plane).  Every load of x, f and the
// halo is issued two planes before its use (two register slots used alternately, so no
// register with a load in flight is ever copied), and offsets inside the patch are 32-bit.
// Physical ghost values outside the domain come from the same formulas as everywhere else,
// the Jacobi factor from the 125-entry distance-class table.
constexpr int ZC_TX = 32, ZC_TY = 8, ZC_W = ZC_TX + 4;

template <int R>
struct ZcGeom {
  static constexpr int TH = ZC_TY * R;                   // tile rows
  static constexpr int SH = TH + 4;                      // shared-plane rows
  static constexpr int NH = 2 * 2 * ZC_TX + 2 * 2 * TH;  // halo cells the stencil reads
};

// x of column ``col`` at patch-local plane k: stored values inside the domain, outside it in
// z Eq. (velBCHomoDiri5th) / Eq. (Neumann5) with homogeneous data from the four planes next
// to the face (a block-uniform branch, taken only by chunks at a z face)
template <typename T>
__device__ __forceinline__ T zc_zval(const T* __restrict__ xb, int col, int sz, int k, int lz, int nzd,
                                     const LevelView& lv) {
  const int g = lz + k;
  if (g >= 0 && g < nzd) return xb[col + (k + NG) * sz];
  const int side = g < 0 ? 0 : 1, layer = side == 0 ? -g : g - nzd + 1, type = lv.bc[4 + side];
  const int k0 = (side == 0 ? 0 : nzd - 1) - lz + NG, dk = side == 0 ? sz : -sz;
  T v = T(0);
#pragma unroll
  for (int m = 0; m < 4; ++m) v += gcoef<T>(type, layer - 1, m) * xb[col + k0 * sz + m * dk];
  return v;
}

template <int I>
using zc_slot = std::integral_constant<int, I>;

template <typename T, int MODE, int R>
__global__ void __launch_bounds__(ZC_TX* ZC_TY, (sizeof(T) == 4 ? 8 : 4) / R)
    k_level_op3d_zc(LevelView lv, int ntx, int ntiles, int kc, const T* __restrict__ x, const T* __restrict__ f,
                    T* __restrict__ out, T alpha, T beta, T omega, const unsigned char* __restrict__ vmask,
                    const unsigned* __restrict__ gate) {
  using G = ZcGeom<R>;
  pdl_wait();
  // stacked component batches: the grid holds ncomp equal parts, part c on replica c
  const int bpc = gridDim.x / lv.ncomp, comp = blockIdx.x / bpc, blk = blockIdx.x % bpc;
  if (gate != nullptr && gate[4 * comp] == 0u) return;  // gated launch: runs only when the flag is set
  if (lv.active != nullptr && !lv.active[comp]) return;  // converged replica of a stacked batch
  __shared__ T sp[2][G::SH * ZC_W];
  __shared__ T wt[125];
  const PatchDesc p = lv.patches[comp];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * ZC_TX + tx;
  const T inv = pick<T>(lv.inv12h2, lv.inv12h2_f);
  if (MODE == OP_JACOBI || MODE == OP_JACOBI0) {
    for (int q = tid; q < 125; q += ZC_TX * ZC_TY) {
      const int a = q % 5, b = (q / 5) % 5, c = q / 25;
      const int cls[3] = {a, b, c};
      T acc = T(-90);
#pragma unroll
      for (int d = 0; d < 3; ++d)
        if (cls[d]) acc += pick<T>(lv.dcorr[2 * d + (cls[d] - 1) / 2][(cls[d] - 1) % 2],
                                   lv.dcorr_f[2 * d + (cls[d] - 1) / 2][(cls[d] - 1) % 2]);
      wt[q] = omega / (alpha + beta * inv * acc);
    }
  }
  const int sy = (int)p.sy, sz = (int)p.sz, nz = p.n[2];
  const int nzd = lv.ndom[2], lz = p.lo[2];
  const T* __restrict__ xb = x + p.off;
  const T* __restrict__ fb = f + p.off;
  T* __restrict__ ob = out + p.off;
  // alpha x + beta L x = kc0 x + kc1 s1 - kc2 s2 with s1, s2 the sums of the six distance-1 and
  // distance-2 neighbours (Eq. discreteOps: 12 h^2 L x = 16 s1 - s2 - 90 x): three multiply-adds
  // after the sums, which matters most in FP64, whose rate on this part is a small fraction of FP32's
  const T kc2 = beta * inv, kc1 = T(16) * kc2, kc0 = alpha - T(90) * kc2;
  // valid mask: only residuals are masked
  const unsigned char* __restrict__ vb = (MODE == OP_RESID && vmask) ? vmask + p.off : nullptr;
  // this thread's halo cell (tile-local): warps 0-1 the two rows below the tile, 2-3 the two
  // rows above, the next ones the two columns on each side (lane pairs share a row)
  int hx = 0, hy = 0;
  const bool has_halo = tid < G::NH;
  {
    const int q = tid;
    if (q < 2 * ZC_TX) {
      hy = -2 + q / ZC_TX;
      hx = q % ZC_TX;
    } else if (q < 4 * ZC_TX) {
      hy = G::TH + (q - 2 * ZC_TX) / ZC_TX;
      hx = q % ZC_TX;
    } else if (q < G::NH) {
      const int r = q - 4 * ZC_TX, side = r / (2 * G::TH), c = r & 1;
      hy = (r % (2 * G::TH)) >> 1;
      hx = side == 0 ? c - 2 : ZC_TX + c;
    }
  }
  const int hs = (hy + 2) * ZC_W + hx + 2;
  const int c0 = (ty + 2) * ZC_W + tx + 2;  // shared index of row r: c0 + r * ZC_TY * ZC_W
  const int tile = blk % ntiles, ka = (blk / ntiles) * kc, kb = min(nz, ka + kc);
  __syncthreads();  // weight table
  if (ka >= kb) return;
  const int i0 = (tile % ntx) * ZC_TX, j0 = (tile / ntx) * G::TH;
  const int i = i0 + tx;
  const int col0 = (i + NG) + (j0 + ty + NG) * sy;  // column of row r: col0 + r * ZC_TY * sy
  const int kx = face_class(p.lo[0] + i, lv.ndom[0]);
  int wxy[R];
#pragma unroll
  for (int r = 0; r < R; ++r) wxy[r] = kx + 5 * face_class(p.lo[1] + j0 + ty + r * ZC_TY, lv.ndom[1]);
  // halo cell: stored value inside the domain (interior, CF or copy ghost).  Outside it (the
  // tile then touches that domain face) the ghost formula along the face normal, evaluated in
  // shared memory from the four staged cells next to the face, after the plane is staged;
  // hsrc / hstep give the face cell's shared index and the inward step (corners of the halo
  // are never read).
  const int hli = i0 + hx, hlj = j0 + hy;
  const int hcol = (hli + NG) + (hlj + NG) * sy;
  int hsrc = 0, hstep = 0, htype = 0, hlayer = 0;
  {
    const int hgi = p.lo[0] + hli, hgj = p.lo[1] + hlj;
    const int d = (hgi < 0 || hgi >= lv.ndom[0]) ? 0 : ((hgj < 0 || hgj >= lv.ndom[1]) ? 1 : -1);
    if (has_halo && d >= 0) {
      const int g = d == 0 ? hgi : hgj, n = lv.ndom[d], side = g < 0 ? 0 : 1;
      hlayer = (side == 0 ? -g : g - n + 1) - 1;
      htype = lv.bc[2 * d + side];
      const int face = (side == 0 ? 0 : n - 1) - p.lo[d] - (d == 0 ? i0 : j0);  // tile-local
      hsrc = d == 0 ? (hy + 2) * ZC_W + face + 2 : (face + 2) * ZC_W + hx + 2;
      const int st = d == 0 ? 1 : ZC_W;
      hstep = side == 0 ? st : -st;
    }
  }
  const bool hload = has_halo && hstep == 0;
  // blocks whose halo leaves the domain fill it after staging (block-uniform)
  const bool face_tile = p.lo[0] + i0 == 0 || p.lo[0] + i0 + ZC_TX == lv.ndom[0] || p.lo[1] + j0 == 0 ||
                         p.lo[1] + j0 + G::TH == lv.ndom[1];
  auto halo = [&](int k) -> T { return hload ? xb[hcol + (k + NG) * sz] : T(0); };
  constexpr int RS = ZC_TY;  // row step of a thread's columns (rows)
  T q[R][5];                 // x of each column at planes k-2..k+2
  T xs[2][R], fs[2][R], hv[2];
#pragma unroll
  for (int r = 0; r < R; ++r) {
#pragma unroll
    for (int m = 0; m < 5; ++m) q[r][m] = T(0);
    xs[0][r] = xs[1][r] = fs[0][r] = fs[1][r] = T(0);
  }
  hv[0] = hv[1] = T(0);
  if (MODE != OP_JACOBI0) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int col = col0 + r * RS * sy;
      q[r][0] = zc_zval<T>(xb, col, sz, ka - 2, lz, nzd, lv);
      q[r][1] = zc_zval<T>(xb, col, sz, ka - 1, lz, nzd, lv);
      q[r][2] = xb[col + (ka + NG) * sz];
      q[r][3] = zc_zval<T>(xb, col, sz, ka + 1, lz, nzd, lv);
      q[r][4] = zc_zval<T>(xb, col, sz, ka + 2, lz, nzd, lv);
      if (ka + 1 < kb) xs[0][r] = zc_zval<T>(xb, col, sz, ka + 3, lz, nzd, lv);  // q4 of plane ka+1
      if (ka + 2 < kb) xs[1][r] = zc_zval<T>(xb, col, sz, ka + 4, lz, nzd, lv);  // q4 of plane ka+2
    }
    if (has_halo) {
      hv[0] = halo(ka);
      if (ka + 1 < kb) hv[1] = halo(ka + 1);
    }
  }
  if (MODE != OP_APPLY) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int col = col0 + r * RS * sy;
      fs[0][r] = fb[col + (ka + NG) * sz];
      if (ka + 1 < kb) fs[1][r] = fb[col + (ka + 1 + NG) * sz];
    }
  }
  // one plane: stage, refill the consumed slots with plane k+2, barrier, compute, advance
  // the queues (q4 from the slot loaded two planes ago, then the slot reloaded)
  auto step = [&](int k, auto slot, auto safe) {
    constexpr int S = decltype(slot)::value;
    constexpr bool SAFE = decltype(safe)::value;  // planes up to k+5 inside the domain
    T* __restrict__ s = sp[S];
    T fk[R];
#pragma unroll
    for (int r = 0; r < R; ++r) fk[r] = fs[S][r];
    if (MODE != OP_JACOBI0) {
#pragma unroll
      for (int r = 0; r < R; ++r) s[c0 + r * RS * ZC_W] = q[r][2];
      if (hload) {
        s[hs] = hv[S];
        if (k + 2 < kb) hv[S] = halo(k + 2);
      }
    }
    if (MODE != OP_APPLY && k + 2 < kb) {
#pragma unroll
      for (int r = 0; r < R; ++r) fs[S][r] = fb[col0 + r * RS * sy + (k + 2 + NG) * sz];
    }
    if (MODE != OP_JACOBI0) {
      __syncthreads();
      if (face_tile) {
        if (hstep != 0) {
          T v = T(0);
#pragma unroll
          for (int m = 0; m < 4; ++m) v += gcoef<T>(htype, hlayer, m) * s[hsrc + m * hstep];
          s[hs] = v;
        }
        __syncthreads();
      }
    }
    const int kz25 = 25 * face_class(lz + k, nzd);
    const int pk = col0 + (k + NG) * sz;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int P = pk + r * RS * sy;
      if (MODE == OP_JACOBI0) {
        ob[P] = wt[wxy[r] + kz25] * fk[r];
      } else {
        const int C = c0 + r * RS * ZC_W;
        const T xc = q[r][2];
        const T s1 = ((s[C - 1] + s[C + 1]) + (s[C - ZC_W] + s[C + ZC_W])) + (q[r][1] + q[r][3]);
        const T s2 = ((s[C - 2] + s[C + 2]) + (s[C - 2 * ZC_W] + s[C + 2 * ZC_W])) + (q[r][0] + q[r][4]);
        if (MODE == OP_APPLY) {
          ob[P] = kc0 * xc + (kc1 * s1 - kc2 * s2);
        } else {
          const T res = fma(kc2, s2, fma(-kc1, s1, fma(-kc0, xc, fk[r])));
          if (MODE == OP_RESID) { if (vb == nullptr || vb[P]) ob[P] = res; }
          else ob[P] = fma(wt[wxy[r] + kz25], res, xc);
        }
      }
    }
    if (MODE != OP_JACOBI0) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        q[r][0] = q[r][1];
        q[r][1] = q[r][2];
        q[r][2] = q[r][3];
        q[r][3] = q[r][4];
        q[r][4] = xs[S][r];
        if (k + 3 < kb) {  // q4 of plane k+3
          if (SAFE) xs[S][r] = xb[col0 + r * RS * sy + (k + 5 + NG) * sz];
          else xs[S][r] = zc_zval<T>(xb, col0 + r * RS * sy, sz, k + 5, lz, nzd, lv);
        }
      }
    }
  };
  for (int k = ka; k < kb; k += 2) {
    if (lz + k + 6 < nzd) {
      step(k, zc_slot<0>{}, std::true_type{});
      if (k + 1 < kb) step(k + 1, zc_slot<1>{}, std::true_type{});
    } else {
      step(k, zc_slot<0>{}, std::false_type{});
      if (k + 1 < kb) step(k + 1, zc_slot<1>{}, std::false_type{});
    }
  }
}

// ------------------------------------------------------------------------ precision conversions
// GB300 executes FP64 instructions (conversions to and from FP64 among them) at a small
// fraction of its integer rate, and the refinement loop converts every cell twice per
// iteration (the FP32 correction to FP64, the FP64 residual to FP32).  These two helpers do
// the conversions with integer instructions and give the results of the hardware
// conversions: FP32 -> FP64 exactly, FP64 -> FP32 rounded to nearest even.  Values outside
// the normal FP32 range (apart from zero) take the hardware conversion.
__device__ __forceinline__ double f32_to_f64(float v) {
  const unsigned u = __float_as_uint(v);
  const unsigned e = (u >> 23) & 0xffu;
  if (e == 0u || e == 0xffu) {
    if ((u & 0x7fffffffu) == 0u) return __hiloint2double((int)(u & 0x80000000u), 0);  // signed zero
    return (double)v;
  }
  // exponent rebased by 1023 - 127, the 23-bit significand at the top of the 52-bit one
  return __hiloint2double((int)((u & 0x80000000u) | ((e + 896u) << 20) | ((u & 0x7fffffu) >> 3)), (int)(u << 29));
}
__device__ __forceinline__ float f64_to_f32(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const unsigned e = (hi >> 20) & 0x7ffu, sg = hi & 0x80000000u;
  if (e >= 897u && e <= 1150u) {  // 2^-126 <= |v| < 2^128
    // the top 23 of the 52 significand bits, rounded on the 29 below (ties to even); a carry
    // out of the significand moves the exponent on (to infinity above the largest float)
    const unsigned keep = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned rem = lo & 0x1fffffffu;
    const unsigned up = (rem > 0x10000000u || (rem == 0x10000000u && (keep & 1u))) ? 1u : 0u;
    return __uint_as_float(sg | (((e - 896u) << 23) + keep + up));
  }
  if ((b << 1) == 0ull) return __uint_as_float(sg);  // signed zero
  return (float)v;
}
// value-type conversion S -> T through the helpers above where one side is FP32
template <typename T, typename S>
__device__ __forceinline__ T cvt(S v) {
  return T(v);
}
template <>
__device__ __forceinline__ double cvt<double, float>(float v) {
  return f32_to_f64(v);
}
template <>
__device__ __forceinline__ float cvt<float, double>(double v) {
  return f64_to_f32(v);
}

// ------------------------------------------------------------------------ 3-D FP64 residual in fixed point
// GB300 issues FP64 arithmetic at a small fraction of its integer rate, and the FP64 residual
// of the refinement loop (13 FP64 operations per cell in floating point) is bound by that
// rate.  Here the sums of the stencil are formed exactly in 64-bit integers: every value of
// x the stencil reads is rounded once to a fixed-point frame set by the level's largest
// interior |x| (its leading bit at bit 52), so that T = 16 s1 - s2 - 90 x (Eq. discreteOps:
// 12 h^2 L x = T) is exact in 64 bits.  Bounds: interior values are below 2^53; a stored ghost
// value (coarse-fine, copy) must stay below 2^55; a physical ghost value is a fixed
// combination of interior values (Eqs. velBCHomoDiri5th, Neumann5: at most 11.7 times the
// largest in layer 1 and 84.4 times in layer 2), and a cell reads at most one ghost per
// direction, so |T| < (16 (3 * 11.7 + 3) + 3 * 84.4 + 3 + 90) 2^53 < 2^63.
// T is rounded once to FP64 and r = f - alpha x - (beta / 12 h^2) 2^-S T takes two FP64
// multiply-adds.  Rounding x to the frame changes it by at most half a unit in the last
// place of the largest |x|, the size of one FP64 rounding of that value, so the result is as
// accurate as the floating-point evaluation, whose sums round several times.  A value outside
// the frame (a stored ghost value more than four times the bound on the interior values, or
// a non-finite value) sets *flag, and the plain FP64 kernel, launched after this one with
// that flag as its gate, recomputes the level.

// round(x 2^(1075 - emax)) to the nearest integer (ties away from zero): the frame of a level
// whose largest |x| has biased exponent emax (so that |x| < 2^(emax - 1022) maps below
// 2^53); a value of 2^lim * 2^(emax - 1022) or more in magnitude (lim = 2 for stored values,
// 7 for physical ghost values), or a non-finite one, sets ovf
__device__ __forceinline__ long long fx_of(double x, int emax, int lim, bool& ovf) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned bh = (unsigned)(b >> 32), bl = (unsigned)b;
  const int e = (int)((bh >> 20) & 0x7ffu);
  const int sh = e - emax;  // x 2^S = m 2^sh, m the 53-bit significand
  unsigned long long u;
  if (sh <= 0 && sh > -32 && e != 0) {
    // the common case, values within 2^31 of the frame's largest, in 32-bit halves:
    // (m + 2^(s-1)) >> s with s = -sh < 32
    const unsigned s = (unsigned)(-sh);
    const unsigned mh = (bh & 0xfffffu) | 0x100000u;
    const unsigned half = (1u << s) >> 1;
    const unsigned lo = bl + half;
    const unsigned hi = mh + (lo < bl ? 1u : 0u);
    u = ((unsigned long long)(hi >> s) << 32) | __funnelshift_r(lo, hi, s);
  } else {
    if (sh > lim || e == 0x7ff) ovf = true;
    // m 2^sh rounded = (m 2^10 + 2^(9 - sh)) >> (10 - sh) for -54 < sh <= lim <= 9 (m 2^10 <
    // 2^63: the sum does not wrap); zero below that, and for zero and subnormal values, which
    // lie below any frame's unit
    const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    const int r = 10 - sh;
    const bool keep = e != 0 && sh <= lim && r < 64;
    u = keep ? ((m << 10) + (1ull << ((r - 1) & 63))) >> (r & 63) : 0ull;
  }
  return (bh >> 31) ? -(long long)u : (long long)u;
}

// a 64-bit integer to FP64, rounded to nearest (ties to even), with integer instructions only
__device__ __forceinline__ double fx_to_double(long long t) {
  if (t == 0) return 0.0;
  const unsigned long long sg = (unsigned long long)t & 0x8000000000000000ull;
  unsigned long long u = sg ? 0ull - (unsigned long long)t : (unsigned long long)t;
  const int lz = __clzll((long long)u);
  u <<= lz;                                // leading one at bit 63
  unsigned long long mant = u >> 11;       // 53 bits, the leading one at bit 52
  const unsigned rem = (unsigned)(u & 0x7ffull);
  mant += (rem > 0x400u || (rem == 0x400u && (mant & 1ull))) ? 1ull : 0ull;
  // biased exponent 1086 - lz; adding the significand with its leading one to (exponent - 1)
  // << 52 carries a rounding overflow into the exponent
  return __longlong_as_double((long long)(sg | ((((unsigned long long)(1085 - lz)) << 52) + mant)));
}

// largest |x| over the interior cells of a single-patch level, as IEEE bits cut to the upper word (non-negative
// doubles order like their bit patterns), into *acc; block size 256
__global__ void __launch_bounds__(256) k_absmax_patch(LevelView lv, const double* __restrict__ x,
                                                      unsigned long long* __restrict__ acc) {
  pdl_wait();
  // stacked component batches: blockIdx.y = replica, its maximum in acc[2 * replica]
  if (lv.active != nullptr && !lv.active[blockIdx.y]) return;  // converged replica of a stacked batch
  const PatchDesc p = lv.patches[blockIdx.y];
  acc += 2 * blockIdx.y;
  const int n0 = p.n[0], n1 = p.n[1], rows = p.n[1] * p.n[2];
  // the frame is set by the exponent alone, so the upper words are compared
  unsigned v = 0u;
  // one warp per row, eight loads of a lane in flight
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  for (int r = blockIdx.x * wpb + (threadIdx.x >> 5); r < rows; r += gridDim.x * wpb) {
    const double* __restrict__ row = x + p.off + (long long)(r / n1 + NG) * p.sz + (long long)(r % n1 + NG) * p.sy + NG;
#pragma unroll 8
    for (int i = lane; i < n0; i += 32) {
      v = max(v, (unsigned)__double2hiint(__ldg(row + i)) & 0x7fffffffu);
    }
  }
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0 && v != 0u) atomicMax(acc, (unsigned long long)v << 32);
}

// The residual f - (alpha x + beta L x) of a z-chunked single-patch 3-D level (same tiles,
// chunks, halo roles and prefetch distances as k_level_op3d_zc with R = 2), the planes staged
// as fixed-point integers.  fxs[0]: largest interior |x| (k_absmax_patch); fxs[1]: flag.
__global__ void __launch_bounds__(ZC_TX* ZC_TY, 2)
    k_resid3d_fx(LevelView lv, int ntx, int ntiles, int kc, const double* __restrict__ x, const double* __restrict__ f,
                 double* __restrict__ out, double alpha, double beta) {
  constexpr int R = 2;
  using G = ZcGeom<R>;
  pdl_wait();
  __shared__ long long sp[2][G::SH * ZC_W];
  // stacked component batches: the grid holds ncomp equal parts, part c on replica c with its
  // own frame and flag (fxs[2c], fxs[2c + 1])
  const int bpc = gridDim.x / lv.ncomp, comp = blockIdx.x / bpc, blk = blockIdx.x % bpc;
  if (lv.active != nullptr && !lv.active[comp]) return;  // converged replica of a stacked batch
  const PatchDesc p = lv.patches[comp];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * ZC_TX + tx;
  unsigned* __restrict__ flag = reinterpret_cast<unsigned*>(lv.fxs + 2 * comp + 1);
  const int emax = (int)((lv.fxs[2 * comp] >> 52) & 0x7ffull);
  if (emax == 0x7ff || (emax != 0 && emax < 53)) {  // non-finite, or a frame below the normal range
    if (tid == 0) *flag = 1u;
    return;
  }
  // beta / (12 h^2) 2^-S with S = 1075 - emax (an all-zero interior: every value rounds to 0)
  const double kT = emax == 0 ? 0.0 : beta * lv.inv12h2 * __longlong_as_double((long long)(emax - 52) << 52);
  bool ovf = false;
  const int sy = (int)p.sy, sz = (int)p.sz, nz = p.n[2];
  const int nzd = lv.ndom[2], lz = p.lo[2];
  const double* __restrict__ xb = x + p.off;
  const double* __restrict__ fb = f + p.off;
  double* __restrict__ ob = out + p.off;
  int hx = 0, hy = 0;
  const bool has_halo = tid < G::NH;
  {
    const int q = tid;
    if (q < 2 * ZC_TX) {
      hy = -2 + q / ZC_TX;
      hx = q % ZC_TX;
    } else if (q < 4 * ZC_TX) {
      hy = G::TH + (q - 2 * ZC_TX) / ZC_TX;
      hx = q % ZC_TX;
    } else if (q < G::NH) {
      const int r = q - 4 * ZC_TX, side = r / (2 * G::TH), c = r & 1;
      hy = (r % (2 * G::TH)) >> 1;
      hx = side == 0 ? c - 2 : ZC_TX + c;
    }
  }
  const int hs = (hy + 2) * ZC_W + hx + 2;
  const int c0 = (ty + 2) * ZC_W + tx + 2;
  const int tile = blk % ntiles, ka = (blk / ntiles) * kc, kb = min(nz, ka + kc);
  if (ka >= kb) return;
  const int i0 = (tile % ntx) * ZC_TX, j0 = (tile / ntx) * G::TH;
  const int i = i0 + tx;
  const int col0 = (i + NG) + (j0 + ty + NG) * sy;
  const int hli = i0 + hx, hlj = j0 + hy;
  const int hcol = (hli + NG) + (hlj + NG) * sy;
  int hsrc = 0, hstep = 0, htype = 0, hlayer = 0;
  {
    const int hgi = p.lo[0] + hli, hgj = p.lo[1] + hlj;
    const int d = (hgi < 0 || hgi >= lv.ndom[0]) ? 0 : ((hgj < 0 || hgj >= lv.ndom[1]) ? 1 : -1);
    if (has_halo && d >= 0) {
      const int g = d == 0 ? hgi : hgj, n = lv.ndom[d], side = g < 0 ? 0 : 1;
      hlayer = (side == 0 ? -g : g - n + 1) - 1;
      htype = lv.bc[2 * d + side];
      const int face = (side == 0 ? 0 : n - 1) - p.lo[d] - (d == 0 ? i0 : j0);
      hsrc = d == 0 ? (hy + 2) * ZC_W + face + 2 : (face + 2) * ZC_W + hx + 2;
      const int st = d == 0 ? 1 : ZC_W;
      hstep = side == 0 ? st : -st;
    }
  }
  const bool hload = has_halo && hstep == 0;
  const bool face_tile = p.lo[0] + i0 == 0 || p.lo[0] + i0 + ZC_TX == lv.ndom[0] || p.lo[1] + j0 == 0 ||
                         p.lo[1] + j0 + G::TH == lv.ndom[1];
  auto halo = [&](int k) -> double { return hload ? xb[hcol + (k + NG) * sz] : 0.0; };
  // frame headroom of the value of plane k (zc_zval): stored inside the domain, else the z
  // ghost formula
  auto zlim = [&](int k) -> int { return (lz + k >= 0 && lz + k < nzd) ? 2 : 7; };
  constexpr int RS = ZC_TY;
  long long q[R][5];  // x of each column at planes k-2..k+2, fixed point
  double xd[R][3];    // x at planes k..k+2 as stored (the alpha x term)
  double xs[2][R], fs[2][R], hv[2];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int col = col0 + r * RS * sy;
    double d[5];
    d[0] = zc_zval<double>(xb, col, sz, ka - 2, lz, nzd, lv);
    d[1] = zc_zval<double>(xb, col, sz, ka - 1, lz, nzd, lv);
    d[2] = xb[col + (ka + NG) * sz];
    d[3] = zc_zval<double>(xb, col, sz, ka + 1, lz, nzd, lv);
    d[4] = zc_zval<double>(xb, col, sz, ka + 2, lz, nzd, lv);
#pragma unroll
    for (int m = 0; m < 5; ++m) q[r][m] = fx_of(d[m], emax, zlim(ka - 2 + m), ovf);
    xd[r][0] = d[2];
    xd[r][1] = d[3];
    xd[r][2] = d[4];
    xs[0][r] = xs[1][r] = 0.0;
    if (ka + 1 < kb) xs[0][r] = zc_zval<double>(xb, col, sz, ka + 3, lz, nzd, lv);
    if (ka + 2 < kb) xs[1][r] = zc_zval<double>(xb, col, sz, ka + 4, lz, nzd, lv);
    fs[0][r] = fb[col + (ka + NG) * sz];
    fs[1][r] = (ka + 1 < kb) ? fb[col + (ka + 1 + NG) * sz] : 0.0;
  }
  hv[0] = hv[1] = 0.0;
  if (has_halo) {
    hv[0] = halo(ka);
    if (ka + 1 < kb) hv[1] = halo(ka + 1);
  }
  auto step = [&](int k, auto slot, auto safe) {
    constexpr int S = decltype(slot)::value;
    constexpr bool SAFE = decltype(safe)::value;  // planes up to k+5 inside the domain
    long long* __restrict__ s = sp[S];
    double fk[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      fk[r] = fs[S][r];
      s[c0 + r * RS * ZC_W] = q[r][2];
    }
    if (hload) {
      s[hs] = fx_of(hv[S], emax, 2, ovf);
      if (k + 2 < kb) hv[S] = halo(k + 2);
    }
    if (k + 2 < kb) {
#pragma unroll
      for (int r = 0; r < R; ++r) fs[S][r] = fb[col0 + r * RS * sy + (k + 2 + NG) * sz];
    }
    __syncthreads();
    if (face_tile) {
      // the ghost formula on the staged (fixed-point, so already scaled by 2^S) face cells: the
      // tile's own interior cells, whose integers are below 2^53 and convert exactly
      if (hstep != 0) {
        double v = 0.0;
#pragma unroll
        for (int m = 0; m < 4; ++m) v += gcoef<double>(htype, hlayer, m) * (double)s[hsrc + m * hstep];
        s[hs] = fx_of(v, 1075, 7, ovf);
      }
      __syncthreads();
    }
    const int pk = col0 + (k + NG) * sz;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int P = pk + r * RS * sy;
      const int C = c0 + r * RS * ZC_W;
      const long long s1 = ((s[C - 1] + s[C + 1]) + (s[C - ZC_W] + s[C + ZC_W])) + (q[r][1] + q[r][3]);
      const long long s2 = ((s[C - 2] + s[C + 2]) + (s[C - 2 * ZC_W] + s[C + 2 * ZC_W])) + (q[r][0] + q[r][4]);
      const long long T = s1 * 16 - s2 - q[r][2] * 90;
      ob[P] = fma(-kT, fx_to_double(T), alpha != 0.0 ? fma(-alpha, xd[r][0], fk[r]) : fk[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      q[r][0] = q[r][1];
      q[r][1] = q[r][2];
      q[r][2] = q[r][3];
      q[r][3] = q[r][4];
      q[r][4] = fx_of(xs[S][r], emax, zlim(k + 3), ovf);
      xd[r][0] = xd[r][1];
      xd[r][1] = xd[r][2];
      xd[r][2] = xs[S][r];
      if (k + 3 < kb) {  // q4 of plane k+3
        if (SAFE) xs[S][r] = xb[col0 + r * RS * sy + (k + 5 + NG) * sz];
        else xs[S][r] = zc_zval<double>(xb, col0 + r * RS * sy, sz, k + 5, lz, nzd, lv);
      }
    }
  };
  for (int k = ka; k < kb; k += 2) {
    if (lz + k + 6 < nzd) {
      step(k, zc_slot<0>{}, std::true_type{});
      if (k + 1 < kb) step(k + 1, zc_slot<1>{}, std::true_type{});
    } else {
      step(k, zc_slot<0>{}, std::false_type{});
      if (k + 1 < kb) step(k + 1, zc_slot<1>{}, std::false_type{});
    }
  }
  if (ovf) *flag = 1u;
}

// ------------------------------------------------------------------------ G and D
// grad: out_d = (-x_{+2} + 8 x_{+1} - 8 x_{-1} + x_{-2}) / (12 h)   (Eq. discreteOps a)
template <typename T, int D>
__global__ void k_gradient(LevelView lv, int nby, const T* __restrict__ x, T* __restrict__ g0, T* __restrict__ g1,
                           T* __restrict__ g2, const T* __restrict__ bc) {
  pdl_wait();
  const PatchDesc p = lv.patches[blockIdx.z];
  int i, j, k;
  if (!thread_cell<D>(p, nby, i, j, k)) return;
  const long long o = poff(p, i, j, k);
  const T inv = pick<T>(lv.inv12h, lv.inv12h_f);
  T* outs[3] = {g0, g1, g2};
  const int c[3] = {i, j, k};
#pragma unroll
  for (int d = 0; d < D; ++d) {
    int cc[3] = {i, j, k};
    cc[d] = c[d] - 1; const T m1 = read_nb<T, D>(x, p, lv, bc, cc[0], cc[1], cc[2], d);
    cc[d] = c[d] + 1; const T p1 = read_nb<T, D>(x, p, lv, bc, cc[0], cc[1], cc[2], d);
    cc[d] = c[d] - 2; const T m2 = read_nb<T, D>(x, p, lv, bc, cc[0], cc[1], cc[2], d);
    cc[d] = c[d] + 2; const T p2 = read_nb<T, D>(x, p, lv, bc, cc[0], cc[1], cc[2], d);
    outs[d][o] = (T(8) * (p1 - m1) - (p2 - m2)) * inv;
  }
}

struct Ptr3 {
  const double* p[3];
};
struct Ptr3m {
  double* p[3];
};

// div: sum_d (-u_{+2} + 8 u_{+1} - 8 u_{-1} + u_{-2}) / (12 h)   (Eq. discreteOps b)
template <int D>
__global__ void k_divergence(LevelView lv, int nby, Ptr3 u, double* __restrict__ out, Ptr3 bc) {
  pdl_wait();
  const PatchDesc p = lv.patches[blockIdx.z];
  int i, j, k;
  if (!thread_cell<D>(p, nby, i, j, k)) return;
  const long long o = poff(p, i, j, k);
  const double inv = lv.inv12h;
  const int c[3] = {i, j, k};
  double acc = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const double* x = u.p[d];
    int cc[3] = {i, j, k};
    cc[d] = c[d] - 1; const double m1 = read_nb<double, D>(x, p, lv, bc.p[d], cc[0], cc[1], cc[2], d);
    cc[d] = c[d] + 1; const double p1 = read_nb<double, D>(x, p, lv, bc.p[d], cc[0], cc[1], cc[2], d);
    cc[d] = c[d] - 2; const double m2 = read_nb<double, D>(x, p, lv, bc.p[d], cc[0], cc[1], cc[2], d);
    cc[d] = c[d] + 2; const double p2 = read_nb<double, D>(x, p, lv, bc.p[d], cc[0], cc[1], cc[2], d);
    acc += 8.0 * (p1 - m1) - (p2 - m2);
  }
  out[o] = acc * inv;
}

// ------------------------------------------------------------------------ AMRCFI / copy
template <typename T, int D>
__global__ void k_cfi(const CfiEntry* __restrict__ list, long long n, const long long* __restrict__ side,
                      const PatchDesc* __restrict__ cpatches, int r, const T* __restrict__ xc, T* __restrict__ xf,
                      int zero) {
  pdl_wait();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const CfiEntry e = list[t];
  if (zero) {
    xf[e.dst] = T(0);
    return;
  }
  const int b0 = (e.pos[0] * r + e.sub[0]) * CFI_W;
  const int b1 = (e.pos[1] * r + e.sub[1]) * CFI_W;
  const int b2 = (e.pos[2] * r + e.sub[2]) * CFI_W;
  T v = T(0);
  if (e.src >= 0) {
    const PatchDesc cp = cpatches[e.cpatch];
    for (int c2 = 0; c2 < (D == 3 ? CFI_W : 1); ++c2)
      for (int c1 = 0; c1 < CFI_W; ++c1) {
        const long long row = e.src + (long long)c1 * cp.sy + (long long)c2 * cp.sz;
        const T wr = cfiw<T>(b1 + c1) * (D == 3 ? cfiw<T>(b2 + c2) : T(1));
#pragma unroll
        for (int c0 = 0; c0 < CFI_W; ++c0) v += cfiw<T>(b0 + c0) * wr * xc[row + c0];
      }
  } else {
    const long long* s = side + (-1 - e.src) * (D == 3 ? 125 : 25);
    int q = 0;
    for (int c2 = 0; c2 < (D == 3 ? CFI_W : 1); ++c2)
      for (int c1 = 0; c1 < CFI_W; ++c1)
        for (int c0 = 0; c0 < CFI_W; ++c0, ++q)
          v += cfiw<T>(b0 + c0) * cfiw<T>(b1 + c1) * (D == 3 ? cfiw<T>(b2 + c2) : T(1)) * xc[s[q]];
  }
  xf[e.dst] = v;
}

// AMRCFI by coarse parent: one thread evaluates the 2^D children of one parent (the tensor
// product of the 1-D quartic weights of Sec. 4 over the shared 5^D window) dimension by
// dimension: per window row the two x sums (one per child column), folded into the two y
// sums per child row, then into the two z sums: 2 5^D + 4 5^(D-1) + 8 5^(D-2) multiply-adds
// for 2^D ghosts, instead of 2^D 5^D products and sums.
template <typename T, int D>
__global__ void k_cfi_grp(const CfiGroup* __restrict__ list, long long n, const long long* __restrict__ side,
                          const PatchDesc* __restrict__ cpatches, const T* __restrict__ xc, T* __restrict__ xf,
                          int zero) {
  pdl_wait();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const CfiGroup& g = list[t];
  constexpr int NC = D == 3 ? 8 : 4;
  if (zero) {
#pragma unroll
    for (int c = 0; c < NC; ++c)
      if (g.dst[c] >= 0) xf[g.dst[c]] = T(0);
    return;
  }
  // weight of window cell w for child sub-position a (ratio 2): cfiw((2 pos + a) W + w)
  const int b0 = 2 * g.pos[0] * CFI_W, b1 = 2 * g.pos[1] * CFI_W, b2 = 2 * g.pos[2] * CFI_W;
  const long long src = g.src;
  PatchDesc cp{};
  if (src >= 0) cp = cpatches[g.cpatch];
  const long long* s = src >= 0 ? nullptr : side + (-1 - src) * (D == 3 ? 125 : 25);
  T acc[2][2][2];
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c & 1][(c >> 1) & 1][c >> 2] = T(0);
  for (int c2 = 0; c2 < (D == 3 ? CFI_W : 1); ++c2) {
    T by[2][2] = {{T(0), T(0)}, {T(0), T(0)}};  // [x child][y child]
    for (int c1 = 0; c1 < CFI_W; ++c1) {
      T v[CFI_W];
      if (s == nullptr) {
        const long long row = src + (long long)c1 * cp.sy + (long long)c2 * cp.sz;
#pragma unroll
        for (int c0 = 0; c0 < CFI_W; ++c0) v[c0] = xc[row + c0];
      } else {
#pragma unroll
        for (int c0 = 0; c0 < CFI_W; ++c0) v[c0] = xc[s[(c2 * CFI_W + c1) * CFI_W + c0]];
      }
      T bx[2] = {T(0), T(0)};
#pragma unroll
      for (int c0 = 0; c0 < CFI_W; ++c0) {
        bx[0] += cfiw<T>(b0 + c0) * v[c0];
        bx[1] += cfiw<T>(b0 + CFI_W + c0) * v[c0];
      }
      const T wy0 = cfiw<T>(b1 + c1), wy1 = cfiw<T>(b1 + CFI_W + c1);
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        by[a][0] += wy0 * bx[a];
        by[a][1] += wy1 * bx[a];
      }
    }
    if (D == 3) {
      const T wz0 = cfiw<T>(b2 + c2), wz1 = cfiw<T>(b2 + CFI_W + c2);
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          acc[a][b][0] += wz0 * by[a][b];
          acc[a][b][1] += wz1 * by[a][b];
        }
    } else {
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) acc[a][b][0] = by[a][b];
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (g.dst[c] >= 0) xf[g.dst[c]] = acc[c & 1][(c >> 1) & 1][c >> 2];
}

// AMRCFI of face rectangles (CfiTile), one block per rectangle: the window columns fold along
// the face normal (both children), the folded plane along the first tangential dimension, then
// along the second.  The first two folds serve every parent whose window holds the column, so a
// parent costs about 92 multiply-adds instead of 390 by itself; in FP64 their rate bounds the
// pass (interface conditions of a 128^3 box, three components: 197 -> 74 us a call).  NS = 1: one field; NS = 4: the fields at four times, each window cell combined by two
// rows of weights first (value and time derivative; AMRCFI and the combination are linear).  The
// derivative's weights cancel: combined after the normal fold, at four multiply-adds fewer of 60, the
// folds' rounding came through with 2.5 times the error on fields that change little in time.
template <typename T, int NS>
struct CfiSource {
  const T* x[NS];
  T w[2][NS];  // NS = 4: weights of the value and of the derivative
};

template <typename T, int NS>
__global__ void __launch_bounds__(128) k_cfi_tile(const CfiTile* __restrict__ tiles, CfiSource<T, NS> s, T* out0, T* out1) {
  constexpr int NR = NS == 1 ? 1 : 2, M = CFI_TILE + CFI_W - 1;
  __shared__ T fa[NR][2][M][M + 1];            // [row][normal child][second][first tangential column]
  __shared__ T fb[NR][2][M][2 * CFI_TILE];     // folded along the first tangential dimension
  pdl_wait();
  const CfiTile t = tiles[blockIdx.x];
  const int tid = threadIdx.x;
  const int m1 = t.n1 + CFI_W - 1, m2 = t.n2 + CFI_W - 1;
  const int nr = (NS == 1 || out1 == nullptr) ? 1 : 2;
  const int bn = 2 * t.posn * CFI_W, bt = 4 * CFI_W;  // weights of the normal window; of a centred one
  for (int q = tid; q < m1 * m2; q += 128) {
    const int j1 = q % m1, j2 = q / m1;
    const long long o = t.src + (long long)j1 * t.s1 + (long long)j2 * t.s2;
    T v[NS][CFI_W], f[NR][2];
#pragma unroll
    for (int i = 0; i < NS; ++i)
#pragma unroll
      for (int c = 0; c < CFI_W; ++c) v[i][c] = s.x[i][o + (long long)c * t.sn];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      f[r][0] = f[r][1] = T(0);
#pragma unroll
      for (int c = 0; c < CFI_W; ++c) {
        T y = v[0][c];
        if (NS > 1) {
          y = s.w[r][0] * v[0][c];
#pragma unroll
          for (int i = 1; i < NS; ++i) y += s.w[r][i] * v[i][c];
        }
        f[r][0] += cfiw<T>(bn + c) * y;
        f[r][1] += cfiw<T>(bn + CFI_W + c) * y;
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int r = 0; r < NR; ++r) fa[r][h][j2][j1] = f[r][h];
  }
  __syncthreads();
  const int w1 = 2 * t.n1, w2 = 2 * t.n2;
  for (int q = tid; q < w1 * m2 * 2 * nr; q += 128) {
    const int o1 = q % w1, u = q / w1, j2 = u % m2, hr = u / m2, h = hr & 1, r = hr >> 1;
    const T* __restrict__ a = &fa[r][h][j2][o1 >> 1];
    const int b = bt + (o1 & 1) * CFI_W;
    T v = T(0);
#pragma unroll
    for (int c = 0; c < CFI_W; ++c) v += cfiw<T>(b + c) * a[c];
    fb[r][h][j2][o1] = v;
  }
  __syncthreads();
  for (int q = tid; q < w1 * w2 * 2 * nr; q += 128) {
    const int o1 = q % w1, u = q / w1, o2 = u % w2, hr = u / w2, h = hr & 1, r = hr >> 1;
    if (!((t.mask >> ((o1 >> 1) + CFI_TILE * (o2 >> 1))) & 1ull)) continue;
    const int b = bt + (o2 & 1) * CFI_W;
    T v = T(0);
#pragma unroll
    for (int c = 0; c < CFI_W; ++c) v += cfiw<T>(b + c) * fb[r][h][(o2 >> 1) + c][o1];
    (r == 0 ? out0 : out1)[t.dst + (long long)h * t.fn + (long long)o1 * t.f1 + (long long)o2 * t.f2] = v;
  }
}

template <typename T>
__global__ void k_copy(const CopyEntry* __restrict__ list, long long n, T* __restrict__ x) {
  pdl_wait();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const CopyEntry e = list[t];
  x[e.dst] = x[e.src];
}

// ------------------------------------------------------------------------ transfers
// Coarse cell g gets the mean of its r^D children (r = 2): of x (average-down,
// Eq. AMR_avergingDownToCrse / restriction), or of f - A x on the fine level (residual
// restriction) when RESID.
template <typename T, int D, bool RESID, bool TR = false>
__device__ __forceinline__ void cell_restrict(const LevelView& fine, const PatchDesc& fp, const PatchDesc& cp,
                                              const int g[3], const T* __restrict__ xf, const T* __restrict__ ff,
                                              T* __restrict__ outc, T alpha, T beta) {
  T acc = T(0);
  const T inv = pick<T>(fine.inv12h2, fine.inv12h2_f);
  for (int q2 = 0; q2 < (D == 3 ? 2 : 1); ++q2)
    for (int q1 = 0; q1 < 2; ++q1)
      for (int q0 = 0; q0 < 2; ++q0) {
        const int fi = 2 * g[0] + q0 - fp.lo[0];
        const int fj = 2 * g[1] + q1 - fp.lo[1];
        const int fk = (D == 3) ? 2 * g[2] + q2 - fp.lo[2] : 0;
        const long long o = poff(fp, fi, fj, fk);
        if (!RESID) {
          acc += xf[o];
        } else {
          const T xc = xf[o];
          const T s = cell_Lx<T, D, TR>(fine, fp, fi, fj, fk, xf, (const T*)nullptr);
          acc += ff[o] - (alpha * xc + beta * (s * inv));
        }
      }
  outc[poff(cp, g[0] - cp.lo[0], g[1] - cp.lo[1], g[2] - cp.lo[2])] = acc * T(D == 3 ? 0.125 : 0.25);
}

template <typename T, int D, bool RESID, bool TR = false>
__global__ void k_restrict(LevelView fine, LevelView crs, const XferBlock* __restrict__ blocks,
                           const T* __restrict__ xf, const T* __restrict__ ff, T* __restrict__ outc,
                           T alpha, T beta, int nby) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int i = blockIdx.x * BX + threadIdx.x;
  const int by = (D == 3) ? (int)(blockIdx.y % nby) : (int)blockIdx.y;
  const int kk = (D == 3) ? (int)(blockIdx.y / nby) : 0;
  const int j = by * BY + threadIdx.y;
  const int g[3] = {b.clo[0] + i, b.clo[1] + j, b.clo[2] + kk};
  if (g[0] > b.chi[0] || g[1] > b.chi[1] || g[2] > b.chi[2]) return;
  cell_restrict<T, D, RESID, TR>(fine, fine.patches[b.fpatch], crs.patches[b.cpatch], g, xf, ff, outc, alpha, beta);
}

// 2-D residual restriction, one lane per fine cell: a warp takes 16 columns of two fine rows, each
// lane the residual of its cell (the sums of edge_op2d next to the faces), and the four children
// of a coarse cell are added by shuffle in cell_restrict's order.  A thread per coarse cell, its
// block in generic code wherever it touched a face, took 11 us per FP64 pass at 128^2.
template <typename T, bool TR>
__global__ void __launch_bounds__(BX* BY) k_restrict2d_resid(LevelView fine, LevelView crs,
                                                             const XferBlock* __restrict__ blocks,
                                                             const T* __restrict__ xf, const T* __restrict__ ff,
                                                             T* __restrict__ outc, T alpha, T beta) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int lane = threadIdx.x;
  const int f0 = 2 * b.clo[0] + blockIdx.x * 16 + (lane & 15);
  const int f1 = 2 * (b.clo[1] + (int)(blockIdx.y * BY + threadIdx.y)) + (lane >> 4);
  const int g0 = f0 >> 1, g1 = f1 >> 1;
  const bool on = g0 <= b.chi[0] && g1 <= b.chi[1];
  const PatchDesc cp = crs.patches[b.cpatch];
  const PatchDesc fp = fine.patches[b.fpatch];
  T r = T(0);
  if (on) {
    const int sy = (int)fp.sy, i = f0 - fp.lo[0], j = f1 - fp.lo[1], o = (j + NG) * sy + i + NG;
    const T* __restrict__ xb = xf + fp.off;
    const T xc = xb[o], fk = ff[fp.off + o];
    T x1, x2, y1, y2, ex = T(0);
    if (TR) {
      if (f0 >= 4 && f0 <= fine.ndom[0] - 5) {
        x1 = xb[o - 1] + xb[o + 1];
        x2 = xb[o - 2] + xb[o + 2];
      } else {
        trans_sums<T>(xb, o, 1, i, fine.ndom[0], fp.lo[0], fp.n[0], fine.bc[0], fine.bc[1], x1, x2, ex);
      }
      if (f1 >= 4 && f1 <= fine.ndom[1] - 5) {
        y1 = xb[o - sy] + xb[o + sy];
        y2 = xb[o - 2 * sy] + xb[o + 2 * sy];
      } else {
        trans_sums<T>(xb, o, sy, j, fine.ndom[1], fp.lo[1], fp.n[1], fine.bc[2], fine.bc[3], y1, y2, ex);
      }
    } else {
      line_sums<T>(xb, o, 1, face_class(f0, fine.ndom[0]) == 0, f0, fine.ndom[0], fine.bc[0], fine.bc[1], x1, x2);
      line_sums<T>(xb, o, sy, face_class(f1, fine.ndom[1]) == 0, f1, fine.ndom[1], fine.bc[2], fine.bc[3], y1, y2);
    }
    const T s1 = x1 + y1, s2 = x2 + y2;
    const T inv = pick<T>(fine.inv12h2, fine.inv12h2_f);
    r = fk - (alpha * xc + beta * (((T(16) * s1 - s2 - T(60) * xc) + ex) * inv));
  }
  const int q = lane & 14;
  T acc = __shfl_sync(0xffffffffu, r, q);
  acc += __shfl_sync(0xffffffffu, r, q + 1);
  acc += __shfl_sync(0xffffffffu, r, q + 16);
  acc += __shfl_sync(0xffffffffu, r, q + 17);
  if (on && lane == q) outc[poff(cp, g0 - cp.lo[0], g1 - cp.lo[1], 0)] = acc * T(0.25);
}

// Fine cell gf += cell-centred tensor linear interpolation of the coarse correction
// (Sec. 6.5 "linear interpolation"; weights 3/4, 1/4 per dimension).  Coarse values outside
// the domain come from the homogeneous physical extension with corners.
template <typename T, int D>
__device__ __forceinline__ void cell_prolong(const LevelView& crs, const PatchDesc& fp, const PatchDesc& cp,
                                             const int gf[3], const T* __restrict__ xc, T* __restrict__ xf,
                                             T* __restrict__ xf2) {
  int par[3], sg[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    par[e] = (e < D) ? (gf[e] >> 1) : 0;
    sg[e] = (e < D) ? (((gf[e] & 1) == 0) ? -1 : 1) : 0;
  }
  T v = T(0);
  for (int q2 = 0; q2 < (D == 3 ? 2 : 1); ++q2)
    for (int q1 = 0; q1 < 2; ++q1)
      for (int q0 = 0; q0 < 2; ++q0) {
        const int q[3] = {q0, q1, q2};
        int cc[3];
        T w = T(1);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          cc[e] = par[e] + q[e] * sg[e] - cp.lo[e];
          if (e < D) w *= (q[e] == 0) ? T(0.75) : T(0.25);
        }
        bool inside = true;
#pragma unroll
        for (int e = 0; e < D; ++e) {
          const int g = cp.lo[e] + cc[e];
          inside = inside && g >= 0 && g < crs.ndom[e];
        }
        const T cv = inside ? xc[poff(cp, cc[0], cc[1], cc[2])] : read_ext<T, D>(xc, cp, crs, cc[0], cc[1], cc[2]);
        v += w * cv;
      }
  const long long o = poff(fp, gf[0] - fp.lo[0], gf[1] - fp.lo[1], gf[2] - fp.lo[2]);
  xf[o] += v;
  if (xf2 != nullptr) xf2[o] += v;
}

template <typename T, int D>
__global__ void k_prolong(LevelView fine, LevelView crs, const XferBlock* __restrict__ blocks,
                          const T* __restrict__ xc, T* __restrict__ xf, T* __restrict__ xf2, int nby) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int i = blockIdx.x * BX + threadIdx.x;  // fine offsets inside the block region
  const int by = (D == 3) ? (int)(blockIdx.y % nby) : (int)blockIdx.y;
  const int kk = (D == 3) ? (int)(blockIdx.y / nby) : 0;
  const int j = by * BY + threadIdx.y;
  const int gf[3] = {2 * b.clo[0] + i, 2 * b.clo[1] + j, D == 3 ? 2 * b.clo[2] + kk : 0};
  if (gf[0] > 2 * b.chi[0] + 1 || gf[1] > 2 * b.chi[1] + 1 || (D == 3 && gf[2] > 2 * b.chi[2] + 1)) return;
  cell_prolong<T, D>(crs, fine.patches[b.fpatch], crs.patches[b.cpatch], gf, xc, xf, xf2);
}

// 2-D prolongation, one thread per fine cell: linear interpolation from its four coarse corners
// (32-bit offsets) when they lie inside the domain and the patch, generic code otherwise (same
// arithmetic).  The grids are small, so the pass lasts as long as one thread next to a face: with
// a thread per coarse cell, four generic children in turn, an FP64 pass took 14 us at 128^2.
template <typename T>
__global__ void __launch_bounds__(BX* BY) k_prolong2d(LevelView fine, LevelView crs, const XferBlock* __restrict__ blocks,
                                                      const T* __restrict__ xc, T* __restrict__ xf, T* __restrict__ xf2) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int f0 = 2 * b.clo[0] + blockIdx.x * BX + threadIdx.x, f1 = 2 * b.clo[1] + blockIdx.y * BY + threadIdx.y;
  const int g0 = f0 >> 1, g1 = f1 >> 1;
  if (g0 > b.chi[0] || g1 > b.chi[1]) return;
  const PatchDesc cp = crs.patches[b.cpatch];
  const PatchDesc fp = fine.patches[b.fpatch];
  const int s0 = (f0 & 1) ? 1 : -1, s1 = (f1 & 1) ? 1 : -1;
  const int e0 = g0 + s0 - cp.lo[0], e1 = g1 + s1 - cp.lo[1];
  if (e0 < 0 || e0 >= cp.n[0] || e1 < 0 || e1 >= cp.n[1]) {
    const int gf[3] = {f0, f1, 0};
    cell_prolong<T, 2>(crs, fp, cp, gf, xc, xf, xf2);
    return;
  }
  const int csy = (int)cp.sy;
  const T* __restrict__ c = xc + cp.off + (g1 - cp.lo[1] + NG) * csy + (g0 - cp.lo[0] + NG);
  // corners in the generic order: (q0, q1) = (0,0), (1,0), (0,1), (1,1) over the parent
  T v = T(0);
  v += (T(0.75) * T(0.75)) * c[0];
  v += (T(0.25) * T(0.75)) * c[s0];
  v += (T(0.75) * T(0.25)) * c[s1 * csy];
  v += (T(0.25) * T(0.25)) * c[s1 * csy + s0];
  const long long o = fp.off + (long long)((f1 - fp.lo[1] + NG) * (int)fp.sy + (f0 - fp.lo[0] + NG));
  xf[o] += v;
  if (xf2 != nullptr) xf2[o] += v;
}

// ------------------------------------------------------------------------ temporally blocked 2-D smoothing
// One block owns a tile of a single-patch 2-D multigrid grid (the patch is the whole
// domain) and keeps a region -- the tile plus a halo, clipped to the domain -- in shared
// memory, laid out with two ghost layers like the global patch.  Before every sweep the
// physical ghost layers of the domain faces the region touches are materialised from the
// current iterate (homogeneous Eqs. velBCHomoDiri5th / Neumann5), so that every cell runs
// the same interior stencil; only the Jacobi diagonal differs within two cells of a face
// (the ghost formulas put weight back on the cell itself).  Sweep s (from 1) updates the
// region shrunk by 2 s on every side that is not a domain face; that region never reads
// past what sweep s-1 produced, so no value from outside the region is ever used, and the
// halo (2 nu, plus 2 for a residual) keeps the shrinkage out of the tile.
struct TileGeom {
  int i0, j0;      // tile origin (patch-local)
  int tw, th;      // tile extents
  int r0, r1;      // region origin (patch-local)
  int rw, rh;      // region extents
  int fl0, fh0, fl1, fh1;  // 1 where the region side is a patch edge (closed: does not shrink)
  int pl0, ph0, pl1, ph1;  // 1 where that edge is a domain face (physical ghosts; else a CF
                           // edge whose ghosts are zero in correction smoothing)
  int g0, g1;              // global index of the region's first cell
};

__device__ __forceinline__ TileGeom tile_geom(const PatchDesc& gp, const LevelView& lv, int tx, int ty, int halo) {
  TileGeom t;
  t.i0 = blockIdx.x * tx;
  t.j0 = blockIdx.y * ty;
  t.tw = min(tx, gp.n[0] - t.i0);
  t.th = min(ty, gp.n[1] - t.j0);
  t.r0 = max(t.i0 - halo, 0);
  t.r1 = max(t.j0 - halo, 0);
  const int e0 = min(t.i0 + t.tw + halo, gp.n[0]);
  const int e1 = min(t.j0 + t.th + halo, gp.n[1]);
  t.rw = e0 - t.r0;
  t.rh = e1 - t.r1;
  t.fl0 = t.r0 == 0;
  t.fl1 = t.r1 == 0;
  t.fh0 = e0 == gp.n[0];
  t.fh1 = e1 == gp.n[1];
  t.pl0 = t.fl0 && gp.lo[0] == 0;
  t.pl1 = t.fl1 && gp.lo[1] == 0;
  t.ph0 = t.fh0 && gp.lo[0] + gp.n[0] == lv.ndom[0];
  t.ph1 = t.fh1 && gp.lo[1] + gp.n[1] == lv.ndom[1];
  t.g0 = gp.lo[0] + t.r0;
  t.g1 = gp.lo[1] + t.r1;
  return t;
}

// region cells updated by sweep s (shrunk by 2 s on the open sides)
__device__ __forceinline__ void sweep_box(const TileGeom& t, int s, int& a0, int& b0, int& a1, int& b1) {
  a0 = t.fl0 ? 0 : 2 * s;
  b0 = t.fh0 ? t.rw : t.rw - 2 * s;
  a1 = t.fl1 ? 0 : 2 * s;
  b1 = t.fh1 ? t.rh : t.rh - 2 * s;
}

__device__ __forceinline__ int blk_tid() { return (int)(threadIdx.y * blockDim.x + threadIdx.x); }
__device__ __forceinline__ int blk_nth() { return (int)(blockDim.x * blockDim.y); }

// The threads that work on a region: the whole block (rows of 32 threads, __syncthreads), or
// its first nth threads (whole warps) synchronised by named barrier 1, so that a small grid
// keeps only the warps it needs busy while the others wait at the block's next barrier.
struct Team {
  int tid, nth;   // linear id and size
  int tx, ty;     // position in rows of 32
  int nty;        // rows
  bool named;
  __device__ __forceinline__ void sync() const {
    if (named) asm volatile("bar.sync 1, %0;" ::"r"(nth) : "memory");
    else __syncthreads();
  }
};
__device__ __forceinline__ Team block_team() {  // blockDim.x == 32
  Team t;
  t.tid = blk_tid();
  t.nth = blk_nth();
  t.tx = (int)threadIdx.x;
  t.ty = (int)threadIdx.y;
  t.nty = (int)blockDim.y;
  t.named = false;
  return t;
}
__device__ __forceinline__ Team sub_team(int cells) {  // enough whole warps for ``cells``
  Team t;
  t.tid = blk_tid();
  t.nth = min(blk_nth(), (cells + 31) / 32 * 32);
  t.tx = t.tid & 31;
  t.ty = t.tid >> 5;
  t.nty = t.nth >> 5;
  t.named = t.nth < blk_nth();
  return t;
}

// Physical ghost layers of the region's domain faces for rows [a1,b1) / columns [a0,b0)
// (only blocks whose region touches a face do any work here).
template <typename T>
__device__ __forceinline__ void region_ghosts(const LevelView& lv, const TileGeom& tg, T* __restrict__ a, int sy, int a0,
                                              int b0, int a1, int b1, const Team& tm) {
  if (!(tg.fl0 | tg.fh0 | tg.fl1 | tg.fh1)) return;
  const int tid = tm.tid, nth = tm.nth;
  const int nr = b1 - a1, nc = b0 - a0;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    if (side == 0 ? tg.fl0 : tg.fh0) {
      const bool phys = side == 0 ? tg.pl0 : tg.ph0;
      const int type = lv.bc[side];
      for (int q = tid; q < 2 * nr; q += nth) {
        const int layer = q & 1, j = a1 + (q >> 1);
        const int row = (j + NG) * sy + NG;
        T v = T(0);
        if (phys) {
#pragma unroll
          for (int m = 0; m < 4; ++m) v += gcoef<T>(type, layer, m) * a[row + (side == 0 ? m : tg.rw - 1 - m)];
        }
        a[row + (side == 0 ? -1 - layer : tg.rw + layer)] = v;
      }
    }
    if (side == 0 ? tg.fl1 : tg.fh1) {
      const bool phys = side == 0 ? tg.pl1 : tg.ph1;
      const int type = lv.bc[2 + side];
      for (int q = tid; q < 2 * nc; q += nth) {
        const int layer = q & 1, col = NG + a0 + (q >> 1);
        T v = T(0);
        if (phys) {
#pragma unroll
          for (int m = 0; m < 4; ++m) v += gcoef<T>(type, layer, m) * a[(NG + (side == 0 ? m : tg.rh - 1 - m)) * sy + col];
        }
        a[(NG + (side == 0 ? -1 - layer : tg.rh + layer)) * sy + col] = v;
      }
    }
  }
}

// Weighted-Jacobi factors omega / diag of a region, table driven: the diagonal differs from
// the interior one only within two cells of a domain face (the ghost formulas put weight back
// on the cell itself), so a cell's factor is wt[kx[i] + 5 ky[j]] with kx, ky in 0..4 (0:
// interior, 1, 2: first, second cell from the low face, 3, 4: from the high face).
constexpr int BLK_MAX_REGION = 64;
struct JacobiTable {
  float wf[25];
  double wd[25];
  unsigned char kx[BLK_MAX_REGION], ky[BLK_MAX_REGION];
};

template <typename T>
__device__ __forceinline__ T jt_get(const JacobiTable& t, int k);
template <>
__device__ __forceinline__ float jt_get<float>(const JacobiTable& t, int k) { return t.wf[k]; }
template <>
__device__ __forceinline__ double jt_get<double>(const JacobiTable& t, int k) { return t.wd[k]; }


template <typename T>
__device__ __forceinline__ void build_jacobi_table(JacobiTable& jt, const LevelView& lv, const TileGeom& tg, T alpha,
                                                   T beta, T omega, T ood, const Team& tm) {
  const T inv = pick<T>(lv.inv12h2, lv.inv12h2_f);
  const int tid = tm.tid, nth = tm.nth;
  for (int q = tid; q < 25; q += nth) {
    const int a = q % 5, b = q / 5;
    // diag_sum's order: -30 D, then the x correction, then the y correction
    const T cx = a == 0 ? T(0) : pick<T>(lv.dcorr[(a - 1) / 2][(a - 1) % 2], lv.dcorr_f[(a - 1) / 2][(a - 1) % 2]);
    const T cy = b == 0 ? T(0) : pick<T>(lv.dcorr[2 + (b - 1) / 2][(b - 1) % 2], lv.dcorr_f[2 + (b - 1) / 2][(b - 1) % 2]);
    const T w = q == 0 ? ood : omega / (alpha + beta * inv * ((T(-60) + cx) + cy));
    if (sizeof(T) == 4) jt.wf[q] = (float)w;
    else jt.wd[q] = (double)w;
  }
  for (int q = tid; q < tg.rw; q += nth) jt.kx[q] = (unsigned char)face_class(tg.g0 + q, lv.ndom[0]);
  for (int q = tid; q < tg.rh; q += nth) jt.ky[q] = (unsigned char)face_class(tg.g1 + q, lv.ndom[1]);
}

// 12 h^2 L x at smem offset o (interior stencil; ghosts materialised), cell_Lx's order
template <typename T>
__device__ __forceinline__ T lap_smem(const T* __restrict__ a, int o, int sy) {
  const T xc = a[o];
  const T s1 = (a[o - 1] + a[o + 1]) + (a[o - sy] + a[o + sy]);
  const T s2 = (a[o - 2] + a[o + 2]) + (a[o - 2 * sy] + a[o + 2 * sy]);
  return (T(16) * s1 - s2 - T(60) * xc) + T(0);
}

// f - (alpha x + beta L x) at smem offset o: kc0 = alpha - 60 kc2, kc1 = 16 kc2, kc2 = beta /
// (12 h^2); the operations of the streamed legs (stream2d.cuh), so that a leg's result does not
// depend on which of the two forms runs it
template <typename T>
__device__ __forceinline__ T resid_smem(const T* __restrict__ a, int o, int sy, T f, T kc0, T kc1, T kc2) {
  const T s1 = (a[o - 1] + a[o + 1]) + (a[o - sy] + a[o + sy]);
  const T s2 = (a[o - 2] + a[o + 2]) + (a[o - 2 * sy] + a[o + 2 * sy]);
  return fma(kc2, s2, fma(-kc1, s1, fma(-kc0, a[o], f)));
}

// f(i, j) for every cell of a w x h box of a block (rows of 32 threads, NT in all).  RM = 0: rows of 32
// threads stride over the box; RM > 0 (w, h <= RM, a compile-time bound): one linear pass
// over RM x RM positions with a fixed trip count, positions outside the box skipped.
template <int RM, int NT = 256, typename F>
__device__ __forceinline__ void for_cells(int w, int h, F&& f) {
  if constexpr (RM == 0) {
    for (int j = (int)threadIdx.y; j < h; j += (int)blockDim.y)
      for (int i = (int)threadIdx.x; i < w; i += (int)blockDim.x) f(i, j);
  } else {
    constexpr int NC = RM * RM, IT = (NC + NT - 1) / NT;
    const int tid = (int)(threadIdx.x + 32 * threadIdx.y);
#pragma unroll 2
    for (int k = 0; k < IT; ++k) {
      const int c = tid + NT * k;
      if (NC % NT == 0 || c < NC) {
        const int i = c % RM, j = c / RM;
        if (i < w && j < h) f(i, j);
      }
    }
  }
}

// nu weighted-Jacobi sweeps on the region; returns the buffer holding the result.  RM > 0:
// the region is at most RM x RM (a compile-time bound, shared-memory pitch sy = RM + 4), cell
// loops have fixed trip counts, and blocks whose region touches no domain face skip the
// ghost pass and its barrier.
template <typename T, bool ZERO, int RM = 0, int NT = 256>
__device__ __forceinline__ T* smooth_region(const LevelView& lv, const TileGeom& tg, const JacobiTable& jt, int sy,
                                            T* cur, T* oth, const T* __restrict__ sb, int nu, T alpha, T beta,
                                            const Team& tm) {
  const T kc2 = beta * pick<T>(lv.inv12h2, lv.inv12h2_f), kc1 = T(16) * kc2, kc0 = fma(T(-60), kc2, alpha);
  if constexpr (RM > 0) {
    constexpr int SY = RM + 2 * NG;
    const bool face = tg.fl0 | tg.fh0 | tg.fl1 | tg.fh1;
    for (int s = 1; s <= nu; ++s) {
      int a0, b0, a1, b1;
      sweep_box(tg, s, a0, b0, a1, b1);
      const bool zero = ZERO && s == 1;
      if (!zero && face) {
        int c0, d0, c1, d1;
        sweep_box(tg, s - 1, c0, d0, c1, d1);
        region_ghosts(lv, tg, cur, SY, c0, d0, c1, d1, tm);
        __syncthreads();
      }
      for_cells<RM, NT>(b0, b1, [&](int i, int j) {
        if (i < a0 || j < a1) return;
        const int o = (j + NG) * SY + (i + NG);
        const T w = jt_get<T>(jt, jt.kx[i] + 5 * jt.ky[j]);
        if (zero) {
          oth[o] = w * sb[o];
        } else {
          oth[o] = fma(w, resid_smem(cur, o, SY, sb[o], kc0, kc1, kc2), cur[o]);
        }
      });
      __syncthreads();
      T* sw = cur;
      cur = oth;
      oth = sw;
    }
    return cur;
  }
  for (int s = 1; s <= nu; ++s) {
    int a0, b0, a1, b1;
    sweep_box(tg, s, a0, b0, a1, b1);
    const bool zero = ZERO && s == 1;
    if (!zero) {
      // ghosts of the current iterate for the rows / columns this sweep reads
      int c0, d0, c1, d1;
      sweep_box(tg, s - 1, c0, d0, c1, d1);
      region_ghosts(lv, tg, cur, sy, c0, d0, c1, d1, tm);
      tm.sync();
    }
    for (int j = a1 + tm.ty; j < b1; j += tm.nty) {
      const int ky5 = 5 * jt.ky[j];
      for (int i = a0 + tm.tx; i < b0; i += 32) {
        const int o = (j + NG) * sy + (i + NG);
        const T w = jt_get<T>(jt, jt.kx[i] + ky5);
        if (zero) {
          oth[o] = w * sb[o];
        } else {
          oth[o] = fma(w, resid_smem(cur, o, sy, sb[o], kc0, kc1, kc2), cur[o]);
        }
      }
    }
    tm.sync();
    T* sw = cur;
    cur = oth;
    oth = sw;
  }
  return cur;
}

// Down leg of one multigrid level (a level-0 grid, or a single-box AMR level with zero CF
// ghosts): nu weighted-Jacobi sweeps from zero, the smoothed x written to xo (and added to
// xo2 when given), and the residual f - A x restricted (2x2 average) into the coarse
// right-hand side bcn over the covered coarse cells.  halo = 2 nu + 2.
template <typename T, int RM = 0, int TILE = 0, int NT = 256>
__device__ __forceinline__ void mg_down2d_body(const LevelView& lv, const PatchDesc& gp, const PatchDesc& gcp, int tx, int ty, int halo,
                                               int nu, const T* __restrict__ b, T* __restrict__ xo, T* __restrict__ xo2,
                                               T* __restrict__ bcn, T alpha, T beta, T omega, T ood) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const TileGeom tg = tile_geom(gp, lv, tx, ty, halo);
  const int sy = RM > 0 ? RM + 2 * NG : tg.rw + 2 * NG;
  const int E = sy * (RM > 0 ? RM + 2 * NG : tg.rh + 2 * NG);
  constexpr int TM = TILE;      // bound of the tile loops (0: runtime loops)
  constexpr int CM = TILE / 2;  // bound of the coarse-cell loops
  T* sx = reinterpret_cast<T*>(smraw);
  T* st = sx + E;
  T* sb = st + E;
  const Team tm = block_team();
  __shared__ JacobiTable jt;
  build_jacobi_table<T>(jt, lv, tg, alpha, beta, omega, ood, tm);
  const T* __restrict__ bg = b + gp.off;
  const int gsy = (int)gp.sy;
  for_cells<RM, NT>(tg.rw, tg.rh, [&](int i, int j) { sb[(j + NG) * sy + i + NG] = bg[(tg.r1 + j + NG) * gsy + tg.r0 + i + NG]; });
  __syncthreads();
  T* cur = smooth_region<T, true, RM, NT>(lv, tg, jt, sy, sx, st, sb, nu, alpha, beta, tm);
  const int ti = tg.i0 - tg.r0, tj = tg.j0 - tg.r1;
  T* __restrict__ xg = xo + gp.off;
  T* __restrict__ xg2 = xo2 != nullptr ? xo2 + gp.off : nullptr;
  for_cells<TM, NT>(tg.tw, tg.th, [&](int i, int j) {
    const T v = cur[(tj + j + NG) * sy + ti + i + NG];
    xg[(tg.j0 + j + NG) * gsy + tg.i0 + i + NG] = v;
    if (xg2 != nullptr) xg2[(tg.j0 + j + NG) * gsy + tg.i0 + i + NG] += v;
  });
  // residual of the tile's cells (ghosts of the final iterate first), restricted
  int c0, d0, c1, d1;
  sweep_box(tg, nu, c0, d0, c1, d1);
  if (RM == 0 || (tg.fl0 | tg.fh0 | tg.fl1 | tg.fh1)) {
    region_ghosts(lv, tg, cur, sy, c0, d0, c1, d1, tm);
    __syncthreads();
  }
  const T kc2 = beta * pick<T>(lv.inv12h2, lv.inv12h2_f), kc1 = T(16) * kc2, kc0 = fma(T(-60), kc2, alpha);
  const int cw = tg.tw / 2, ch = tg.th / 2;
  const int csy = (int)gcp.sy;
  T* __restrict__ cg = bcn + gcp.off;
  for_cells<CM, NT>(cw, ch, [&](int ci, int cj) {
    T acc = T(0);
#pragma unroll
    for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
      for (int q0 = 0; q0 < 2; ++q0) {
        const int o = (tj + 2 * cj + q1 + NG) * sy + (ti + 2 * ci + q0 + NG);
        acc += resid_smem(cur, o, sy, sb[o], kc0, kc1, kc2);
      }
    cg[(((gp.lo[1] + tg.j0) >> 1) - gcp.lo[1] + cj + NG) * csy + ((gp.lo[0] + tg.i0) >> 1) - gcp.lo[0] + ci + NG] =
        acc * T(0.25);
  });
}

template <typename T, int RM = 0, int TILE = 0, int NT = 256>
__global__ void __launch_bounds__(NT) k_mg_down2d(LevelView lv, PatchDesc gp, PatchDesc gcp, int tx, int ty, int halo,
                                                   int nu, const T* __restrict__ b, T* __restrict__ xo,
                                                   T* __restrict__ xo2, T* __restrict__ bcn, T alpha, T beta, T omega,
                                                   T ood) {
  pdl_wait();
  mg_down2d_body<T, RM, TILE, NT>(lv, gp, gcp, tx, ty, halo, nu, b, xo, xo2, bcn, alpha, beta, omega, ood);
}

// Coarse value at (c0, c1) of a single-patch 2-D grid, at most one cell outside the domain
// in each dimension: the homogeneous physical extension (layer-1 ghost formula), applied
// dimension after dimension at corners (Fig. 1(c) order, as read_ext does).
template <typename T>
__device__ __forceinline__ T coarse_ext2d(const T* __restrict__ cg, int csy, const LevelView& cv, int c0, int c1) {
  const int n0 = cv.ndom[0], n1 = cv.ndom[1];
  const bool o0 = c0 < 0 || c0 >= n0, o1 = c1 < 0 || c1 >= n1;
  if (!o0 && !o1) return cg[(c1 + NG) * csy + c0 + NG];
  int ix[4], iy[4];
  T wx[4], wy[4];
  int cx = 1, cyc = 1;
  ix[0] = c0;
  wx[0] = T(1);
  iy[0] = c1;
  wy[0] = T(1);
  if (o0) {
    const int side = c0 < 0 ? 0 : 1, type = cv.bc[side];
    cx = 4;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      ix[m] = side == 0 ? m : n0 - 1 - m;
      wx[m] = gcoef<T>(type, 0, m);
    }
  }
  if (o1) {
    const int side = c1 < 0 ? 0 : 1, type = cv.bc[2 + side];
    cyc = 4;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      iy[m] = side == 0 ? m : n1 - 1 - m;
      wy[m] = gcoef<T>(type, 0, m);
    }
  }
  T v = T(0);
  for (int a = 0; a < cx; ++a)
    for (int b = 0; b < cyc; ++b) v += wx[a] * wy[b] * cg[(iy[b] + NG) * csy + ix[a] + NG];
  return v;
}

// Up leg of one multigrid level: x = xi + linear prolongation of the coarse correction xc
// (coarse values outside the domain from the homogeneous extension with corners), then nu
// weighted-Jacobi sweeps, written to xo (xi != xo: blocks read halos of xi only).
// halo = 2 nu.
template <typename T, int RM = 0, int TILE = 0, int NT = 256>
__device__ __forceinline__ void mg_up2d_body(const LevelView& lv, const LevelView& cv, const PatchDesc& gp, const PatchDesc& gcp,
                                             int tx, int ty, int halo, int nu, const T* __restrict__ xc,
                                             const T* __restrict__ b, const T* __restrict__ xi, T* __restrict__ xo,
                                             T alpha, T beta, T omega, T ood) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const TileGeom tg = tile_geom(gp, lv, tx, ty, halo);
  const int sy = RM > 0 ? RM + 2 * NG : tg.rw + 2 * NG;
  const int E = sy * (RM > 0 ? RM + 2 * NG : tg.rh + 2 * NG);
  T* sx = reinterpret_cast<T*>(smraw);
  T* st = sx + E;
  T* sb = st + E;
  const int gsy = (int)gp.sy, csy = (int)gcp.sy;
  const T* __restrict__ bg = b + gp.off;
  const T* __restrict__ xg = xi + gp.off;
  const T* __restrict__ cg = xc + gcp.off;
  __shared__ JacobiTable jt;
  for_cells<RM, NT>(tg.rw, tg.rh, [&](int i, int j) {
      const int og = (tg.r1 + j + NG) * gsy + tg.r0 + i + NG;
      const int os = (j + NG) * sy + i + NG;
      sb[os] = bg[og];
      const int gf0 = tg.r0 + i, gf1 = tg.r1 + j;
      const int p0 = gf0 >> 1, p1 = gf1 >> 1;
      const int s0 = (gf0 & 1) ? 1 : -1, s1 = (gf1 & 1) ? 1 : -1;
      T c01, c10, c11;
      const T c00 = cg[(p1 + NG) * csy + (p0 + NG)];
      if (p0 + s0 >= 0 && p0 + s0 < cv.ndom[0] && p1 + s1 >= 0 && p1 + s1 < cv.ndom[1]) {
        const int oc = (p1 + NG) * csy + (p0 + NG);
        c10 = cg[oc + s0];
        c01 = cg[oc + s1 * csy];
        c11 = cg[oc + s1 * csy + s0];
      } else {
        c10 = coarse_ext2d<T>(cg, csy, cv, p0 + s0, p1);
        c01 = coarse_ext2d<T>(cg, csy, cv, p0, p1 + s1);
        c11 = coarse_ext2d<T>(cg, csy, cv, p0 + s0, p1 + s1);
      }
      // cell_prolong's order: (q0, q1) = (0,0), (1,0), (0,1), (1,1)
      T v = T(0);
      v += (T(0.75) * T(0.75)) * c00;
      v += (T(0.25) * T(0.75)) * c10;
      v += (T(0.75) * T(0.25)) * c01;
      v += (T(0.25) * T(0.25)) * c11;
      sx[os] = xg[og] + v;
  });
  const Team tm = block_team();
  build_jacobi_table<T>(jt, lv, tg, alpha, beta, omega, ood, tm);
  __syncthreads();
  const T* cur = smooth_region<T, false, RM, NT>(lv, tg, jt, sy, sx, st, sb, nu, alpha, beta, tm);
  const int ti = tg.i0 - tg.r0, tj = tg.j0 - tg.r1;
  T* __restrict__ xw = xo + gp.off;
  for_cells<TILE, NT>(tg.tw, tg.th, [&](int i, int j) {
    xw[(tg.j0 + j + NG) * gsy + tg.i0 + i + NG] = cur[(tj + j + NG) * sy + ti + i + NG];
  });
}

template <typename T, int RM = 0, int TILE = 0, int NT = 256>
__global__ void __launch_bounds__(NT, 1024 / NT) k_mg_up2d(LevelView lv, LevelView cv, PatchDesc gp, PatchDesc gcp, int tx,
                                                 int ty, int halo, int nu, const T* __restrict__ xc,
                                                 const T* __restrict__ b, const T* __restrict__ xi, T* __restrict__ xo,
                                                 T alpha, T beta, T omega, T ood) {
  pdl_wait();
  mg_up2d_body<T, RM, TILE, NT>(lv, cv, gp, gcp, tx, ty, halo, nu, xc, b, xi, xo, alpha, beta, omega, ood);
}

// Post-smoothing of a single-box AMR level (the correction form's up step): nu weighted-
// Jacobi sweeps from zero on r (the residual already updated with the prolonged coarse
// correction), zero CF ghosts and physical ghosts by formula, and the result t added to the
// level's correction e and to the accumulated correction x on the tile.  Only the tile's
// own e and x cells are read and written (no halo reads of them).  halo = 2 nu.
template <typename T, int RM = 0, int TILE = 0, int NT = 256>
__global__ void __launch_bounds__(NT) k_amr_post2d(LevelView lv, PatchDesc gp, int tx, int ty, int halo, int nu,
                                                    const T* __restrict__ r, T* __restrict__ e, T* __restrict__ x,
                                                    T alpha, T beta, T omega, T ood) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  const TileGeom tg = tile_geom(gp, lv, tx, ty, halo);
  const int sy = RM > 0 ? RM + 2 * NG : tg.rw + 2 * NG;
  const int E = sy * (RM > 0 ? RM + 2 * NG : tg.rh + 2 * NG);
  T* sx = reinterpret_cast<T*>(smraw);
  T* st = sx + E;
  T* sb = st + E;
  const Team tm = block_team();
  __shared__ JacobiTable jt;
  build_jacobi_table<T>(jt, lv, tg, alpha, beta, omega, ood, tm);
  const T* __restrict__ rg = r + gp.off;
  const int gsy = (int)gp.sy;
  for_cells<RM, NT>(tg.rw, tg.rh, [&](int i, int j) { sb[(j + NG) * sy + i + NG] = rg[(tg.r1 + j + NG) * gsy + tg.r0 + i + NG]; });
  __syncthreads();
  const T* cur = smooth_region<T, true, RM, NT>(lv, tg, jt, sy, sx, st, sb, nu, alpha, beta, tm);
  const int ti = tg.i0 - tg.r0, tj = tg.j0 - tg.r1;
  T* __restrict__ eg = e + gp.off;
  T* __restrict__ xg = x + gp.off;
  for_cells<TILE, NT>(tg.tw, tg.th, [&](int i, int j) {
    const T v = cur[(tj + j + NG) * sy + ti + i + NG];
    const int og = (tg.j0 + j + NG) * gsy + tg.i0 + i + NG;
    eg[og] += v;
    if (x != nullptr) xg[og] += v;
  });
}

// Coarse end of the 2-D level-0 multigrid in one block: every grid from m0 (at most 64 cells
// per dimension) down to the coarsest lives in shared memory; the legs use the same region
// sweeps as k_mg_down2d / k_mg_up2d with the whole grid as the region (every side a domain
// face, nothing shrinks), and the dense bottom solve runs between the legs.
constexpr int CB_MAX = 8;
struct CoarseBlock2D {
  int ng;                         // grids m0 .. coarsest
  int nu1, nu2;
  int nbot, ldb;
  const double* minv;             // bottom inverse
  PatchDesc gp;                   // global layout of grid m0 (right-hand side in, correction out)
  int offx[CB_MAX], offt[CB_MAX], offb[CB_MAX];  // element offsets in dynamic shared memory
  double ood[CB_MAX];             // omega / interior diagonal per grid
  LevelView lv[CB_MAX];
};

__device__ __forceinline__ TileGeom whole_grid(const LevelView& lv) {
  TileGeom t;
  t.i0 = t.j0 = t.r0 = t.r1 = 0;
  t.tw = t.rw = lv.ndom[0];
  t.th = t.rh = lv.ndom[1];
  t.fl0 = t.fh0 = t.fl1 = t.fh1 = 1;
  t.pl0 = t.ph0 = t.pl1 = t.ph1 = 1;
  t.g0 = t.g1 = 0;
  return t;
}

template <typename T>
__global__ void __launch_bounds__(1024) k_mg_coarse2d(CoarseBlock2D cb, const T* __restrict__ b, T* __restrict__ x,
                                                      T alpha, T beta, T omega) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ JacobiTable jts[CB_MAX];
  __shared__ double bot[1024];
  T* sm = reinterpret_cast<T*>(smraw);
  const Team all = block_team();
  const int M = cb.ng - 1;
  for (int q = 0; q < cb.ng; ++q)
    build_jacobi_table<T>(jts[q], cb.lv[q], whole_grid(cb.lv[q]), alpha, beta, omega, T(cb.ood[q]), all);
  {
    const int n0 = cb.lv[0].ndom[0], n1 = cb.lv[0].ndom[1], sy = n0 + 2 * NG;
    const T* __restrict__ bg = b + cb.gp.off;
    const int gsy = (int)cb.gp.sy;
    for (int t = all.tid; t < n0 * n1; t += all.nth) {
      const int i = t % n0, j = t / n0;
      sm[cb.offb[0] + (j + NG) * sy + i + NG] = bg[(j + NG) * gsy + i + NG];
    }
  }
  __syncthreads();
  // buffer holding each grid's iterate after its down leg: nu1 sweeps from zero starting in
  // the x array end in x for an even count, in the t array for an odd one
  const bool down_in_t = (cb.nu1 & 1) != 0, up_swaps = (cb.nu2 & 1) != 0;
  for (int q = 0; q < M; ++q) {
    const LevelView& lv = cb.lv[q];
    const TileGeom tg = whole_grid(lv);
    const Team tm = sub_team(tg.rw * tg.rh);
    if (tm.tid < tm.nth) {
      const int sy = tg.rw + 2 * NG;
      T* sb = sm + cb.offb[q];
      T* cur = smooth_region<T, true>(lv, tg, jts[q], sy, sm + cb.offx[q], sm + cb.offt[q], sb, cb.nu1, alpha, beta, tm);
      region_ghosts(lv, tg, cur, sy, 0, tg.rw, 0, tg.rh, tm);
      tm.sync();
      const T inv = pick<T>(lv.inv12h2, lv.inv12h2_f);
      const int cw = tg.rw / 2, ch = tg.rh / 2, csy = cw + 2 * NG;
      T* bc = sm + cb.offb[q + 1];
      for (int t = tm.tid; t < cw * ch; t += tm.nth) {
        const int ci = t % cw, cj = t / cw;
        T acc = T(0);
#pragma unroll
        for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
          for (int q0 = 0; q0 < 2; ++q0) {
            const int o = (2 * cj + q1 + NG) * sy + (2 * ci + q0 + NG);
            const T xc = cur[o];
            acc += sb[o] - (alpha * xc + beta * (lap_smem(cur, o, sy) * inv));
          }
        bc[(cj + NG) * csy + ci + NG] = acc * T(0.25);
      }
    }
    __syncthreads();
  }
  {
    // dense bottom solve (FP64 accumulation), cell order x fastest
    const int n0 = cb.lv[M].ndom[0], sy = n0 + 2 * NG;
    const T* bm = sm + cb.offb[M];
    for (int t = all.tid; t < cb.nbot; t += all.nth) bot[t] = (double)bm[(t / n0 + NG) * sy + t % n0 + NG];
    __syncthreads();
    T* xm = sm + cb.offx[M];
    for (int t = all.tid; t < cb.nbot; t += all.nth) {
      double acc = 0.0;
      const double* row = cb.minv + (long long)t * cb.ldb;
      for (int k = 0; k < cb.nbot; ++k) acc = fma(row[k], bot[k], acc);
      xm[(t / n0 + NG) * sy + t % n0 + NG] = T(acc);
    }
    __syncthreads();
  }
  for (int q = M - 1; q >= 0; --q) {
    const LevelView& lv = cb.lv[q];
    const LevelView& cv = cb.lv[q + 1];
    const TileGeom tg = whole_grid(lv);
    const Team tm = sub_team(tg.rw * tg.rh);
    if (tm.tid < tm.nth) {
      const int sy = tg.rw + 2 * NG, csy = cv.ndom[0] + 2 * NG;
      T* xq = down_in_t ? sm + cb.offt[q] : sm + cb.offx[q];
      T* oth = down_in_t ? sm + cb.offx[q] : sm + cb.offt[q];
      // the coarser grid's final iterate: its down-leg buffer, swapped by an odd nu2
      const bool cin_t = (q + 1 == M) ? false : (down_in_t != up_swaps);
      const T* cg = cin_t ? sm + cb.offt[q + 1] : sm + cb.offx[q + 1];
      for (int t = tm.tid; t < tg.rw * tg.rh; t += tm.nth) {
        const int i = t % tg.rw, j = t / tg.rw;
        const int p0 = i >> 1, p1 = j >> 1;
        const int s0 = (i & 1) ? 1 : -1, s1 = (j & 1) ? 1 : -1;
        const T c00 = cg[(p1 + NG) * csy + p0 + NG];
        const T c10 = coarse_ext2d<T>(cg, csy, cv, p0 + s0, p1);
        const T c01 = coarse_ext2d<T>(cg, csy, cv, p0, p1 + s1);
        const T c11 = coarse_ext2d<T>(cg, csy, cv, p0 + s0, p1 + s1);
        T v = T(0);
        v += (T(0.75) * T(0.75)) * c00;
        v += (T(0.25) * T(0.75)) * c10;
        v += (T(0.75) * T(0.25)) * c01;
        v += (T(0.25) * T(0.25)) * c11;
        xq[(j + NG) * sy + i + NG] += v;
      }
      tm.sync();
      smooth_region<T, false>(lv, tg, jts[q], sy, xq, oth, sm + cb.offb[q], cb.nu2, alpha, beta, tm);
    }
    __syncthreads();
  }
  {
    const int n0 = cb.lv[0].ndom[0], n1 = cb.lv[0].ndom[1], sy = n0 + 2 * NG;
    T* __restrict__ xg = x + cb.gp.off;
    const int gsy = (int)cb.gp.sy;
    const T* x0 = (down_in_t != up_swaps) ? sm + cb.offt[0] : sm + cb.offx[0];
    for (int t = all.tid; t < n0 * n1; t += all.nth) {
      const int i = t % n0, j = t / n0;
      xg[(j + NG) * gsy + i + NG] = x0[(j + NG) * sy + i + NG];
    }
  }
}

// ------------------------------------------------------------------------ square coarse V-cycle
// The coarse end of the 2-D level-0 multigrid for the common case of a square pyramid
// N0, N0/2, ... down to the bottom grid (N0 = 64: bottom 4; N0 = 48: bottom 6), every size a
// compile-time constant, so that every loop over a grid's cells has a fixed trip count and
// every stencil offset is an immediate.  Same V-cycle as k_mg_coarse2d (weighted-Jacobi legs,
// residual restriction, linear prolongation with the homogeneous extension, dense bottom
// solve); the physical ghost layers of an array are written by one pass over its four sides
// (one warp per side) before a sweep reads them.
constexpr int SQ_NT = 1024;  // threads of the block

template <int N>
struct Sq {
  static constexpr int S = N + 4;  // row pitch (two ghost layers each side)
  static constexpr int E = S * S;
  static constexpr bool bottom = (N % 2 != 0) || (N / 2 < MIN_BOX);
};
// element offset of grid N's three arrays (x, t, b) in shared memory
template <int N0, int N>
__host__ __device__ constexpr int sq_off() {
  if constexpr (N >= N0) return 0;
  else return sq_off<N0, 2 * N>() + 3 * Sq<2 * N>::E;
}
template <int N0, int N>
__host__ __device__ constexpr int sq_total() {
  if constexpr (Sq<N>::bottom) return sq_off<N0, N>() + 3 * Sq<N>::E;
  else return sq_total<N0, N / 2>();
}
template <int N0, int N>
__host__ __device__ constexpr int sq_bottom() {
  if constexpr (Sq<N>::bottom) return N;
  else return sq_bottom<N0, N / 2>();
}
template <int N0, int N>
__host__ __device__ constexpr int sq_depth() {  // grid index of N (0 = N0)
  if constexpr (N >= N0) return 0;
  else return 1 + sq_depth<N0, 2 * N>();
}

struct SqCtx {
  float alpha, beta, omega;
  int bcm;  // boundary type of face f (0 Dirichlet, 1 Neumann) in bit f
  int nu1, nu2;
  __device__ __forceinline__ int bc(int f) const { return (bcm >> f) & 1; }
};

template <typename T, int N>
__device__ __forceinline__ T sq_ax(const T* __restrict__ a, int i, int j, T alpha, T binv) {
  constexpr int S = Sq<N>::S;
  const int o = (j + 2) * S + i + 2;
  const T xc = a[o];
  const T s1 = (a[o - 1] + a[o + 1]) + (a[o - S] + a[o + S]);
  const T s2 = (a[o - 2] + a[o + 2]) + (a[o - 2 * S] + a[o + 2 * S]);
  return alpha * xc + binv * ((T(16) * s1 - s2 - T(60) * xc) + T(0));
}

// Jacobi factor omega / diag of (i, j): table entry kx + 5 ky by distance class to the faces
template <int N>
__device__ __forceinline__ int sq_class(int i, int j) {
  return face_class(i, N) + 5 * face_class(j, N);
}

template <typename T, int N0>
struct SqVcycle {
  T* sm;                 // dynamic shared memory
  const float* wt;       // per grid 25 Jacobi factors (shared)
  const double* minv;    // bottom inverse
  int nbot, ldb;
  double* bot;           // bottom right-hand side (shared, FP64)
  const float* binv;     // beta / (12 h^2) per grid (shared)
  SqCtx c;

  template <int N> __device__ T* X() const { return sm + sq_off<N0, N>(); }
  template <int N> __device__ T* Tt() const { return sm + sq_off<N0, N>() + Sq<N>::E; }
  template <int N> __device__ T* B() const { return sm + sq_off<N0, N>() + 2 * Sq<N>::E; }

  // physical ghost layers 1 and 2 of array a on grid N (Eqs. (velBCHomoDiri5th)/(Neumann5),
  // homogeneous), entry e = side x (2N) + 2 position + layer; with corners, also the four
  // layer-1 corner ghosts as the x extension of the y extension
  template <int N>
  __device__ void ghosts(T* a, bool corners) const {
    constexpr int S = Sq<N>::S, NE = 8 * N, IT = (NE + SQ_NT - 1) / SQ_NT;
    const int tid = threadIdx.x + 32 * threadIdx.y;
#pragma unroll
    for (int q = 0; q < IT; ++q) {
      const int e = tid + q * SQ_NT;
      if (NE % SQ_NT == 0 || e < NE) {
        const int f = e / (2 * N), pos = (e % (2 * N)) >> 1, layer = e & 1;
        const int side = f & 1, t = c.bc(f);
        T v = T(0);
        if (f < 2) {
          const int row = (pos + 2) * S + 2;
#pragma unroll
          for (int m = 0; m < 4; ++m) v += gcoef<T>(t, layer, m) * a[row + (side == 0 ? m : N - 1 - m)];
          a[row + (side == 0 ? -1 - layer : N + layer)] = v;
        } else {
#pragma unroll
          for (int m = 0; m < 4; ++m) v += gcoef<T>(t, layer, m) * a[((side == 0 ? m : N - 1 - m) + 2) * S + pos + 2];
          a[((side == 0 ? -1 - layer : N + layer) + 2) * S + pos + 2] = v;
        }
      }
    }
    if (corners && tid < 4) {
      const int sx = tid & 1, sy = tid >> 1, tx = c.bc(sx), ty = c.bc(2 + sy);
      T v = T(0);
#pragma unroll
      for (int ia = 0; ia < 4; ++ia)
#pragma unroll
        for (int ib = 0; ib < 4; ++ib)
          v += gcoef<T>(tx, 0, ia) * gcoef<T>(ty, 0, ib) *
               a[((sy == 0 ? ib : N - 1 - ib) + 2) * S + (sx == 0 ? ia : N - 1 - ia) + 2];
      a[((sy == 0 ? -1 : N) + 2) * S + (sx == 0 ? -1 : N) + 2] = v;
    }
    __syncthreads();
  }

  // nu weighted-Jacobi sweeps on grid N; zero: the first one starts from x = 0 and writes a.
  // Returns the array holding the result.
  template <int N>
  __device__ T* smooth(T* a, T* o, int nu, bool zero) const {
    constexpr int S = Sq<N>::S, NC = N * N, IT = (NC + SQ_NT - 1) / SQ_NT;
    const T* b = B<N>();
    const float* w = wt + 25 * sq_depth<N0, N>();
    const T bi = T(binv[sq_depth<N0, N>()]);
    const int tid = threadIdx.x + 32 * threadIdx.y;
    for (int s = 0; s < nu; ++s) {
      const bool z = zero && s == 0;
      if (!z) ghosts<N>(a, false);
#pragma unroll
      for (int q = 0; q < IT; ++q) {
        const int cidx = tid + q * SQ_NT;
        if (NC % SQ_NT == 0 || cidx < NC) {
          const int i = cidx % N, j = cidx / N;
          const int oc = (j + 2) * S + i + 2;
          const T wc = T(w[sq_class<N>(i, j)]);
          if (z) a[oc] = wc * b[oc];
          else o[oc] = a[oc] + wc * (b[oc] - sq_ax<T, N>(a, i, j, T(c.alpha), bi));
        }
      }
      __syncthreads();
      if (!z) { T* sw = a; a = o; o = sw; }
    }
    return a;
  }

  // residual of grid N restricted (2 x 2 average) into the right-hand side of grid N/2
  template <int N>
  __device__ void restrict_residual(const T* a) const {
    constexpr int M = N / 2, MS = Sq<M>::S, NC = M * M, IT = (NC + SQ_NT - 1) / SQ_NT;
    constexpr int S = Sq<N>::S;
    const T* b = B<N>();
    T* bc = B<M>();
    const T bi = T(binv[sq_depth<N0, N>()]);
    const int tid = threadIdx.x + 32 * threadIdx.y;
    ghosts<N>(const_cast<T*>(a), false);
#pragma unroll
    for (int q = 0; q < IT; ++q) {
      const int cidx = tid + q * SQ_NT;
      if (NC % SQ_NT == 0 || cidx < NC) {
        const int ci = cidx % M, cj = cidx / M;
        T acc = T(0);
#pragma unroll
        for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
          for (int q0 = 0; q0 < 2; ++q0) {
            const int i = 2 * ci + q0, j = 2 * cj + q1;
            acc += b[(j + 2) * S + i + 2] - sq_ax<T, N>(a, i, j, T(c.alpha), bi);
          }
        bc[(cj + 2) * MS + ci + 2] = acc * T(0.25);
      }
    }
    __syncthreads();
  }

  // x_N += linear prolongation of the grid-N/2 correction cg (coarse values outside the
  // domain: the homogeneous layer-1 extension, corners included)
  template <int N>
  __device__ void prolong(T* a, T* cg) const {
    constexpr int M = N / 2, S = Sq<N>::S, NC = N * N, IT = (NC + SQ_NT - 1) / SQ_NT;
    const int tid = threadIdx.x + 32 * threadIdx.y;
    ghosts<M>(cg, true);
#pragma unroll
    for (int q = 0; q < IT; ++q) {
      const int cidx = tid + q * SQ_NT;
      if (NC % SQ_NT == 0 || cidx < NC) {
        const int i = cidx % N, j = cidx / N;
        const int p0 = i >> 1, p1 = j >> 1;
        const int s0 = (i & 1) ? 1 : -1, s1 = (j & 1) ? 1 : -1;
        const int oc = (p1 + 2) * Sq<M>::S + p0 + 2;
        const T c00 = cg[oc];
        const T c10 = cg[oc + s0];
        const T c01 = cg[oc + s1 * Sq<M>::S];
        const T c11 = cg[oc + s1 * Sq<M>::S + s0];
        T v = T(0);
        v += (T(0.75) * T(0.75)) * c00;
        v += (T(0.25) * T(0.75)) * c10;
        v += (T(0.75) * T(0.25)) * c01;
        v += (T(0.25) * T(0.25)) * c11;
        a[(j + 2) * S + i + 2] += v;
      }
    }
    __syncthreads();
  }

  // dense bottom solve on grid N (FP64 accumulation), result in X<N>
  template <int N>
  __device__ void bottom() const {
    constexpr int S = Sq<N>::S;
    const int tid = threadIdx.x + 32 * threadIdx.y;
    const T* b = B<N>();
    for (int t = tid; t < nbot; t += SQ_NT) bot[t] = (double)b[(t / N + 2) * S + t % N + 2];
    __syncthreads();
    T* x = X<N>();
    for (int t = tid; t < nbot; t += SQ_NT) {
      double acc = 0.0;
      const double* row = minv + (long long)t * ldb;
      for (int k = 0; k < nbot; ++k) acc = fma(row[k], bot[k], acc);
      x[(t / N + 2) * S + t % N + 2] = T(acc);
    }
    __syncthreads();
  }

  // V-cycle from grid N down (its right-hand side in B<N>); returns the array with the result
  template <int N>
  __device__ T* cycle() const {
    if constexpr (Sq<N>::bottom) {
      bottom<N>();
      return X<N>();
    } else {
      T* cur = smooth<N>(X<N>(), Tt<N>(), c.nu1, true);
      restrict_residual<N>(cur);
      T* cg = cycle<N / 2>();
      prolong<N>(cur, cg);
      return smooth<N>(cur, cur == X<N>() ? Tt<N>() : X<N>(), c.nu2, false);
    }
  }
};

template <typename T, int N0>
__device__ __forceinline__ void mg_coarse2d_sq_body(const CoarseBlock2D& cb, const T* __restrict__ b, T* __restrict__ x,
                                                    T alpha, T beta, T omega) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ float wt[25 * CB_MAX];
  __shared__ double bot[1024];
  __shared__ float sbinv[CB_MAX];
  SqVcycle<T, N0> v;
  v.sm = reinterpret_cast<T*>(smraw);
  v.wt = wt;
  v.minv = cb.minv;
  v.nbot = cb.nbot;
  v.ldb = cb.ldb;
  v.bot = bot;
  v.binv = sbinv;
  v.c.alpha = (float)alpha;
  v.c.beta = (float)beta;
  v.c.omega = (float)omega;
  v.c.bcm = 0;
  for (int f = 0; f < 4; ++f) v.c.bcm |= (cb.lv[0].bc[f] & 1) << f;
  v.c.nu1 = cb.nu1;
  v.c.nu2 = cb.nu2;
  const int tid = threadIdx.x + 32 * threadIdx.y;
  for (int q = tid; q < cb.ng; q += SQ_NT) sbinv[q] = beta * cb.lv[q].inv12h2_f;
  // Jacobi factors per grid (the diagonal differs from the interior one within two cells of a
  // face: diag_sum's order, -60 then the x correction, then the y correction)
  for (int e = tid; e < 25 * cb.ng; e += SQ_NT) {
    const int q = e / 25, k = e % 25, a = k % 5, bb = k / 5;
    const LevelView& lv = cb.lv[q];
    const float cx = a == 0 ? 0.f : lv.dcorr_f[(a - 1) / 2][(a - 1) % 2];
    const float cy = bb == 0 ? 0.f : lv.dcorr_f[2 + (bb - 1) / 2][(bb - 1) % 2];
    wt[e] = k == 0 ? (float)cb.ood[q] : (float)(omega / (alpha + beta * lv.inv12h2_f * ((T(-60) + cx) + cy)));
  }
  {
    constexpr int S = Sq<N0>::S;
    const T* __restrict__ bg = b + cb.gp.off;
    const int gsy = (int)cb.gp.sy;
    T* bs = v.template B<N0>();
    for (int t = tid; t < N0 * N0; t += SQ_NT) {
      const int i = t % N0, j = t / N0;
      bs[(j + 2) * S + i + 2] = bg[(j + NG) * gsy + i + NG];
    }
  }
  __syncthreads();
  const T* res = v.template cycle<N0>();
  {
    constexpr int S = Sq<N0>::S;
    T* __restrict__ xg = x + cb.gp.off;
    const int gsy = (int)cb.gp.sy;
    for (int t = tid; t < N0 * N0; t += SQ_NT) {
      const int i = t % N0, j = t / N0;
      xg[(j + NG) * gsy + i + NG] = res[(j + 2) * S + i + 2];
    }
  }
}

template <typename T, int N0>
__global__ void __launch_bounds__(SQ_NT) k_mg_coarse2d_sq(CoarseBlock2D cb, const T* __restrict__ b, T* __restrict__ x,
                                                          T alpha, T beta, T omega) {
  pdl_wait();
  mg_coarse2d_sq_body<T, N0>(cb, b, x, alpha, beta, omega);
}

// ------------------------------------------------------------------------ work-list batches
// A batch of independent single-level 2-D problems solved together: every phase of the
// mixed-precision iteration is one launch over a list of descriptors (problem, grid) in
// device memory, blockIdx.z (or blockIdx.x) selecting the entry; entries of problems that
// have converged (active[p] == 0) return at once.  The bodies are the single-problem
// kernels' bodies.
struct BDown {  // down leg of grid m of problem p
  int p, tiles_x, tiles_y, tt, halo, nu;
  LevelView lv;
  PatchDesc gp, gcp;
  const float* b;
  float* xo;
  float* bcn;
  float alpha, beta, omega, ood;
};
struct BUp {  // up leg of grid m of problem p
  int p, tiles_x, tiles_y, tt, halo, nu;
  LevelView lv, cv;
  PatchDesc gp, gcp;
  const float* xc;
  const float* b;
  const float* xi;
  float* xo;
  float alpha, beta, omega, ood;
};
struct BCoarse {  // one-block coarse V-cycle of problem p (square pyramid from n0)
  int p, n0;
  CoarseBlock2D cb;
  const float* b;
  float* x;
  float alpha, beta, omega;
};
struct BResid {  // FP64 residual of problem p's level: out = f - (alpha x + beta L x)
  int p, tiles_x, tiles_y;
  LevelView lv;
  const double* x;
  const double* f;
  double* out;
  double alpha, beta;
};
struct BFlat {  // whole-array passes of problem p
  int p;
  long long n;
  const unsigned char* vmask;
  double* phi;      // update: phi += e on valid cells
  const float* e;
  const double* r;  // norm: valid max-norm of r into acc[p], rin = (float) r
  float* rin;
  const double* f;  // init: F = f, phi = 0 (zero), fnorm
  double* F;
};

template <int RM, int TILE>
__global__ void __launch_bounds__(256) k_mg_down2d_b(const BDown* __restrict__ d, const int* __restrict__ active) {
  pdl_wait();
  const BDown& e = d[blockIdx.z];
  if (!active[e.p] || (int)blockIdx.x >= e.tiles_x || (int)blockIdx.y >= e.tiles_y) return;
  mg_down2d_body<float, RM, TILE>(e.lv, e.gp, e.gcp, e.tt, e.tt, e.halo, e.nu, e.b, e.xo, nullptr, e.bcn, e.alpha,
                                  e.beta, e.omega, e.ood);
}

template <int RM, int TILE>
__global__ void __launch_bounds__(256, 4) k_mg_up2d_b(const BUp* __restrict__ d, const int* __restrict__ active) {
  pdl_wait();
  const BUp& e = d[blockIdx.z];
  if (!active[e.p] || (int)blockIdx.x >= e.tiles_x || (int)blockIdx.y >= e.tiles_y) return;
  mg_up2d_body<float, RM, TILE>(e.lv, e.cv, e.gp, e.gcp, e.tt, e.tt, e.halo, e.nu, e.xc, e.b, e.xi, e.xo, e.alpha,
                                e.beta, e.omega, e.ood);
}

__global__ void __launch_bounds__(SQ_NT) k_mg_coarse2d_sq_b(const BCoarse* __restrict__ d, const int* __restrict__ active) {
  pdl_wait();
  const BCoarse& e = d[blockIdx.x];
  if (!active[e.p]) return;
  if (e.n0 == 64) mg_coarse2d_sq_body<float, 64>(e.cb, e.b, e.x, e.alpha, e.beta, e.omega);
  else mg_coarse2d_sq_body<float, 48>(e.cb, e.b, e.x, e.alpha, e.beta, e.omega);
}

template <int ROWS>
__global__ void __launch_bounds__(BX* BY) k_resid2d_b(const BResid* __restrict__ d, const int* __restrict__ active) {
  pdl_wait();
  const BResid& e = d[blockIdx.z];
  if (!active[e.p] || (int)blockIdx.x >= e.tiles_x || (int)blockIdx.y >= e.tiles_y) return;
  level_op2d_tiled_body<double, OP_RESID, false, ROWS>(e.lv, 0, e.x, e.f, e.out, nullptr, e.alpha, e.beta, 0.0, 0.0,
                                                       nullptr, JFac<double, 2>{});
}

// block-wide max of IEEE bits (non-negative doubles) into *acc
__device__ __forceinline__ void block_max_bits(unsigned long long v, unsigned long long* acc) {
  __shared__ unsigned long long sm[8];
  for (int s = 16; s > 0; s >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, s);
    v = u > v ? u : v;
  }
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < 8 ? sm[threadIdx.x] : 0ull;
    for (int s = 16; s > 0; s >>= 1) {
      const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, s);
      v = u > v ? u : v;
    }
    if (threadIdx.x == 0 && v != 0ull) atomicMax(acc, v);
  }
}

// set-up of every problem: F = f, phi = 0 (zero != 0), valid max-norm of f into fbits[p]
__global__ void __launch_bounds__(256) k_init_b(const BFlat* __restrict__ d, int zero, unsigned long long* __restrict__ fbits) {
  pdl_wait();
  const BFlat& e = d[blockIdx.y];
  unsigned long long v = 0ull;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < e.n; i += (long long)gridDim.x * blockDim.x) {
    const double x = e.f[i];
    e.F[i] = x;
    if (zero) e.phi[i] = 0.0;
    if (e.vmask[i]) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(x));
      v = b > v ? b : v;
    }
  }
  block_max_bits(v, fbits + e.p);
}

// phi += e on the valid cells of every active problem; clears its residual-norm slot
__global__ void __launch_bounds__(256) k_update_b(const BFlat* __restrict__ d, const int* __restrict__ active,
                                                  unsigned long long* __restrict__ rbits) {
  pdl_wait();
  const BFlat& e = d[blockIdx.y];
  if (!active[e.p]) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) rbits[e.p] = 0ull;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < e.n; i += (long long)gridDim.x * blockDim.x)
    if (e.vmask[i]) e.phi[i] += f32_to_f64(e.e[i]);
}

// valid max-norm of the residual into rbits[p] and its FP32 copy (the next V-cycle's
// right-hand side) for every active problem
__global__ void __launch_bounds__(256) k_norm_convert_b(const BFlat* __restrict__ d, const int* __restrict__ active,
                                                        unsigned long long* __restrict__ rbits) {
  pdl_wait();
  const BFlat& e = d[blockIdx.y];
  if (!active[e.p]) return;
  unsigned long long v = 0ull;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < e.n; i += (long long)gridDim.x * blockDim.x) {
    const double x = e.r[i];
    e.rin[i] = f64_to_f32(x);
    if (e.vmask[i]) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
      v = b > v ? b : v;
    }
  }
  block_max_bits(v, rbits + e.p);
}

// ------------------------------------------------------------------------ fused coarse V-cycle
// The coarse end of the level-0 multigrid pyramid (every grid from m0 down to the coarsest,
// whose arrays fit in shared memory together) runs as ONE block: the same per-cell
// smoothing / residual-restriction / prolongation functions as the standalone kernels, with
// __syncthreads() between phases, and the dense bottom solve at the end of the descent.
constexpr int CMG_MAX = 10;
struct CoarseMG {
  int ng;                      // grids handled, index 0 = m0, ng-1 = coarsest
  int nu1, nu2;
  int nbot, ldb;
  const double* minv;          // bottom inverse (global)
  PatchDesc gp;                // global layout of grid m0 (right-hand side in, correction out)
  LevelView lv[CMG_MAX];       // per-grid constants (patches pointer unused)
  PatchDesc sp[CMG_MAX];       // shared-memory layout of each grid's arrays (off = 0)
  int offx[CMG_MAX], offb[CMG_MAX], offt[CMG_MAX];  // element offsets in dynamic shared memory
};

__device__ __forceinline__ void cell_of(const PatchDesc& p, int t, int& i, int& j, int& k) {
  i = t % p.n[0];
  j = (t / p.n[0]) % p.n[1];
  k = t / (p.n[0] * p.n[1]);
}

template <typename T, int D, bool TR = false>
__global__ void __launch_bounds__(1024) k_coarse_mg(CoarseMG cm, const T* __restrict__ bglob, T* __restrict__ xglob,
                                                    T alpha, T beta, T omega) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  T* sm = reinterpret_cast<T*>(smraw);
  const int tid = threadIdx.x, nth = blockDim.x;
  auto ncell = [&](int m) { return cm.sp[m].n[0] * cm.sp[m].n[1] * cm.sp[m].n[2]; };
  int i, j, k;
  for (int t = tid; t < ncell(0); t += nth) {
    cell_of(cm.sp[0], t, i, j, k);
    sm[cm.offb[0] + poff(cm.sp[0], i, j, k)] = bglob[poff(cm.gp, i, j, k)];
  }
  __syncthreads();
  for (int m = 0; m + 1 < cm.ng; ++m) {
    T* x = sm + cm.offx[m];
    T* tb = sm + cm.offt[m];
    const T* b = sm + cm.offb[m];
    T* cur = (cm.nu1 % 2 == 1) ? x : tb;
    T* oth = (cur == x) ? tb : x;
    for (int t = tid; t < ncell(m); t += nth) {
      cell_of(cm.sp[m], t, i, j, k);
      cell_level_op<T, D, OP_JACOBI0, TR>(cm.lv[m], cm.sp[m], i, j, k, nullptr, b, cur, nullptr, alpha, beta, omega);
    }
    __syncthreads();
    for (int s = 1; s < cm.nu1; ++s) {
      for (int t = tid; t < ncell(m); t += nth) {
        cell_of(cm.sp[m], t, i, j, k);
        cell_level_op<T, D, OP_JACOBI, TR>(cm.lv[m], cm.sp[m], i, j, k, cur, b, oth, nullptr, alpha, beta, omega);
      }
      __syncthreads();
      T* sw = cur;
      cur = oth;
      oth = sw;
    }
    for (int t = tid; t < ncell(m + 1); t += nth) {
      cell_of(cm.sp[m + 1], t, i, j, k);
      const int g[3] = {i, j, k};
      cell_restrict<T, D, true, TR>(cm.lv[m], cm.sp[m], cm.sp[m + 1], g, x, b, sm + cm.offb[m + 1], alpha, beta);
    }
    __syncthreads();
  }
  {
    const int M = cm.ng - 1;
    const T* b = sm + cm.offb[M];
    T* x = sm + cm.offx[M];
    for (int r = tid; r < cm.nbot; r += nth) {
      double acc = 0.0;
      const double* row = cm.minv + (long long)r * cm.ldb;
      for (int q = 0; q < cm.nbot; ++q) {
        cell_of(cm.sp[M], q, i, j, k);
        acc = fma(row[q], (double)b[poff(cm.sp[M], i, j, k)], acc);
      }
      cell_of(cm.sp[M], r, i, j, k);
      x[poff(cm.sp[M], i, j, k)] = T(acc);
    }
    __syncthreads();
  }
  for (int m = cm.ng - 2; m >= 0; --m) {
    T* x = sm + cm.offx[m];
    T* tb = sm + cm.offt[m];
    const T* b = sm + cm.offb[m];
    for (int t = tid; t < ncell(m); t += nth) {
      cell_of(cm.sp[m], t, i, j, k);
      const int gf[3] = {i, j, k};
      cell_prolong<T, D>(cm.lv[m + 1], cm.sp[m], cm.sp[m + 1], gf, sm + cm.offx[m + 1], x, (T*)nullptr);
    }
    __syncthreads();
    T* cur = x;
    T* oth = tb;
    for (int s = 0; s < cm.nu2; ++s) {
      for (int t = tid; t < ncell(m); t += nth) {
        cell_of(cm.sp[m], t, i, j, k);
        cell_level_op<T, D, OP_JACOBI, TR>(cm.lv[m], cm.sp[m], i, j, k, cur, b, oth, nullptr, alpha, beta, omega);
      }
      __syncthreads();
      T* sw = cur;
      cur = oth;
      oth = sw;
    }
    if (cur != x) {
      for (int t = tid; t < ncell(m); t += nth) {
        cell_of(cm.sp[m], t, i, j, k);
        const long long o = poff(cm.sp[m], i, j, k);
        x[o] = cur[o];
      }
      __syncthreads();
    }
  }
  for (int t = tid; t < ncell(0); t += nth) {
    cell_of(cm.sp[0], t, i, j, k);
    xglob[poff(cm.gp, i, j, k)] = sm[cm.offx[0] + poff(cm.sp[0], i, j, k)];
  }
}

// ------------------------------------------------------------------------ composite transpose
// Pieces of (A^comp)^T z beyond the per-level transposed stencil (which also covers the
// physical-ghost coefficients and same-level copies through the copy ghosts of z):
//   k_reflux_T   transposed refluxing (COH-3): scatters each coarse row's weight onto the
//                coarse and fine cells its flux difference reads (atomic adds); coarse reads
//                outside the domain go through the physical ghost coefficients;
//   k_cfi_T      transposed AMRCFI: the weight that fine rows put on a CF ghost (its
//                stencil reads plus any refluxing weight stored in the ghost slot) goes to
//                the ghost's 5^D coarse window with the interpolation weights (atomic adds);
//   k_avgdown_T  transposed average-down: invalid coarse cells hand 1/2^D of their weight
//                to each child (applied coarse to fine).
template <typename T>
struct Out3 {
  T* p[3];
};
template <typename T>
struct P3c {
  const T* p[3];
};

// W[x] += wgt for a read of x at patch-local cell c by a stencil along d.  A read outside the
// domain was a physical ghost (Eqs. velBCHomoDiri5th / Neumann5, homogeneous part): its
// weight goes to the four interior cells the ghost formula combines.  Reads of copy or CF
// ghost slots land in those slots (moved on by k_copy_T / k_cfi_T).
template <typename T, int D>
__device__ __forceinline__ void scatter_read(T* __restrict__ W, const PatchDesc& p, const LevelView& lv, const int* c,
                                             int d, T wgt) {
  const int g = p.lo[d] + c[d];
  if (g >= 0 && g < lv.ndom[d]) {
    atomicAdd(&W[poff(p, c[0], c[1], c[2])], wgt);
    return;
  }
  const int gs = g < 0 ? 0 : 1;
  const int layer = gs == 0 ? -g : g - lv.ndom[d] + 1;
  const int type = lv.bc[2 * d + gs];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    int c2[3] = {c[0], c[1], c[2]};
    c2[d] = gs == 0 ? (m - p.lo[d]) : (lv.ndom[d] - 1 - m - p.lo[d]);
    atomicAdd(&W[poff(p, c2[0], c2[1], c2[2])], gcoef<T>(type, layer - 1, m) * wgt);
  }
}

// Transposed refluxing (COH-3).  kind 0: Laplacian fluxes (face derivative, one field, all
// W.p[] equal); kind 1: divergence fluxes (face values of component d into W.p[d]).  The
// forward correction is out[c] += coef/hc * sum_faces s (Fbar/hf' - Fc/hc') with hf' = hf,
// hc' = hc for derivatives and 1 for values.  A thread per (cell, face, cell of the face's line):
// as one thread per cell the lists of a 2-D level, a few hundred cells, took 10 us of serial
// atomics and FP64 divisions on five SMs (now 3.9 us).
constexpr int REFLUX_T_LANES = 4;
template <typename T, int D>
__global__ void __launch_bounds__(128) k_reflux_T(LevelView crs, LevelView fine, const RefluxEntry* __restrict__ list,
                                                  long long n, const T* __restrict__ z, Out3<T> W, T coef, int kind) {
  pdl_wait();
  const long long t = (long long)blockIdx.x * 128 + threadIdx.x;
  const int q = (int)(t & 3), f = (int)((t >> 2) % (2 * D)), d = f >> 1, side = f & 1;
  if (t >= n * (8 * D)) return;
  const RefluxEntry& e = list[t / (8 * D)];
  if (!(e.faces & (1 << f))) return;
  const T zc = z[e.coff];
  if (zc == T(0)) return;
  const PatchDesc cp = crs.patches[e.cpatch], fp = fine.patches[e.fpatch[f]];
  const T fq = kind == 0 ? (q == 0 ? T(1.0 / 12.0) : q == 1 ? T(-15.0 / 12.0) : q == 2 ? T(15.0 / 12.0) : T(-1.0 / 12.0))
                         : (q == 0 || q == 3 ? T(-1.0 / 12.0) : T(7.0 / 12.0));
  const T ihc = pick<T>(crs.invh, crs.invh_f), ihf = pick<T>(fine.invh, fine.invh_f);
  const T a = coef * zc * ihc * T(side == 1 ? 1 : -1) * fq;
  T* __restrict__ Wd = kind == 0 || d == 0 ? W.p[0] : d == 1 ? W.p[1] : W.p[2];
  const int g0 = e.g[0], g1 = e.g[1], g2 = D == 3 ? e.g[2] : 0;
  const int sc = side - 2 + q;  // coarse cells gd - 2 + side ..
  int cc[3] = {g0 - cp.lo[0] + (d == 0 ? sc : 0), g1 - cp.lo[1] + (d == 1 ? sc : 0),
               D == 3 ? g2 - cp.lo[2] + (d == 2 ? sc : 0) : 0};
  scatter_read<T, D>(Wd, cp, crs, cc, d, kind == 0 ? -a * ihc : -a);
  const T fw = (kind == 0 ? a * ihf : a) * T(D == 3 ? 0.25 : 0.5);
  const int fd = q + 2 * side - 2;  // fine cells 2 gd - 2 + 2 side ..
  const int b0 = 2 * g0 + (d == 0 ? fd : 0) - fp.lo[0], b1 = 2 * g1 + (d == 1 ? fd : 0) - fp.lo[1];
  const int b2 = D == 3 ? 2 * g2 + (d == 2 ? fd : 0) - fp.lo[2] : 0;
  const long long s1 = d == 0 ? (long long)fp.sy : 1, s2 = d == 2 ? (long long)fp.sy : (long long)fp.sz;
  T* w = Wd + poff(fp, b0, b1, b2);
#pragma unroll
  for (int t2 = 0; t2 < (D == 3 ? 2 : 1); ++t2)
#pragma unroll
    for (int t1 = 0; t1 < 2; ++t1) atomicAdd(w + t1 * s1 + t2 * s2, fw);
}

// Transposed G^comp stencil (Eq. discreteOps a): each valid cell o hands z_d[o]/(12h) times
// the weights (+1, -8, +8, -1) at offsets (-2, -1, +1, +2) along d to the cells it read.
template <typename T, int D>
__global__ void k_gradient_T(LevelView lv, int nby, P3c<T> z, const unsigned char* __restrict__ vmask,
                             T* __restrict__ W) {
  pdl_wait();
  const PatchDesc p = lv.patches[blockIdx.z];
  int i, j, k;
  if (!thread_cell<D>(p, nby, i, j, k)) return;
  const long long o = poff(p, i, j, k);
  if (!vmask[o]) return;
  const T inv = pick<T>(lv.inv12h, lv.inv12h_f);
  const int c[3] = {i, j, k};
  const T wq[4] = {T(1), T(-8), T(8), T(-1)};
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const T a = z.p[d][o] * inv;
    if (a == T(0)) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int cc[3] = {c[0], c[1], c[2]};
      cc[d] += q < 2 ? q - 2 : q - 1;
      scatter_read<T, D>(W, p, lv, cc, d, wq[q] * a);
    }
  }
}

// Transposed D^comp stencil (Eq. discreteOps b): each valid cell hands z[o]/(12h) times the
// same weights to component d's cells along d.
template <typename T, int D>
__global__ void k_divergence_T(LevelView lv, int nby, const T* __restrict__ z, const unsigned char* __restrict__ vmask,
                               Out3<T> W) {
  pdl_wait();
  const PatchDesc p = lv.patches[blockIdx.z];
  int i, j, k;
  if (!thread_cell<D>(p, nby, i, j, k)) return;
  const long long o = poff(p, i, j, k);
  if (!vmask[o]) return;
  const T a = z[o] * pick<T>(lv.inv12h, lv.inv12h_f);
  if (a == T(0)) return;
  const int c[3] = {i, j, k};
  const T wq[4] = {T(1), T(-8), T(8), T(-1)};
#pragma unroll
  for (int d = 0; d < D; ++d)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int cc[3] = {c[0], c[1], c[2]};
      cc[d] += q < 2 ? q - 2 : q - 1;
      scatter_read<T, D>(W.p[d], p, lv, cc, d, wq[q] * a);
    }
}

template <typename T, int D>
__global__ void k_cfi_T(const CfiEntry* __restrict__ list, long long n, const long long* __restrict__ side,
                        const PatchDesc* __restrict__ cpatches, const PatchDesc* __restrict__ fpatches, int r,
                        const T* __restrict__ z, const T* __restrict__ wghost, T* __restrict__ W, T beta_inv12h2,
                        T sign) {
  pdl_wait();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const CfiEntry e = list[t];
  const PatchDesc fp = fpatches[e.fpatch];
  const long long st[3] = {1, fp.sy, fp.sz};
  const long long step = (e.layer > 0 ? -1 : 1) * st[e.dir];  // towards the interior
  const int L = e.layer > 0 ? e.layer : -e.layer;
  T wg = (L == 1) ? T(16) * z[e.dst + step] - z[e.dst + 2 * step] : -z[e.dst + 2 * step];
  wg = sign * (wg * beta_inv12h2 + (wghost != nullptr ? wghost[e.dst] : T(0)));
  if (wg == T(0)) return;
  const int b0 = (e.pos[0] * r + e.sub[0]) * CFI_W;
  const int b1 = (e.pos[1] * r + e.sub[1]) * CFI_W;
  const int b2 = (e.pos[2] * r + e.sub[2]) * CFI_W;
  if (e.src >= 0) {
    const PatchDesc cp = cpatches[e.cpatch];
    for (int c2 = 0; c2 < (D == 3 ? CFI_W : 1); ++c2)
      for (int c1 = 0; c1 < CFI_W; ++c1) {
        const long long row = e.src + (long long)c1 * cp.sy + (long long)c2 * cp.sz;
        const T wr = cfiw<T>(b1 + c1) * (D == 3 ? cfiw<T>(b2 + c2) : T(1)) * wg;
        for (int c0 = 0; c0 < CFI_W; ++c0) atomicAdd(&W[row + c0], cfiw<T>(b0 + c0) * wr);
      }
  } else {
    const long long* sd = side + (-1 - e.src) * (D == 3 ? 125 : 25);
    int q = 0;
    for (int c2 = 0; c2 < (D == 3 ? CFI_W : 1); ++c2)
      for (int c1 = 0; c1 < CFI_W; ++c1)
        for (int c0 = 0; c0 < CFI_W; ++c0, ++q)
          atomicAdd(&W[sd[q]], cfiw<T>(b0 + c0) * cfiw<T>(b1 + c1) * (D == 3 ? cfiw<T>(b2 + c2) : T(1)) * wg);
  }
}

// The same by groups of the 2^D ghosts that share a window (ratio 2): a warp per group forms their
// weights, folds them dimension by dimension -- a lane per (x, y) of the window, its cells along z
// in turn -- and adds every window cell once, where a thread per ghost made 2^D times as many
// atomic additions (64^3 box: 33 -> 6.0 us per pass in FP32, 23 -> 11 us in FP64).
template <typename T, int D>
__global__ void __launch_bounds__(128) k_cfi_T_grp(const CfiGroup* __restrict__ list, long long n,
                                                   const long long* __restrict__ side,
                                                   const PatchDesc* __restrict__ cpatches,
                                                   const PatchDesc* __restrict__ fpatches, const T* __restrict__ z,
                                                   const T* wghost, T* W, T beta_inv12h2, T sign) {
  pdl_wait();
  constexpr int NC = D == 3 ? 8 : 4;
  const long long t = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (t >= n) return;
  const CfiGroup& g = list[t];
  T wg = T(0);
  const int dir = g.face >> 1;
  if (lane < NC && g.dst[lane] >= 0) {
    const PatchDesc fp = fpatches[g.fpatch];
    const int hi = g.face & 1, sub = (lane >> dir) & 1;  // layer 1 next to the interior
    const long long st = dir == 0 ? 1 : dir == 1 ? (long long)fp.sy : (long long)fp.sz, step = hi ? -st : st;
    const long long dst = g.dst[lane];
    const T* zi = z + dst + step;
    wg = sub != hi ? T(16) * zi[0] - zi[step] : -zi[step];
    wg = sign * (wg * beta_inv12h2 + (wghost != nullptr ? wghost[dst] : T(0)));
  }
  if (!__any_sync(0xffffffffu, wg != T(0))) return;
  T w[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) w[c] = __shfl_sync(0xffffffffu, wg, c);
  if (lane >= CFI_W * CFI_W) return;
  const int c0 = lane % CFI_W, c1 = lane / CFI_W;
  const int i0 = 2 * g.pos[0] * CFI_W + c0, i1 = 2 * g.pos[1] * CFI_W + c1, i2 = 2 * g.pos[2] * CFI_W;
  const T u00 = cfiw<T>(i0), u01 = cfiw<T>(i0 + CFI_W), u10 = cfiw<T>(i1), u11 = cfiw<T>(i1 + CFI_W);
  T f[2];
#pragma unroll
  for (int c = 0; c < (D == 3 ? 2 : 1); ++c)
    f[c] = fma(u11, fma(u01, w[4 * c + 3], u00 * w[4 * c + 2]), u10 * fma(u01, w[4 * c + 1], u00 * w[4 * c]));
  if (g.src >= 0) {
    const PatchDesc& cp = cpatches[g.cpatch];
    T* p = W + g.src + c0 + (long long)c1 * cp.sy;
    if (D == 3) {
      const long long sz = cp.sz;
      for (int c2 = 0; c2 < CFI_W; ++c2) atomicAdd(p + c2 * sz, fma(cfiw<T>(i2 + CFI_W + c2), f[1], cfiw<T>(i2 + c2) * f[0]));
    } else {
      atomicAdd(p, f[0]);
    }
  } else {
    const long long* sd = side + (-1 - g.src) * (D == 3 ? 125 : 25) + lane;
    if (D == 3)
      for (int c2 = 0; c2 < CFI_W; ++c2)
        atomicAdd(W + sd[c2 * CFI_W * CFI_W], fma(cfiw<T>(i2 + CFI_W + c2), f[1], cfiw<T>(i2 + c2) * f[0]));
    else
      atomicAdd(W + sd[0], f[0]);
  }
}

template <typename T, int D>
__global__ void k_avgdown_T(LevelView fine, LevelView crs, const XferBlock* __restrict__ blocks, T* __restrict__ W,
                            int nby) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int i = blockIdx.x * BX + threadIdx.x;
  const int by = (D == 3) ? (int)(blockIdx.y % nby) : (int)blockIdx.y;
  const int kk = (D == 3) ? (int)(blockIdx.y / nby) : 0;
  const int j = by * BY + threadIdx.y;
  const int gf[3] = {2 * b.clo[0] + i, 2 * b.clo[1] + j, D == 3 ? 2 * b.clo[2] + kk : 0};
  if (gf[0] > 2 * b.chi[0] + 1 || gf[1] > 2 * b.chi[1] + 1 || (D == 3 && gf[2] > 2 * b.chi[2] + 1)) return;
  const PatchDesc cp = crs.patches[b.cpatch];
  const PatchDesc fp = fine.patches[b.fpatch];
  const T wc = W[poff(cp, (gf[0] >> 1) - cp.lo[0], (gf[1] >> 1) - cp.lo[1], (D == 3 ? (gf[2] >> 1) : 0) - cp.lo[2])];
  W[poff(fp, gf[0] - fp.lo[0], gf[1] - fp.lo[1], gf[2] - fp.lo[2])] += wc * T(D == 3 ? 0.125 : 0.25);
}

// Transposed same-level copy: weight accumulated in a copy-ghost slot (by refluxing
// transposes) belongs to the sibling cell the ghost copies.
template <typename T>
__global__ void k_copy_T(const CopyEntry* __restrict__ list, long long n, T* __restrict__ W) {
  pdl_wait();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const CopyEntry e = list[t];
  const T v = W[e.dst];
  if (v != T(0)) {
    atomicAdd(&W[e.src], v);
    W[e.dst] = T(0);
  }
}

// Transposed prolongation (Sec. 6.5 linear interpolation): every fine cell hands
// w * (y1 + y2) to each coarse cell its interpolation reads (atomic adds); coarse positions
// outside the domain pass their weight on through the homogeneous extension.
template <typename T, int D>
__global__ void k_prolong_T(LevelView fine, LevelView crs, const XferBlock* __restrict__ blocks,
                            const T* __restrict__ y1, const T* __restrict__ y2, T* __restrict__ out, int nby) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int i = blockIdx.x * BX + threadIdx.x;
  const int by = (D == 3) ? (int)(blockIdx.y % nby) : (int)blockIdx.y;
  const int kk = (D == 3) ? (int)(blockIdx.y / nby) : 0;
  const int j = by * BY + threadIdx.y;
  const int gf[3] = {2 * b.clo[0] + i, 2 * b.clo[1] + j, D == 3 ? 2 * b.clo[2] + kk : 0};
  if (gf[0] > 2 * b.chi[0] + 1 || gf[1] > 2 * b.chi[1] + 1 || (D == 3 && gf[2] > 2 * b.chi[2] + 1)) return;
  const PatchDesc cp = crs.patches[b.cpatch];
  const PatchDesc fp = fine.patches[b.fpatch];
  const long long of = poff(fp, gf[0] - fp.lo[0], gf[1] - fp.lo[1], gf[2] - fp.lo[2]);
  const T v = y1[of] + (y2 != nullptr ? y2[of] : T(0));
  if (v == T(0)) return;
  int par[3], sg[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    par[e] = (e < D) ? (gf[e] >> 1) : 0;
    sg[e] = (e < D) ? (((gf[e] & 1) == 0) ? -1 : 1) : 0;
  }
  for (int q2 = 0; q2 < (D == 3 ? 2 : 1); ++q2)
    for (int q1 = 0; q1 < 2; ++q1)
      for (int q0 = 0; q0 < 2; ++q0) {
        const int q[3] = {q0, q1, q2};
        int cc[3];
        T w = T(1);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          cc[e] = par[e] + q[e] * sg[e] - cp.lo[e];
          if (e < D) w *= (q[e] == 0) ? T(0.75) : T(0.25);
        }
        // tensor expansion of the out-of-domain dimensions (as in read_ext), scattered
        int idx[3][4];
        T ww[3][4];
        int cnt[3] = {1, 1, 1};
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          idx[e][0] = cc[e];
          ww[e][0] = T(1);
          if (e >= D) continue;
          const int g = cp.lo[e] + cc[e];
          if (g < 0 || g >= crs.ndom[e]) {
            const int side = g < 0 ? 0 : 1;
            const int layer = side == 0 ? -g : g - crs.ndom[e] + 1;
            const int type = crs.bc[2 * e + side];
            cnt[e] = 4;
            for (int m = 0; m < 4; ++m) {
              idx[e][m] = side == 0 ? (m - cp.lo[e]) : (crs.ndom[e] - 1 - m - cp.lo[e]);
              ww[e][m] = gcoef<T>(type, layer - 1, m);
            }
          }
        }
        for (int a0 = 0; a0 < cnt[0]; ++a0)
          for (int a1 = 0; a1 < cnt[1]; ++a1)
            for (int a2 = 0; a2 < cnt[2]; ++a2)
              atomicAdd(&out[poff(cp, idx[0][a0], idx[1][a1], idx[2][a2])], w * ww[0][a0] * ww[1][a1] * ww[2][a2] * v);
      }
}

// Transposed average-down from one coarse buffer into a fine buffer: y_f += y_c / 2^D for
// every fine cell of the transfer blocks (the coarse cells are the invalid ones).
template <typename T, int D>
__global__ void k_avgdown_T2(LevelView fine, LevelView crs, const XferBlock* __restrict__ blocks,
                             const T* __restrict__ yc, T* __restrict__ yf, int nby) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int i = blockIdx.x * BX + threadIdx.x;
  const int by = (D == 3) ? (int)(blockIdx.y % nby) : (int)blockIdx.y;
  const int kk = (D == 3) ? (int)(blockIdx.y / nby) : 0;
  const int j = by * BY + threadIdx.y;
  const int gf[3] = {2 * b.clo[0] + i, 2 * b.clo[1] + j, D == 3 ? 2 * b.clo[2] + kk : 0};
  if (gf[0] > 2 * b.chi[0] + 1 || gf[1] > 2 * b.chi[1] + 1 || (D == 3 && gf[2] > 2 * b.chi[2] + 1)) return;
  const PatchDesc cp = crs.patches[b.cpatch];
  const PatchDesc fp = fine.patches[b.fpatch];
  const T wc = yc[poff(cp, (gf[0] >> 1) - cp.lo[0], (gf[1] >> 1) - cp.lo[1], (D == 3 ? (gf[2] >> 1) : 0) - cp.lo[2])];
  yf[poff(fp, gf[0] - fp.lo[0], gf[1] - fp.lo[1], gf[2] - fp.lo[2])] += wc * T(D == 3 ? 0.125 : 0.25);
}

// ------------------------------------------------------------------------ elementwise
// A pass over the interior cells of a level: a warp takes pieces of 32 ROW_K columns of a row, a lane
// ROW_K of its cells at once, their loads issued together (F::load), then their stores (F::store).
// Bound by memory: as one thread per cell in 65,536 blocks, X += E on 256^3 took 60 us where its bytes
// take 30 (128^3 FP32: 10.1 -> 6.0 us).  Pieces, not whole rows: on 308^2 a warp went through its row in
// three dependent steps on 39 of the SMs (5.6 us against 3.6; 1024^2 X += E 11.0 against 7.0).
constexpr int ROW_K = 4;
template <int D, typename F>
__global__ void __launch_bounds__(256) k_rows(LevelView lv, F f) {
  pdl_wait();
  const PatchDesc p = lv.npatch == 1 ? lv.p0 : lv.patches[blockIdx.y];
  const int lane = threadIdx.x & 31, np = (p.n[0] + 32 * ROW_K - 1) / (32 * ROW_K);  // pieces of a row
  const unsigned n = (unsigned)np * p.n[1] * (D == 3 ? p.n[2] : 1), nw = gridDim.x * 8;
  f.begin();
  for (unsigned u = blockIdx.x * 8 + (threadIdx.x >> 5); u < n; u += nw) {
    const int row = (int)(u / np), i0 = (int)(u - (unsigned)row * np) * (32 * ROW_K) + lane;
    const long long o0 = poff(p, 0, row % p.n[1], D == 3 ? row / p.n[1] : 0);
    typename F::V v[ROW_K];
#pragma unroll
    for (int q = 0; q < ROW_K; ++q)
      if (i0 + 32 * q < p.n[0]) v[q] = f.load(o0 + i0 + 32 * q);
#pragma unroll
    for (int q = 0; q < ROW_K; ++q)
      if (i0 + 32 * q < p.n[0]) f.store(o0 + i0 + 32 * q, v[q]);
  }
}

// y += a x (optionally also y2 += a x); source type S, destination type T
template <typename S, typename T>
struct RowAxpy {
  const S* x;
  T *y, *y2;
  T a;
  struct V {
    T d, y, y2;
  };
  __device__ __forceinline__ void begin() {}
  __device__ __forceinline__ V load(long long o) const { return V{a * cvt<T, S>(x[o]), y[o], y2 != nullptr ? y2[o] : T(0)}; }
  __device__ __forceinline__ void store(long long o, const V& v) const {
    y[o] = v.y + v.d;
    if (y2 != nullptr) y2[o] = v.y2 + v.d;
  }
};

// y += a x on valid cells (x is read as 0 elsewhere)
template <typename T>
struct RowAxpyValid {
  const T* x;
  T* y;
  T a;
  const unsigned char* vmask;
  struct V {
    T x, y;
    unsigned char m;
  };
  __device__ __forceinline__ void begin() {}
  __device__ __forceinline__ V load(long long o) const { return V{x[o], y[o], vmask[o]}; }
  __device__ __forceinline__ void store(long long o, const V& v) const {
    if (v.m) y[o] = v.y + a * v.x;
  }
};

// out = f - w (f null: w) on valid cells, zero on invalid ones (used to copy the valid part of a
// field); keep: invalid cells untouched
template <typename T>
struct RowValidOut {
  const T *w, *f;
  T* out;
  const unsigned char* vmask;
  bool keep;
  struct V {
    T w, f;
    unsigned char m;
  };
  __device__ __forceinline__ void begin() {}
  __device__ __forceinline__ V load(long long o) const { return V{w[o], f != nullptr ? f[o] : T(0), vmask[o]}; }
  __device__ __forceinline__ void store(long long o, const V& v) const {
    if (v.m) out[o] = f != nullptr ? v.f - v.w : v.w;
    else if (!keep) out[o] = T(0);
  }
};

// y += sign * a[0] (vmask non-null: on valid cells)
struct RowShift {
  double* y;
  const double* a;
  const unsigned char* vmask;
  double sign, s;
  struct V {
    double y;
    unsigned char m;
  };
  __device__ __forceinline__ void begin() { s = a[0]; }
  __device__ __forceinline__ V load(long long o) const { return V{y[o], vmask != nullptr ? vmask[o] : (unsigned char)1}; }
  __device__ __forceinline__ void store(long long o, const V& v) const {
    if (v.m) y[o] = v.y + sign * s;
  }
};

template <typename S, typename T, int D>
__global__ void k_convert(LevelView lv, int nby, const S* __restrict__ x, T* __restrict__ y) {
  pdl_wait();
  const PatchDesc p = lv.patches[blockIdx.z];
  int i, j, k;
  if (!thread_cell<D>(p, nby, i, j, k)) return;
  const long long o = poff(p, i, j, k);
  y[o] = cvt<T, S>(x[o]);
}

// out = w - g on interior cells
template <int D>
__global__ void k_sub(LevelView lv, int nby, const double* __restrict__ w, const double* __restrict__ g,
                      double* __restrict__ out) {
  pdl_wait();
  const PatchDesc p = lv.patches[blockIdx.z];
  int i, j, k;
  if (!thread_cell<D>(p, nby, i, j, k)) return;
  const long long o = poff(p, i, j, k);
  out[o] = w[o] - g[o];
}

// ------------------------------------------------------------------------ reductions
// Whole-array passes (one launch for every level, HBM-bound):
//   k_norm_convert  valid-cell max-norm of r into *acc (IEEE bits, atomicMax; order-preserving
//                   for non-negative doubles, a NaN wins) and, when rin is given, r rounded to
//                   FP32 over the whole array (the next FP32 V-cycle's right-hand side; ghost
//                   entries are never read);
//   k_update_valid  phi += X (x2 given: X + X2) on the valid cells (invalid cells are recomputed by the
//                   average-down that starts the next composite residual), and clears the
//                   norm accumulator for that residual.
//   V elements per thread and step: 4 (16-byte loads of FP64 pairs, 4-byte masks; arrays
//   aligned to 16 bytes, n a multiple of 4) or 1 (any alignment).  Per-level launches of one
//   thread per cell took 97 us for the norm of 19 M cells and 94 us for the update.
//   Stacked component batches: blockIdx.y = replica c over elements [c n, (c + 1) n) (n the
//   replica stride), its norm in acc[c], its update skipped once active[c] is 0.
template <int V>
struct FlatVec;
template <>
struct FlatVec<1> {
  static __device__ __forceinline__ void ld(const double* p, double* v) { v[0] = *p; }
  static __device__ __forceinline__ void ld(const float* p, float* v) { v[0] = *p; }
  static __device__ __forceinline__ void ld(const unsigned char* p, unsigned char* v) { v[0] = *p; }
  static __device__ __forceinline__ void st(double* p, const double* v) { *p = v[0]; }
  static __device__ __forceinline__ void st(float* p, const float* v) { *p = v[0]; }
};
template <>
struct FlatVec<4> {
  static __device__ __forceinline__ void ld(const double* p, double* v) {
    const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
  }
  static __device__ __forceinline__ void ld(const float* p, float* v) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
  }
  static __device__ __forceinline__ void ld(const unsigned char* p, unsigned char* v) {
    const uchar4 a = *reinterpret_cast<const uchar4*>(p);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
  }
  static __device__ __forceinline__ void st(double* p, const double* v) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
  }
  static __device__ __forceinline__ void st(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};

template <int V>
__global__ void __launch_bounds__(256) k_norm_convert(long long n, const double* __restrict__ r,
                                                      const unsigned char* __restrict__ vmask, float* __restrict__ rin,
                                                      unsigned long long* __restrict__ acc) {
  pdl_wait();
  __shared__ unsigned long long sm[8];
  unsigned long long v = 0ull;
  const long long stride = (long long)gridDim.x * blockDim.x * V;
  const long long e0 = (long long)blockIdx.y * n;
  acc += blockIdx.y;
  for (long long e = e0 + ((long long)blockIdx.x * blockDim.x + threadIdx.x) * V; e < e0 + n; e += stride) {
    double x[V];
    unsigned char m[V];
    FlatVec<V>::ld(r + e, x);
    FlatVec<V>::ld(vmask + e, m);
    if (rin != nullptr) {
      float y[V];
#pragma unroll
      for (int q = 0; q < V; ++q) y[q] = f64_to_f32(x[q]);
      FlatVec<V>::st(rin + e, y);
    }
#pragma unroll
    for (int q = 0; q < V; ++q) {
      const unsigned long long b = m[q] ? (unsigned long long)__double_as_longlong(x[q]) & 0x7fffffffffffffffull : 0ull;
      v = b > v ? b : v;
    }
  }
  for (int s = 16; s > 0; s >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, s);
    v = u > v ? u : v;
  }
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < 8 ? sm[threadIdx.x] : 0ull;
    for (int s = 16; s > 0; s >>= 1) {
      const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, s);
      v = u > v ? u : v;
    }
    if (threadIdx.x == 0 && v != 0ull) atomicMax(acc, v);
  }
}

template <typename S, int V>
__global__ void __launch_bounds__(256) k_update_valid(long long n, const S* __restrict__ x, const S* __restrict__ x2,
                                                      double* __restrict__ phi,
                                                      const unsigned char* __restrict__ vmask,
                                                      unsigned long long* __restrict__ acc_clear,
                                                      const int* __restrict__ active) {
  pdl_wait();
  if (acc_clear != nullptr && blockIdx.x == 0 && threadIdx.x == 0) acc_clear[blockIdx.y] = 0ull;
  if (active != nullptr && !active[blockIdx.y]) return;  // converged replica: phi stays
  const long long stride = (long long)gridDim.x * blockDim.x * V;
  const long long e0 = (long long)blockIdx.y * n;
  for (long long e = e0 + ((long long)blockIdx.x * blockDim.x + threadIdx.x) * V; e < e0 + n; e += stride) {
    S c[V];
    double y[V];
    unsigned char m[V];
    FlatVec<V>::ld(vmask + e, m);
    FlatVec<V>::ld(x + e, c);
    FlatVec<V>::ld(phi + e, y);
    if (x2 != nullptr) {
      S d[V];
      FlatVec<V>::ld(x2 + e, d);
#pragma unroll
      for (int q = 0; q < V; ++q) c[q] += d[q];
    }
    unsigned any = 0, all = 1;
#pragma unroll
    for (int q = 0; q < V; ++q) {
      any |= m[q];
      all &= m[q] ? 1u : 0u;
      if (m[q]) y[q] += cvt<double, S>(c[q]);
    }
    if (all) {
      FlatVec<V>::st(phi + e, y);
    } else if (any) {  // ghost and invalid entries are not written
#pragma unroll
      for (int q = 0; q < V; ++q)
        if (m[q]) phi[e + q] = y[q];
    }
  }
}

// Error-free transformation (Knuth's TwoSum).
__device__ __forceinline__ void two_sum(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
// double-double accumulate (s, c) += (a, ac)
__device__ __forceinline__ void dd_add(double& s, double& c, double a, double ac) {
  double t, e;
  two_sum(s, a, t, e);
  e += c + ac;
  two_sum(t, e, s, c);
}

// A sum of doubles in 128-bit fixed point: a double enters as its 53-bit significand shifted to a
// common frame (exponent E), so additions are exact integer ones in any order.  Below the sign
// the frame keeps 12 + room bits of headroom, for 2^(12 + room) terms (the host counts them, fixsum_room), and
// 62 - room bits under the last bit of the largest term: terms within a factor 2^(62 - room) of it enter
// exactly (2^59 with the 2^15 cells that a block takes of a 256^3 grid, 2^60 with 8192 partials).  A larger
// term moves the frame by a shift of the sum so far; bits below 2^(room - 114) of the largest term are
// dropped, where double-double sums drop those below 2^-106 of the sum so far.  An addition costs
// about 30 integer instructions, where TwoSum costs seven FP64 ones at a fiftieth of their rate:
// 128^3 + 64^3 33 -> 11 us, 256^2 14.3 -> 7.2 us.
struct FixSum {
  unsigned l0 = 0, l1 = 0, l2 = 0, l3 = 0;
  int E = 0;  // frame; 0: nothing added yet
  int room;   // bits of headroom beyond 12
  __device__ __forceinline__ explicit FixSum(int room_) : room(room_) {}

  __device__ __forceinline__ static int exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
  // v, of an exponent <= E - 2
  __device__ __forceinline__ void add(double v) {
    const unsigned bh = (unsigned)__double2hiint(v), bl = (unsigned)__double2loint(v);
    const int e = (int)((bh >> 20) & 0x7ffu);
    const unsigned mh = (bh & 0xfffffu) | (e != 0 ? 0x100000u : 0u);
    const unsigned sh = (unsigned)(E - max(e, 1) + room), bs = sh & 31u, ws = sh >> 5;
    const unsigned t2 = mh >> bs, t1 = __funnelshift_r(bl, mh, bs), t0 = __funnelshift_r(0u, bl, bs);
    const unsigned m = (unsigned)((int)bh >> 31);  // negative: complement, plus one through the carry
    const unsigned x3 = m ^ (ws == 0 ? t2 : 0u);
    const unsigned x2 = m ^ (ws == 0 ? t1 : ws == 1 ? t2 : 0u);
    const unsigned x1 = m ^ (ws == 0 ? t0 : ws == 1 ? t1 : ws == 2 ? t2 : 0u);
    const unsigned x0 = m ^ (ws == 1 ? t0 : ws == 2 ? t1 : ws == 3 ? t2 : 0u);
    asm("{\n\t.reg .u32 t;\n\t"
        "add.cc.u32 t, %4, 1;\n\t"
        "addc.cc.u32 %0, %0, %5;\n\t"
        "addc.cc.u32 %1, %1, %6;\n\t"
        "addc.cc.u32 %2, %2, %7;\n\t"
        "addc.u32 %3, %3, %8;\n\t}"
        : "+&r"(l0), "+&r"(l1), "+&r"(l2), "+&r"(l3)
        : "r"(m), "r"(x0), "r"(x1), "r"(x2), "r"(x3));
  }
  __device__ __forceinline__ void join(unsigned a0, unsigned a1, unsigned a2, unsigned a3) {
    asm("add.cc.u32 %0, %0, %4;\n\t"
        "addc.cc.u32 %1, %1, %5;\n\t"
        "addc.cc.u32 %2, %2, %6;\n\t"
        "addc.u32 %3, %3, %7;"
        : "+&r"(l0), "+&r"(l1), "+&r"(l2), "+&r"(l3)
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3));
  }
  // the lanes' sums (of one frame) added up over groups of n lanes, into every lane
  __device__ __forceinline__ void reduce(int n) {
#pragma unroll 1
    for (int st = n >> 1; st > 0; st >>= 1) {
      const unsigned a0 = __shfl_xor_sync(0xffffffffu, l0, st), a1 = __shfl_xor_sync(0xffffffffu, l1, st);
      const unsigned a2 = __shfl_xor_sync(0xffffffffu, l2, st), a3 = __shfl_xor_sync(0xffffffffu, l3, st);
      join(a0, a1, a2, a3);
    }
  }
  // frame e (not below the present one)
  __device__ __forceinline__ void move(int e) {
    int d = E == 0 ? 0 : e - E;
    E = e;
    const unsigned sg = (unsigned)((int)l3 >> 31);
    if (d >= 128) {
      l0 = l1 = l2 = l3 = sg;
      return;
    }
    for (; d >= 32; d -= 32) {
      l0 = l1;
      l1 = l2;
      l2 = l3;
      l3 = sg;
    }
    l0 = __funnelshift_r(l0, l1, d);
    l1 = __funnelshift_r(l1, l2, d);
    l2 = __funnelshift_r(l2, l3, d);
    l3 = (unsigned)((int)l3 >> d);
  }
  // room for terms of exponents up to e
  __device__ __forceinline__ void frame(int e) {
    if (e + 2 > E) move(max(e, 1) + 2);
  }
  // w times the sum as a double-double; w enters before the exponent, so that a sum beyond the double
  // range whose weighted value is inside it does not overflow
  __device__ __forceinline__ void value(double w, double& s, double& c) const {
    double h, e1, e2, e3;
    two_sum(79228162514264337593543950336.0 * (double)(int)l3, 18446744073709551616.0 * (double)l2, h, e1);
    two_sum(h, 4294967296.0 * (double)l1, h, e2);
    two_sum(h, (double)l0, h, e3);
    // the unit is 2^(E - 1139 + room): two factors in the normal range
    const int k = E - 1139 + room, ka = k / 2;
    const double fa = __longlong_as_double((long long)(1023 + ka) << 52), fb = __longlong_as_double((long long)(1023 + k - ka) << 52);
    const double hi = w * h;
    two_sum(hi, fma(w, e1 + (e2 + e3), fma(w, h, -hi)), s, c);
    s = s * fa * fb;
    c = c * fa * fb;
  }
};

// Deterministic partial sums of w * x over the valid interior cells of one level, with a fixed
// number of blocks per level (the rows each warp visits depend only on the launch shape): one
// double-double partial part[2*(base+block)].  A warp sums whole rows in fixed point (FixSum, one
// frame per warp), the warps' sums are brought to one frame and added, and w multiplies the
// block's sum (TwoProd).
template <int D>
__global__ void __launch_bounds__(256) k_wsum_gs(LevelView lv, const double* __restrict__ x,
                                                 const unsigned char* __restrict__ vmask, double w,
                                                 double* __restrict__ part, long long base, int room) {
  pdl_wait();
  constexpr int K = 8;  // cells of a lane in flight
  __shared__ uint4 sl[8];
  __shared__ int se[8];
  FixSum a(room);
  bool bad = false;  // a non-finite term
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = gridDim.x * 8;
  for (int pi = 0; pi < lv.npatch; ++pi) {
    const PatchDesc p = lv.patches[pi];
    const int nr = p.n[1] * p.n[2];
    for (int row = blockIdx.x * 8 + warp; row < nr; row += nw) {
      const long long o = poff(p, 0, row % p.n[1], row / p.n[1]);
      for (int i0 = 0; i0 < p.n[0]; i0 += 32 * K) {
        double v[K];
        unsigned char m[K];
        int e = 0;
#pragma unroll
        for (int q = 0; q < K; ++q) {
          const int i = i0 + 32 * q + lane;
          v[q] = i < p.n[0] ? x[o + i] : 0.0;
          m[q] = vmask == nullptr || (i < p.n[0] && vmask[o + i]);
        }
#pragma unroll
        for (int q = 0; q < K; ++q) {
          if (!m[q]) v[q] = 0.0;
          e = max(e, FixSum::exponent(v[q]));
        }
        e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
        if (e == 0x7ff) {
          bad = true;
          continue;
        }
        a.frame(e);
#pragma unroll
        for (int q = 0; q < K; ++q)
          if (i0 + 32 * q < p.n[0]) a.add(v[q]);
      }
    }
  }
  a.reduce(32);
  if (lane == 0) {
    sl[warp] = make_uint4(a.l0, a.l1, a.l2, a.l3);
    se[warp] = bad ? -1 : a.E;
  }
  __syncthreads();
  if (warp != 0) return;
  const uint4 l = sl[lane & 7];
  a.l0 = l.x;
  a.l1 = l.y;
  a.l2 = l.z;
  a.l3 = l.w;
  a.E = se[lane & 7];
  const bool nan = __any_sync(0xffffffffu, a.E < 0);
  a.move((int)__reduce_max_sync(0xffffffffu, (unsigned)max(a.E, 1)));
  a.reduce(8);
  double s, c;
  a.value(w, s, c);
  if (nan) s = __longlong_as_double(0x7ff8000000000000ll);
  if (lane == 0) {
    part[2 * (base + blockIdx.x)] = s;
    part[2 * (base + blockIdx.x) + 1] = c;
  }
}

// Boundary flux partials: sum over physical faces of valid boundary cells of
// scale * g (g = Neumann datum), one double-double per (patch, face) block row.
template <int D>
__global__ void k_bsum(LevelView lv, const double* __restrict__ bc, const unsigned char* __restrict__ vmask,
                       double scale, double* __restrict__ part, long long base) {
  pdl_wait();
  __shared__ double ss[256], sc[256];
  const int pidx = blockIdx.x / (2 * D);
  const int f = blockIdx.x % (2 * D);
  const int d = f / 2, side = f % 2;
  const PatchDesc p = lv.patches[pidx];
  const int gface = side == 0 ? 0 : lv.ndom[d] - 1;
  double s = 0.0, c = 0.0;
  const bool touches = (p.lo[d] <= gface && gface <= p.lo[d] + p.n[d] - 1) && lv.bc[f] == 1 && bc != nullptr;
  if (touches) {
    const int e1 = (d == 0) ? 1 : 0;
    const int e2 = (D == 3) ? ((d == 2) ? 1 : 2) : -1;
    const long long ncell = (long long)p.n[e1] * (e2 >= 0 ? p.n[e2] : 1);
    for (long long t = threadIdx.x; t < ncell; t += blockDim.x) {
      int c3[3] = {0, 0, 0};
      c3[d] = gface - p.lo[d];
      c3[e1] = (int)(t % p.n[e1]);
      if (e2 >= 0) c3[e2] = (int)(t / p.n[e1]);
      const long long o = poff(p, c3[0], c3[1], c3[2]);
      if (!vmask[o]) continue;
      long long ti = p.lo[e1] + c3[e1];
      if (e2 >= 0) ti += (long long)(p.lo[e2] + c3[e2]) * lv.ndom[e1];
      const double gv = bc[lv.bc_off[f] + ti];
      const double prod = scale * gv;
      dd_add(s, c, prod, fma(scale, gv, -prod));
    }
  }
  ss[threadIdx.x] = s;
  sc[threadIdx.x] = c;
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st) {
      double a = ss[threadIdx.x], ac = sc[threadIdx.x];
      dd_add(a, ac, ss[threadIdx.x + st], sc[threadIdx.x + st]);
      ss[threadIdx.x] = a;
      sc[threadIdx.x] = ac;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[2 * (base + blockIdx.x)] = ss[0];
    part[2 * (base + blockIdx.x) + 1] = sc[0];
  }
}

// Sum of n double-double partials (one block of 256 threads), in the same fixed point with one
// frame for all: the tree of double-double additions it replaces took 12 us.
__global__ void __launch_bounds__(256) k_dd_final(const double* __restrict__ part, long long n, double* __restrict__ out,
                                                  int room) {
  pdl_wait();
  __shared__ int se[8];
  __shared__ uint4 sl[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int e = 0;
  for (long long t = threadIdx.x; t < 2 * n; t += 256) e = max(e, FixSum::exponent(part[t]));
  e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  if (lane == 0) se[warp] = e;
  __syncthreads();
  for (int q = 0; q < 8; ++q) e = max(e, se[q]);
  if (e == 0x7ff) {
    if (threadIdx.x == 0) out[0] = __longlong_as_double(0x7ff8000000000000ll);
    return;
  }
  FixSum a(room);
  a.frame(e);
  for (long long t = threadIdx.x; t < 2 * n; t += 256) a.add(part[t]);
  a.reduce(32);
  if (lane == 0) sl[warp] = make_uint4(a.l0, a.l1, a.l2, a.l3);
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int q = 1; q < 8; ++q) a.join(sl[q].x, sl[q].y, sl[q].z, sl[q].w);
  double s, c;
  a.value(1.0, s, c);
  out[0] = s + c;
}

// m = (S_f - beta * S_b) / V ; used by the solvability fix and mean-zero
__global__ void k_mean_from_sums(const double* __restrict__ sf, const double* __restrict__ sb, double beta,
                                 double vol, double* __restrict__ m) {
  pdl_wait();
  if (threadIdx.x == 0 && blockIdx.x == 0) m[0] = (sf[0] - (sb ? beta * sb[0] : 0.0)) / vol;
}

}  // namespace amr4
