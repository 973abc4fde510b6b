// op3d.cuh -- 3-D level operator, residual restriction and prolongation on patches of any size.
//
// The multigrid grids below the tile-multiple ones, ragged boxes and levels of several patches
// are small (1e2 .. 1e6 cells, resident in L2), so a launch lasts as long as one thread's chain
// of dependent work.  These kernels therefore give every cell (or short z run of cells) its own
// thread, read the neighbours straight from L1 / L2 with 32-bit offsets, use no shared memory
// and no barrier, and evaluate the ghost formulas of Eqs. (velBCHomoDiri5th)/(Neumann5) only in
// the lanes next to a domain face, from four inward cells with the coefficients in registers.
#pragma once

#include "kernels.cuh"

namespace amr4 {

// One dimension of the transposed operator (trans_sums) with what does not depend on the plane
// formed once per column: which neighbours exist, and the weights of the two cells next to the
// near face that the cell's rows of the ghost formulas put on it.  Domains of eight cells and
// more, so that a cell is near one face only.  Against the generic kernel of one thread per cell: a
// transposed FP32 sweep of 128^3 22.6 -> 17.6 us, an FP64 application 108 -> 82 us.
template <typename T>
struct TransLine {
  T a, b;          // ex += a x[f] + b x[f + s]
  int f, s;        // offset of the face cell from the cell; step into the domain
  bool near, m1, p1, m2, p2;
  __device__ __forceinline__ TransLine(int g, int n, int plo, int pn, int st, int tlo, int thi) {
    m1 = g >= 1;
    p1 = g + 1 < n;
    m2 = g >= 2;
    p2 = g + 2 < n;
    const bool low = g <= 3 && plo == 0, high = n - 1 - g <= 3 && plo + pn == n;
    near = g < 4 || n - 1 - g < 4;
    a = b = T(0);
    f = s = 0;
    if (low || high) {
      const int m = low ? g : n - 1 - g, t = low ? tlo : thi;
      const T c0 = gcoef<T>(t, 0, m), c1 = gcoef<T>(t, 1, m);
      a = T(16) * c0 - c1;
      b = -c0;
      s = low ? st : -st;
      f = -m * s;
    }
  }
  __device__ __forceinline__ void sums(const T* __restrict__ xb, int o, int st, T& s1, T& s2, T& ex) const {
    if constexpr (sizeof(T) == 8) {  // adds once for both kinds of lane: the FP64 rate bounds the pass
      const T v1 = m1 ? xb[o - st] : T(0), w1 = p1 ? xb[o + st] : T(0), v2 = m2 ? xb[o - 2 * st] : T(0),
              w2 = p2 ? xb[o + 2 * st] : T(0);
      s1 = v1 + w1;
      s2 = v2 + w2;
      if (near) ex = fma(a, xb[o + f], fma(b, xb[o + f + s], ex));
      return;
    }
    if (!near) {
      s1 = xb[o - st] + xb[o + st];
      s2 = xb[o - 2 * st] + xb[o + 2 * st];
      return;
    }
    const T v1 = m1 ? xb[o - st] : T(0), w1 = p1 ? xb[o + st] : T(0), v2 = m2 ? xb[o - 2 * st] : T(0),
            w2 = p2 ? xb[o + 2 * st] : T(0);
    s1 = v1 + w1;
    s2 = v2 + w2;
    ex = fma(a, xb[o + f], fma(b, xb[o + f + s], ex));
  }
};

// Level operator (OP_APPLY, OP_RESID, OP_JACOBI, OP_JACOBI0; homogeneous data; TR: its transpose).  A thread owns
// one (x, y) column of a patch -- columns numbered linearly, so narrow grids fill their warps --
// and kz planes of it, its z neighbours in a register queue.  The host sizes kz so that small
// grids spread over every SM (kz = 1 on the coarsest) and large ones keep the queue.
// Replaces a shared-memory marching kernel with a barrier and 64-bit ghost code per plane, which
// took 10 us on every FP32 grid down to 6 x 5 x 4 cells and 34 us per FP64 sweep of 72^3.
// Results that leave the library (OP_APPLY, OP_RESID, the sweeps of amr_smooth) form L x from the
// neighbour sums first (``lap``) and add alpha x to it: with the coefficients folded as in the V-cycle's
// sweeps, alpha - 90 kc2 is rounded once for all cells and f - A x of a Helmholtz system (small beta) has
// twice the error (72^3, N(0,1) fields: rms 8.9e-17 and 1.6e-16, largest 7.1e-16 and 1.5e-15).  Levels
// that the tile kernels (k_level_op3d_zc, k_sweep3d) also serve keep their folded form, bit for bit
// (lap = 0), and so do the V-cycle's FP64 sweeps, whose FP64 rate it saves (144^3 solve 7.52 against 7.83 ms).  With
// the restriction, prolongation and bottom solve below, the FP64 Helmholtz solve on 72^3 + a
// 56 x 52 x 72 box went from 6.05 to 2.95 ms and the mixed pressure solve on 96 x 80 x 64 with two
// ragged boxes from 10.1 to 5.8 ms.
// FP32 at 64 registers, the 32 warps per SM that the host counts on: left free, the transposed sweep takes
// 80 and 23.6 us on 128^3 instead of 17.6, the mixed solve on 144^3 2137 instead of 2021 us.  FP64 has no
// bound (0: its transposed application of 128^3 takes 82 us, at 80 registers 86; a bound of one block makes
// the compiler take more registers, 72^3 solve 1165 -> 1184 us).
template <typename T, int MODE, bool TR>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 8 : 0) k_level_op3d_col(LevelView lv, int kz, const T* __restrict__ x,
                                                        const T* f, T* out, T alpha, T beta,
                                                        const __grid_constant__ JFac<T, 3> jf,
                                                        const unsigned char* __restrict__ vmask, int lap) {
  const int pz = blockIdx.z;
  const PatchDesc p = lv.npatch == 1 ? lv.p0 : lv.patches[pz];
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  const int k0 = blockIdx.y * kz, k1 = min(k0 + kz, p.n[2]);
  if (col >= p.n[0] * p.n[1] || k0 >= k1) {
    pdl_wait();
    return;
  }
  const int i = col % p.n[0], j = col / p.n[0];
  const int sy = (int)p.sy, sz = (int)p.sz;
  const int gx = p.lo[0] + i, gy = p.lo[1] + j, lz = p.lo[2], nzd = lv.ndom[2];
  const int cx = face_class(gx, lv.ndom[0]), cy = face_class(gy, lv.ndom[1]);
  // transposed: small domains take trans_sums plane by plane
  const bool wide = TR && lv.ndom[0] >= 8 && lv.ndom[1] >= 8;
  const TransLine<T> tx(gx, lv.ndom[0], p.lo[0], p.n[0], 1, lv.bc[0], lv.bc[1]);
  const TransLine<T> ty(gy, lv.ndom[1], p.lo[1], p.n[1], sy, lv.bc[2], lv.bc[3]);
  const T* __restrict__ xb = x + p.off;
  const T* fb = f + p.off;  // may be out (in-place residual)
  T* ob = out + p.off;
  const unsigned char* __restrict__ vb = (MODE == OP_RESID && vmask != nullptr) ? vmask + p.off : nullptr;
  int o = (k0 + NG) * sz + (j + NG) * sy + i + NG;
  pdl_wait();
  if (MODE == OP_JACOBI0) {
    for (int k = k0; k < k1; ++k, o += sz) ob[o] = jf.w[cx + 5 * cy + 25 * face_class(lz + k, nzd)] * fb[o];
    return;
  }
  const T inv = pick<T>(lv.inv12h2, lv.inv12h2_f);
  const T kc2 = beta * inv, kc1 = T(16) * kc2, kc0 = alpha - T(90) * kc2;
  T q0, q1, q2, q3;
  q2 = xb[o];
  q3 = (lz + k0 + 1 < nzd) ? xb[o + sz] : T(0);
  q0 = (lz + k0 - 2 >= 0) ? xb[o - 2 * sz] : T(0);
  q1 = (lz + k0 - 1 >= 0) ? xb[o - sz] : T(0);
#pragma unroll 2
  for (int k = k0; k < k1; ++k, o += sz) {
    const int gz = lz + k;
    const int cz = face_class(gz, nzd);
    const T q4 = (gz + 2 < nzd) ? xb[o + 2 * sz] : T(0);
    T fk = T(0);
    if (MODE != OP_APPLY) fk = fb[o];
    T x1, x2, y1, y2, z1, z2, ex = T(0);
    if (TR) {
      if (wide) {
        tx.sums(xb, o, 1, x1, x2, ex);
        ty.sums(xb, o, sy, y1, y2, ex);
      } else {
        trans_sums<T>(xb, o, 1, i, lv.ndom[0], p.lo[0], p.n[0], lv.bc[0], lv.bc[1], x1, x2, ex);
        trans_sums<T>(xb, o, sy, j, lv.ndom[1], p.lo[1], p.n[1], lv.bc[2], lv.bc[3], y1, y2, ex);
      }
      if (gz >= 4 && gz <= nzd - 5) {
        z1 = q1 + q3;
        z2 = q0 + q4;
      } else {
        trans_sums<T>(xb, o, sz, k, nzd, lz, p.n[2], lv.bc[4], lv.bc[5], z1, z2, ex);
      }
    } else {
      line_sums<T>(xb, o, 1, cx == 0, gx, lv.ndom[0], lv.bc[0], lv.bc[1], x1, x2);
      line_sums<T>(xb, o, sy, cy == 0, gy, lv.ndom[1], lv.bc[2], lv.bc[3], y1, y2);
      if (cz == 0) {
        z1 = q1 + q3;
        z2 = q0 + q4;
      } else {
        face_sums<T>(xb, o, sz, gz, nzd, lv.bc[4], lv.bc[5], z1, z2);
      }
    }
    const T s1 = (x1 + y1) + z1;
    const T s2 = (x2 + y2) + z2;
    if (vb == nullptr || vb[o]) {
      // FP32 and transposed sweeps belong to V-cycles only (the choice alone costs an FP32 sweep 12 %)
      if (MODE == OP_JACOBI ? (sizeof(T) == 8 && !TR && lap) : (TR || lap)) {
        T l = fma(T(-90), q2, fma(T(16), s1, -s2));
        if (TR) l += ex;
        const T ax = fma(alpha, q2, kc2 * l);
        ob[o] = MODE == OP_APPLY ? ax : MODE == OP_RESID ? fk - ax : fma(jf.w[cx + 5 * cy + 25 * cz], fk - ax, q2);
      } else if (MODE == OP_APPLY) {
        ob[o] = kc0 * q2 + (kc1 * s1 - kc2 * s2);
      } else {
        T r = fma(kc2, s2, fma(-kc1, s1, fma(-kc0, q2, fk)));
        if (TR) r = fma(-kc2, ex, r);
        if (MODE == OP_RESID) ob[o] = r;
        else ob[o] = fma(jf.w[cx + 5 * cy + 25 * cz], r, q2);
      }
    }
    q0 = q1;
    q1 = q2;
    q2 = q3;
    q3 = q4;
  }
}

// ------------------------------------------------------------------------ level 0 around the refined region
// In a composite V-cycle the correction on level 0 is zero before the level-0 multigrid except
// under the level-1 boxes, where it is the average of the fine correction.  The level-0
// residual r - A x then equals r outside the boxes grown by three cells (two for the stencil,
// one more because a ghost formula reaches four cells inward).  These passes visit only that
// region (70^3 of 256^3 cells on the benchmark's hierarchy) instead of whole fields, of which the
// level-0 residual alone took 55 us.
constexpr int RGN_RESID = 3;  // cells around a box where the residual differs from r
constexpr int RGN_READ = 5;   // cells around a box that the residual or the AMRCFI windows read

// cell of region t of transfer block b grown by ``grow`` cells, clipped to the domain
template <int D>
__device__ __forceinline__ bool region_cell(const LevelView& lv, const XferBlock& b, int grow, long long t, int g[3]) {
  int lo[3] = {0, 0, 0}, w[3] = {1, 1, 1};
#pragma unroll
  for (int d = 0; d < D; ++d) {
    lo[d] = max(b.clo[d] - grow, 0);
    w[d] = min(b.chi[d] + grow, lv.ndom[d] - 1) - lo[d] + 1;
  }
  if (t >= (long long)w[0] * w[1] * w[2]) return false;
  const unsigned u = (unsigned)t;
  g[0] = lo[0] + (int)(u % w[0]);
  g[1] = lo[1] + (int)((u / w[0]) % w[1]);
  g[2] = lo[2] + (int)(u / ((unsigned)w[0] * w[1]));
  return true;
}

// x = 0 and keep = r on the regions grown by RGN_READ (r may be overwritten there afterwards;
// idempotent where regions overlap)
template <typename T, int D>
__global__ void __launch_bounds__(256) k_region_begin(LevelView lv, const XferBlock* __restrict__ blocks,
                                                      const T* __restrict__ r, T* __restrict__ x, T* __restrict__ keep) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.y];
  int g[3];
  if (!region_cell<D>(lv, b, RGN_READ, (long long)blockIdx.x * 256 + threadIdx.x, g)) return;
  const PatchDesc p = lv.npatch == 1 ? lv.p0 : lv.patches[b.cpatch];
  const long long o = poff(p, g[0] - p.lo[0], g[1] - p.lo[1], D == 3 ? g[2] - p.lo[2] : 0);
  x[o] = T(0);
  keep[o] = r[o];
}

// r = keep - A x on the valid cells of the regions grown by RGN_RESID
template <typename T, int D>
__global__ void __launch_bounds__(256) k_region_resid(LevelView lv, const XferBlock* __restrict__ blocks,
                                                      const T* __restrict__ x, const T* __restrict__ keep,
                                                      T* __restrict__ r, const unsigned char* __restrict__ vmask, T alpha,
                                                      T beta) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.y];
  int g[3];
  if (!region_cell<D>(lv, b, RGN_RESID, (long long)blockIdx.x * 256 + threadIdx.x, g)) return;
  const PatchDesc p = lv.npatch == 1 ? lv.p0 : lv.patches[b.cpatch];
  const long long og = poff(p, g[0] - p.lo[0], g[1] - p.lo[1], D == 3 ? g[2] - p.lo[2] : 0);
  if (!vmask[og]) return;
  const T* __restrict__ xb = x + p.off;
  const int o = (int)(og - p.off);
  const T inv = pick<T>(lv.inv12h2, lv.inv12h2_f);
  const T kc2 = beta * inv, kc1 = T(16) * kc2, kc0 = alpha - T(30 * D) * kc2;
  T a1, a2, s1 = T(0), s2 = T(0);
  line_sums<T>(xb, o, 1, face_class(g[0], lv.ndom[0]) == 0, g[0], lv.ndom[0], lv.bc[0], lv.bc[1], a1, a2);
  s1 += a1;
  s2 += a2;
  line_sums<T>(xb, o, (int)p.sy, face_class(g[1], lv.ndom[1]) == 0, g[1], lv.ndom[1], lv.bc[2], lv.bc[3], a1, a2);
  s1 += a1;
  s2 += a2;
  if (D == 3) {
    line_sums<T>(xb, o, (int)p.sz, face_class(g[2], lv.ndom[2]) == 0, g[2], lv.ndom[2], lv.bc[4], lv.bc[5], a1, a2);
    s1 += a1;
    s2 += a2;
  }
  r[og] = fma(kc2, s2, fma(-kc1, s1, fma(-kc0, xb[o], keep[og])));
}

// copy (add = 0) or add (add = 1) src into dst on the regions grown by ``grow``; adding is
// done on the boxes themselves only (grow = 0: disjoint)
template <typename T, int D>
__global__ void __launch_bounds__(256) k_region_move(LevelView lv, const XferBlock* __restrict__ blocks, int grow,
                                                     const T* __restrict__ src, T* __restrict__ dst, int add) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.y];
  int g[3];
  if (!region_cell<D>(lv, b, grow, (long long)blockIdx.x * 256 + threadIdx.x, g)) return;
  const PatchDesc p = lv.npatch == 1 ? lv.p0 : lv.patches[b.cpatch];
  const long long o = poff(p, g[0] - p.lo[0], g[1] - p.lo[1], D == 3 ? g[2] - p.lo[2] : 0);
  if (add) dst[o] += src[o];
  else dst[o] = src[o];
}

// Residual restriction: eight lanes per coarse cell, one per child, instead of one thread for
// all eight (the chain of 8 x 13 loads took 15 us on every grid, 53 us in FP64 on a 72^3 one).
// Each lane forms its child's residual with cell_Lx's arithmetic; lane 0's sum adds them in
// cell_restrict's order, so the result is bit for bit the one-thread form's.  A warp holds
// four coarse cells along x: the loads of a row of eight children are contiguous.
template <typename T>
__global__ void __launch_bounds__(256) k_restrict3d_resid(LevelView fine, LevelView crs,
                                                          const XferBlock* __restrict__ blocks,
                                                          const T* __restrict__ xf, const T* __restrict__ ff,
                                                          T* __restrict__ outc, T alpha, T beta) {
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int w0 = b.chi[0] - b.clo[0] + 1, w1 = b.chi[1] - b.clo[1] + 1, w2 = b.chi[2] - b.clo[2] + 1;
  const int lane = threadIdx.x & 31, child = lane & 7;
  // coarse cells of a warp: four along x (the last group of a row may be short)
  const int gw = (w0 + 3) / 4;
  const int grp = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (grp >= gw * w1 * w2) return;
  const int ci = (grp % gw) * 4 + (lane >> 3), cj = (grp / gw) % w1, ck = grp / (gw * w1);
  const bool act = ci < w0;
  const PatchDesc cp = crs.patches[b.cpatch];
  const PatchDesc fp = fine.patches[b.fpatch];
  const int g0 = b.clo[0] + ci, g1 = b.clo[1] + cj, g2 = b.clo[2] + ck;
  T r = T(0);
  if (act) {
    const int sy = (int)fp.sy, sz = (int)fp.sz;
    const int fx = 2 * g0 + (child & 1), fy = 2 * g1 + ((child >> 1) & 1), fz = 2 * g2 + (child >> 2);
    const int o = (fz - fp.lo[2] + NG) * sz + (fy - fp.lo[1] + NG) * sy + (fx - fp.lo[0] + NG);
    const T* __restrict__ xb = xf + fp.off;
    const T fk = ff[fp.off + o], xc = xb[o];
    const int n0 = fine.ndom[0], n1 = fine.ndom[1], n2 = fine.ndom[2];
    T x1, x2, y1, y2, z1, z2;
    line_sums<T>(xb, o, 1, face_class(fx, n0) == 0, fx, n0, fine.bc[0], fine.bc[1], x1, x2);
    line_sums<T>(xb, o, sy, face_class(fy, n1) == 0, fy, n1, fine.bc[2], fine.bc[3], y1, y2);
    line_sums<T>(xb, o, sz, face_class(fz, n2) == 0, fz, n2, fine.bc[4], fine.bc[5], z1, z2);
    const T s1 = (x1 + y1) + z1, s2 = (x2 + y2) + z2;
    const T inv = pick<T>(fine.inv12h2, fine.inv12h2_f);
    const T s = (T(16) * s1 - s2 - T(90) * xc) + T(0);
    r = fk - (alpha * xc + beta * (s * inv));
  }
  T acc = T(0);
#pragma unroll
  for (int c = 0; c < 8; ++c) acc += __shfl_sync(0xffffffffu, r, (lane & 24) + c);
  if (act && child == 0)
    outc[cp.off + (long long)(g2 - cp.lo[2] + NG) * cp.sz + (long long)(g1 - cp.lo[1] + NG) * cp.sy + (g0 - cp.lo[0] + NG)] =
        acc * T(0.125);
}

// Prolongation by coarse parent on any grid: one thread per coarse cell gathers the 27 coarse
// values around it, with the homogeneous layer-1 extension where the neighbourhood leaves the
// domain (dimension after dimension, Fig. 1(c); four inward cells per dimension instead of
// three), and updates its eight children.
// Replaces one thread per fine cell with the face cells' 64-term products inline: 143 us for
// an FP64 72^3 grid, 45 us for 36^3.
template <typename T>
__device__ __forceinline__ void ext_row(const T* __restrict__ cb, int o, int st, bool lo, bool hi, const T* __restrict__ glo,
                                        const T* __restrict__ ghi, T& a, T& b, T& c) {
  b = cb[o];
  if (!lo) a = cb[o - st];
  if (!hi) c = cb[o + st];
  if (lo) a = fma(glo[3], cb[o + 3 * st], fma(glo[2], cb[o + 2 * st], fma(glo[1], c, glo[0] * b)));
  if (hi) c = fma(ghi[3], cb[o - 3 * st], fma(ghi[2], cb[o - 2 * st], fma(ghi[1], a, ghi[0] * b)));
}

template <typename T>
__global__ void __launch_bounds__(128) k_prolong3d_ext(LevelView fine, LevelView crs, const XferBlock* __restrict__ blocks,
                                                       const T* __restrict__ xc, T* __restrict__ xf, T* __restrict__ xf2) {
  using V2 = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
  pdl_wait();
  const XferBlock b = blocks[blockIdx.z];
  const int w0 = b.chi[0] - b.clo[0] + 1, w1 = b.chi[1] - b.clo[1] + 1;
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  const int g2 = b.clo[2] + (int)blockIdx.y;
  if (col >= w0 * w1 || g2 > b.chi[2]) return;
  const int g0 = b.clo[0] + col % w0, g1 = b.clo[1] + col / w0;
  const PatchDesc cp = crs.patches[b.cpatch];
  const PatchDesc fp = fine.patches[b.fpatch];
  const int fsy = (int)fp.sy, fsz = (int)fp.sz;
  const long long of = fp.off + (long long)(2 * g2 - fp.lo[2] + NG) * fsz + (long long)(2 * g1 - fp.lo[1] + NG) * fsy +
                       (2 * g0 - fp.lo[0] + NG);
  V2 fv[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) fv[q] = *reinterpret_cast<const V2*>(xf + of + (q >> 1) * fsz + (q & 1) * fsy);
  const T* __restrict__ cb = xc + cp.off;
  const int csy = (int)cp.sy, csz = (int)cp.sz;
  const int oc = (g2 - cp.lo[2] + NG) * csz + (g1 - cp.lo[1] + NG) * csy + (g0 - cp.lo[0] + NG);
  const bool xl = g0 == 0, xh = g0 == crs.ndom[0] - 1, yl = g1 == 0, yh = g1 == crs.ndom[1] - 1, zl = g2 == 0,
             zh = g2 == crs.ndom[2] - 1;
  T c[3][3][3];  // [dz + 1][dy + 1][dx + 1]
  if (!(xl || xh || yl || yh || zl || zh)) {
#pragma unroll
    for (int dz = 0; dz < 3; ++dz)
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) c[dz][dy][dx] = cb[oc + (dz - 1) * csz + (dy - 1) * csy + (dx - 1)];
  } else {
    // layer-1 ghost coefficients of the two faces of each dimension
    T gx[2][4], gy[2][4], gz[2][4];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        gx[s][m] = gcoef<T>(crs.bc[s], 0, m);
        gy[s][m] = gcoef<T>(crs.bc[2 + s], 0, m);
        gz[s][m] = gcoef<T>(crs.bc[4 + s], 0, m);
      }
    // one plane: its three rows (extended in x), the outer ones extended in y
    auto plane = [&](int op, T pl[3][3]) {
      ext_row<T>(cb, op, 1, xl, xh, gx[0], gx[1], pl[1][0], pl[1][1], pl[1][2]);
      if (!yl) ext_row<T>(cb, op - csy, 1, xl, xh, gx[0], gx[1], pl[0][0], pl[0][1], pl[0][2]);
      if (!yh) ext_row<T>(cb, op + csy, 1, xl, xh, gx[0], gx[1], pl[2][0], pl[2][1], pl[2][2]);
      if (yl || yh) {
        const int d = yl ? csy : -csy;
        const T h0 = yl ? gy[0][0] : gy[1][0], h1 = yl ? gy[0][1] : gy[1][1], h2 = yl ? gy[0][2] : gy[1][2],
                h3 = yl ? gy[0][3] : gy[1][3];
        T r2[3], r3[3];
        ext_row<T>(cb, op + 2 * d, 1, xl, xh, gx[0], gx[1], r2[0], r2[1], r2[2]);
        ext_row<T>(cb, op + 3 * d, 1, xl, xh, gx[0], gx[1], r3[0], r3[1], r3[2]);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const T fr = yl ? pl[2][q] : pl[0][q];
          const T v = fma(h3, r3[q], fma(h2, r2[q], fma(h1, fr, h0 * pl[1][q])));
          if (yl) pl[0][q] = v;
          else pl[2][q] = v;
        }
      }
    };
    plane(oc, c[1]);
    if (!zl) plane(oc - csz, c[0]);
    if (!zh) plane(oc + csz, c[2]);
    if (zl || zh) {
      const int d = zl ? csz : -csz;
      T p2[3][3], p3[3][3];
      plane(oc + 2 * d, p2);
      plane(oc + 3 * d, p3);
      const T h0 = zl ? gz[0][0] : gz[1][0], h1 = zl ? gz[0][1] : gz[1][1], h2 = zl ? gz[0][2] : gz[1][2],
              h3 = zl ? gz[0][3] : gz[1][3];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const T fr = zl ? c[2][a][q] : c[0][a][q];
          const T v = fma(h3, p3[a][q], fma(h2, p2[a][q], fma(h1, fr, h0 * c[1][a][q])));
          if (zl) c[0][a][q] = v;
          else c[2][a][q] = v;
        }
    }
  }
#pragma unroll
  for (int cz = 0; cz < 2; ++cz)
#pragma unroll
    for (int cy = 0; cy < 2; ++cy) {
      T v[2];
#pragma unroll
      for (int cx = 0; cx < 2; ++cx) {
        const int sx = cx ? 1 : -1, sy = cy ? 1 : -1, sz = cz ? 1 : -1;
        T a = T(0);
#pragma unroll
        for (int q2 = 0; q2 < 2; ++q2)
#pragma unroll
          for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
            for (int q0 = 0; q0 < 2; ++q0) {
              const T w = ((T(1) * (q0 == 0 ? T(0.75) : T(0.25))) * (q1 == 0 ? T(0.75) : T(0.25))) *
                          (q2 == 0 ? T(0.75) : T(0.25));
              a += w * c[1 + q2 * sz][1 + q1 * sy][1 + q0 * sx];
            }
        v[cx] = a;
      }
      const long long oo = of + cz * fsz + cy * fsy;
      V2 t = fv[2 * cz + cy];
      t.x += v[0];
      t.y += v[1];
      *reinterpret_cast<V2*>(xf + oo) = t;
      if (xf2 != nullptr) {
        V2 u = *reinterpret_cast<const V2*>(xf2 + oo);
        u.x += v[0];
        u.y += v[1];
        *reinterpret_cast<V2*>(xf2 + oo) = u;
      }
    }
}

// Bottom solve x = Minv b with one warp per row (the bordered Neumann systems use the leading
// n x n block).  One block for all rows read the 4 MB inverse of a 729-cell bottom grid through
// one SM: 279 us; spread over the chip it is one L2 read of the inverse.
template <typename T>
__global__ void __launch_bounds__(128) k_bottom_rows(const double* __restrict__ minv, int n, int ld, PatchDesc p,
                                                     const T* __restrict__ b, T* __restrict__ x, long long cstride) {
  const int row = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  p.off += blockIdx.y * cstride;  // stacked component batches: one grid row per replica
  pdl_wait();
  if (row >= n) return;
  auto at = [&](int t) -> long long {
    const int i = t % p.n[0], jk = t / p.n[0];
    return p.off + (long long)(i + NG) + (long long)(jk % p.n[1] + NG) * p.sy +
           (p.sz ? (long long)(jk / p.n[1] + NG) * p.sz : 0ll);
  };
  const double* __restrict__ m = minv + (long long)row * ld;
  double acc = 0.0;
  for (int q = lane; q < n; q += 32) acc = fma(m[q], (double)b[at(q)], acc);
  for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
  if (lane == 0) x[at(row)] = T(acc);
}

}  // namespace amr4
