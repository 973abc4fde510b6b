// mgcluster.cuh -- the coarse end of the level-0 multigrid in one thread-block cluster, every
// array in distributed shared memory.
//
// On grids of a few thousand cells a V-cycle phase (sweep, restriction, prolongation) is over in
// less time than a launch takes, and in FP64 one block cannot hold the work either (two FP64
// multiply-adds per clock and SM).  One cluster of up to 16 blocks runs all phases of the grids
// m0 .. M: each grid's slowest dimension (rows in 2-D, planes in 3-D) is cut into slabs, a block
// keeps its slabs of x, t and b in shared memory and reads the neighbours' edge slabs through
// the cluster's shared-memory window; phases are separated by the hardware cluster barrier.
//
// No ghost values are stored: along each dimension the operator is a band of five (transposed:
// six) coefficients per distance class of the cell to the domain faces -- the interior stencil,
// or the interior stencil with Eqs. (velBCHomoDiri5th)/(Neumann5) substituted (transposed: the
// columns of that) -- so every cell runs the same multiply-adds with no branch and no ghost pass
// or barrier between sweeps, forward and adjoint alike.
//
// Bound by the phases' latency (cluster barrier, remote loads, one chain of multiply-adds: about
// 1 us each).  FP64 Poisson solve on 64^2, 23 V-cycles of 45 launches before: 7.65 -> 1.97 ms;
// three-level FP64 projection and its adjoint 22.6 -> 15.3 ms; mixed pressure solve on 96 x 80 x
// 64 with ragged boxes 5.6 -> 5.1 ms; FP32 16^3 .. 4^3 in one block took 47 us a cycle.
#pragma once

#include "coarse3d.cuh"
#include "op3d.cuh"

namespace amr4 {

constexpr int MC_MAX = 7;        // grids of one cluster V-cycle
constexpr int MC_THREADS = 512;  // threads per block
constexpr int MC_BOT = 256;      // largest bottom grid (the dense solve is FP64-bound beyond)

__device__ __forceinline__ void mc_sync() {
  __syncwarp();  // the barrier's aligned form takes whole warps
  cluster_barrier();
}

template <typename T, int D>
struct MgCluster {
  static constexpr int NWT = D == 3 ? 125 : 25;
  int ng, nu1, nu2, nbot, ldb;
  const double* minv;     // bottom inverse (transposed for adjoint cycles)
  PatchDesc gp;           // layout of grid 0's right-hand side and correction
  long long cstride;      // stacked component batches: one cluster per replica, this many elements apart
  int n[MC_MAX][3];
  int R[MC_MAX];          // slabs per block
  int mul[MC_MAX];        // slab k belongs to block (k * mul) >> 16
  int off[MC_MAX];        // element offset of the grid's arrays in shared memory
  T kc[MC_MAX];           // beta / (12 h^2)
  T wt[MC_MAX][NWT];      // Jacobi factors omega / diag by class
  T band[3][9][6];        // 12 h^2 times the 1-D operator: class 0 interior (cells -2 .. 3), 1 + q: cell q from
                          // the low face (cells 0 .. 5), 5 + q: cell q from the high face (cells n-1 .. n-6)
  T ghost[6][4];          // layer-1 ghost coefficients per face (prolongation's extension)
  T alpha;
};

template <typename T, int D, bool TR>
struct MgClusterRun {
  static constexpr int NW = TR ? 6 : 5;  // band width
  static constexpr int NF = TR ? 4 : 2;  // cells per face with a band of their own
  const MgCluster<T, D>& c;
  T* sm;
  const T* band;  // shared copies
  const T* wt;
  const T* gh;
  int rank;

  __device__ __forceinline__ T* arr(int g, int a) const {
    return sm + c.off[g] + a * c.R[g] * (c.n[g][0] * (D == 3 ? c.n[g][1] : 1));
  }
  // slab k of array a of grid g, wherever it lives
  __device__ __forceinline__ T* slab(int g, int a, int k) const {
    const int P = c.n[g][0] * (D == 3 ? c.n[g][1] : 1);
    const int ow = (k * c.mul[g]) >> 16;
    T* l = arr(g, a) + (k - ow * c.R[g]) * P;
    if (ow == rank) return l;
    unsigned long long r;
    asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<unsigned long long>(l)), "r"(ow));
    return reinterpret_cast<T*>(r);
  }
  __device__ __forceinline__ int slabs(int g) const {  // of this block
    return max(0, min(c.R[g], c.n[g][D - 1] - rank * c.R[g]));
  }
  // band class of cell i of n; start and step of its window
  __device__ __forceinline__ int window(int i, int n, int& start, int& step) const {
    if (i < NF) {
      start = 0;
      step = 1;
      return 1 + i;
    }
    if (i >= n - NF) {
      start = n - 1;
      step = -1;
      return 5 + (n - 1 - i);
    }
    start = i - 2;
    step = 1;
    return 0;
  }
  // f(local index, i, j, k) for this block's cells of grid g
  template <typename F>
  __device__ __forceinline__ void cells(int g, F&& f) const {
    const int n0 = c.n[g][0], n1 = D == 3 ? c.n[g][1] : 1, P = n0 * n1, nc = slabs(g) * P;
    for (int q = threadIdx.x; q < nc; q += MC_THREADS) {
      const int s = q / P, r = q - s * P, j = D == 3 ? r / n0 : 0, i = r - j * n0;
      f(q, i, j, s + rank * c.R[g]);
    }
  }
  // One cell of the operator: its windows in array 0 (array 1 lies R P elements further), band
  // rows, right-hand side and Jacobi factor, set up once per grid and leg.
  struct Cell {
    const T* own;        // the cell in array 0
    const T* wx[D];      // band rows
    int st[D], sp[D];    // window start relative to the cell and step (elements), all but the slab dimension
    const T* sl[NW];     // window cells along the slab dimension
    T b, f;
  };
  __device__ __forceinline__ Cell cell(int g, int q, int i, int j, int k) const {
    Cell c_;
    const int n0 = c.n[g][0];
    c_.own = arr(g, 0) + q;
    int st, sp;
    c_.wx[0] = band + 6 * window(i, n0, st, sp);
    c_.st[0] = st - i;
    c_.sp[0] = sp;
    if (D == 3) {
      c_.wx[1] = band + 54 + 6 * window(j, c.n[g][1], st, sp);
      c_.st[1] = (st - j) * n0;
      c_.sp[1] = sp * n0;
    }
    c_.wx[D - 1] = band + 54 * (D - 1) + 6 * window(k, c.n[g][D - 1], st, sp);
    const int o = D == 3 ? j * n0 + i : i;
#pragma unroll
    for (int m = 0; m < NW; ++m) c_.sl[m] = slab(g, 0, st + m * sp) + o;
    c_.b = arr(g, 2)[q];
    c_.f = factor(g, i, j, k);
    return c_;
  }
  // f - A x (or f - A^T x) of a cell, x at element offset ao from array 0.  One accumulator per
  // dimension: the chains of dependent multiply-adds are NW long, not D NW.
  __device__ __forceinline__ T resid(int g, const Cell& e, int ao) const {
    T s[D];
#pragma unroll
    for (int d = 0; d < D; ++d) s[d] = T(0);
#pragma unroll
    for (int m = 0; m < NW; ++m) {
      s[D - 1] = fma(e.wx[D - 1][m], e.sl[m][ao], s[D - 1]);
#pragma unroll
      for (int d = 0; d + 1 < D; ++d) s[d] = fma(e.wx[d][m], e.own[ao + e.st[d] + m * e.sp[d]], s[d]);
    }
    T t = s[0];
#pragma unroll
    for (int d = 1; d < D; ++d) t += s[d];
    return fma(-c.kc[g], t, fma(-c.alpha, e.own[ao], e.b));
  }
  __device__ __forceinline__ T factor(int g, int i, int j, int k) const {
    int q = face_class(i, c.n[g][0]);
    if (D == 3) q += 5 * face_class(j, c.n[g][1]) + 25 * face_class(k, c.n[g][2]);
    else q += 5 * face_class(k, c.n[g][1]);
    return wt[g * MgCluster<T, D>::NWT + q];
  }
  // nu sweeps from array a, then (RES) the residual of the result into the other array; returns
  // the array with the result.  Grids of at most one cell per thread keep the cell's set-up in
  // registers across the sweeps.
  template <bool RES>
  __device__ int smooth(int g, int a, int nu) const {
    const int n0 = c.n[g][0], P = n0 * (D == 3 ? c.n[g][1] : 1), nc = slabs(g) * P, AO = c.R[g] * P;
    if (c.R[g] * P <= MC_THREADS) {
      const int q = threadIdx.x;
      const bool act = q < nc;
      Cell e;
      if (act) {
        const int s = q / P, r = q - s * P, j = D == 3 ? r / n0 : 0, i = r - j * n0;
        e = cell(g, q, i, j, s + rank * c.R[g]);
      }
      for (int s = 0; s < nu + (RES ? 1 : 0); ++s) {
        if (act) {
          const T r = resid(g, e, a * AO);
          const_cast<T*>(e.own)[(1 - a) * AO] = (RES && s == nu) ? r : fma(e.f, r, e.own[a * AO]);
        }
        mc_sync();
        a = 1 - a;
      }
    } else {
      for (int s = 0; s < nu + (RES ? 1 : 0); ++s) {
        cells(g, [&](int q, int i, int j, int k) {
          const Cell e = cell(g, q, i, j, k);
          const T r = resid(g, e, a * AO);
          const_cast<T*>(e.own)[(1 - a) * AO] = (RES && s == nu) ? r : fma(e.f, r, e.own[a * AO]);
        });
        mc_sync();
        a = 1 - a;
      }
    }
    return RES ? 1 - a : a;
  }
  // coarse taps of fine cell i along one dimension (n coarse cells): cell index and weight
  __device__ __forceinline__ int taps(int i, int n, int face, int ix[4], T w[4]) const {
    const int p = i >> 1, s = (i & 1) ? 1 : -1;
    if (p + s >= 0 && p + s < n) {
      ix[0] = p;
      ix[1] = p + s;
      w[0] = T(0.75);
      w[1] = T(0.25);
      ix[2] = ix[3] = p;
      w[2] = w[3] = T(0);
      return 2;
    }
    const int side = s > 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      ix[m] = side ? n - 1 - m : m;
      w[m] = T(0.25) * gh[4 * (2 * face + side) + m] + (m == 0 ? T(0.75) : T(0));
    }
    return 4;
  }

  __device__ void run(const T* __restrict__ b, T* __restrict__ x, double* bot) const {
    const int M = c.ng - 1;
    // right-hand side of grid 0, and its first sweep from x = 0
    {
      T* bs = arr(0, 2);
      T* xs = arr(0, 0);
      const T* __restrict__ bg = b + c.gp.off;
      cells(0, [&](int q, int i, int j, int k) {
        const long long o = D == 3 ? (long long)(k + NG) * c.gp.sz + (long long)(j + NG) * c.gp.sy + i + NG
                                   : (long long)(k + NG) * c.gp.sy + i + NG;
        const T v = bg[o];
        bs[q] = v;
        xs[q] = factor(0, i, j, k) * v;
      });
    }
    mc_sync();
    int cur[MC_MAX];
    for (int g = 0; g < M; ++g) {
      // sweeps, the residuals into the other array, then their means (and the next grid's first sweep)
      const int a = smooth<true>(g, 0, c.nu1 - 1);
      cur[g] = a;
      T* bs = arr(g + 1, 2);
      T* xs = arr(g + 1, 0);
      const int n0 = c.n[g][0];
      const bool last = g + 1 == M;
      cells(g + 1, [&](int q, int i, int j, int k) {
        T v = T(0);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const T* f = slab(g, 1 - a, 2 * k + s) + 2 * i + (D == 3 ? 2 * j * n0 : 0);
          v += f[0];
          v += f[1];
          if (D == 3) {
            v += f[n0];
            v += f[n0 + 1];
          }
        }
        v *= T(D == 3 ? 0.125 : 0.25);
        bs[q] = v;
        if (!last) xs[q] = factor(g + 1, i, j, k) * v;
      });
      mc_sync();
    }
    // dense bottom solve: every block gathers the right-hand side, one warp per row
    {
      const int n0 = c.n[M][0], P = n0 * (D == 3 ? c.n[M][1] : 1);
      for (int t = threadIdx.x; t < c.nbot; t += MC_THREADS) bot[t] = (double)slab(M, 2, t / P)[t % P];
      __syncthreads();
      unsigned nranks;
      asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nranks));
      const int lane = threadIdx.x & 31;
      for (int t = rank * (MC_THREADS / 32) + (threadIdx.x >> 5); t < c.nbot; t += nranks * (MC_THREADS / 32)) {
        const double* __restrict__ row = c.minv + (long long)t * c.ldb;
        double acc = 0.0;
        for (int q = lane; q < c.nbot; q += 32) acc = fma(row[q], bot[q], acc);
        for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
        if (lane == 0) slab(M, 0, t / P)[t % P] = T(acc);
      }
      cur[M] = 0;
      mc_sync();
    }
    for (int g = M - 1; g >= 0; --g) {
      T* xs = arr(g, cur[g]);
      const int m0 = c.n[g + 1][0], ca = cur[g + 1];
      cells(g, [&](int q, int i, int j, int k) {
        int ix[4], iy[4], iz[4];
        T wx[4], wy[4], wz[4];
        const int cx = taps(i, m0, 0, ix, wx);
        const int cy = D == 3 ? taps(j, c.n[g + 1][1], 1, iy, wy) : 1;
        const int cz = taps(k, c.n[g + 1][D - 1], D - 1, iz, wz);
        T v = T(0);
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          if (z >= cz) break;
          const T* pl = slab(g + 1, ca, iz[z]);
          T vz = T(0);
#pragma unroll
          for (int y = 0; y < (D == 3 ? 4 : 1); ++y) {
            if (y >= cy) break;
            const T* row = D == 3 ? pl + iy[y] * m0 : pl;
            T vy = fma(wx[1], row[ix[1]], wx[0] * row[ix[0]]);
            if (cx == 4) vy = fma(wx[3], row[ix[3]], fma(wx[2], row[ix[2]], vy));
            vz = D == 3 ? fma(wy[y], vy, vz) : vy;
          }
          v = fma(wz[z], vz, v);
        }
        xs[q] += v;
      });
      mc_sync();
      cur[g] = smooth<false>(g, cur[g], c.nu2);
    }
    {
      const T* xs = arr(0, cur[0]);
      T* __restrict__ xg = x + c.gp.off;
      cells(0, [&](int q, int i, int j, int k) {
        const long long o = D == 3 ? (long long)(k + NG) * c.gp.sz + (long long)(j + NG) * c.gp.sy + i + NG
                                   : (long long)(k + NG) * c.gp.sy + i + NG;
        xg[o] = xs[q];
      });
    }
    mc_sync();  // no block leaves while another still reads its slabs
  }
};

template <typename T, int D, bool TR>
__global__ void __launch_bounds__(MC_THREADS) k_mg_cluster(const __grid_constant__ MgCluster<T, D> c,
                                                           const T* __restrict__ b, T* __restrict__ x) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ T sband[3 * 54];
  __shared__ T swt[MC_MAX * MgCluster<T, D>::NWT];
  __shared__ T sgh[24];
  __shared__ double bot[MC_BOT];
  unsigned rank, nranks;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nranks));
  const long long rep = (blockIdx.x / nranks) * c.cstride;
  for (int q = threadIdx.x; q < 3 * 54; q += MC_THREADS) sband[q] = (&c.band[0][0][0])[q];
  for (int q = threadIdx.x; q < c.ng * MgCluster<T, D>::NWT; q += MC_THREADS) swt[q] = (&c.wt[0][0])[q];
  if (threadIdx.x < 24) sgh[threadIdx.x] = (&c.ghost[0][0])[threadIdx.x];
  __syncthreads();
  const MgClusterRun<T, D, TR> v{c, reinterpret_cast<T*>(smraw), sband, swt, sgh, (int)rank};
  mc_sync();  // every block's shared memory exists before it is read
  pdl_wait();
  v.run(b + rep, x + rep, bot);
}

}  // namespace amr4
