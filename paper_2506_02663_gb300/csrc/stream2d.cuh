// stream2d.cuh -- four weighted-Jacobi sweeps of a 2-D FP32 level in one pass, the iterates
// streaming through registers.
//
// A multigrid leg is four sweeps and a residual restriction (down), a prolongation and four
// sweeps (up), or four sweeps from zero added to a correction (post-smoothing of an AMR level).
// The tiled form keeps a tile and its halo in shared memory and recomputes a 52^2 (48^2) region
// for 32^2 cells at about 23 instructions a cell and sweep: issue-bound, 385 (426) us per
// 4096^2 leg whose bytes take 22 (33) us.  Here one warp owns a strip of 128 columns, four per
// lane, and marches up the rows: at step t it reads row t, sweep s produces row t - 2 s (+ 2 in
// the down form, whose first sweep is a product), each from a five-row register window of the
// previous iterate; x neighbours come by shuffle from the two adjacent lanes.  A sweep costs ten
// arithmetic instructions a cell plus one shuffle, and the halo is 2 x 12 of 128 columns
// (1.2) and 18 rows per chunk: the 4096^2 Helmholtz solve went from 29.8 to 17.5 ms.  Rows are
// requested four steps ahead by cp.async into slots private to their lane (no barrier): a step
// waited for the row asked for one step earlier.
//
// Physical faces: the first and last lane of a face strip evaluate the two ghost cells of
// Eqs. (velBCHomoDiri5th)/(Neumann5) from their own four cells; at the low y face row 0 is
// produced together with row 1 (its ghosts need row 3), at the high y face the two ghost rows
// are pushed after the last row.  Coarse-fine edges use zero coefficients (zero ghosts).
#pragma once

#include "kernels.cuh"

namespace amr4 {

enum { LEG_DOWN = 0, LEG_UP = 1, LEG_POST = 2 };
constexpr int LEG_NU = 4;        // sweeps per pass
constexpr int LEG_W = 128;       // columns of a strip (four per lane)
constexpr int LEG_WARPS = 4;     // warps per block
constexpr int LEG_RING = 16;     // rows of f kept per warp (ten in use, LEG_AHEAD on their way)
constexpr int LEG_AHEAD = 4;     // rows requested ahead of their step
constexpr int LEG_CRING = 8;     // up: coarse rows kept per warp

struct Leg2D {
  PatchDesc gp, gcp;             // the level's patch and the coarser one's
  int nd0, nd1;                  // domain extents at the level
  int ns, ch, nch;               // strips, rows per chunk, chunks
  int p, pad;                    // batches: problem index
  float kc0, kc1, kc2;           // A x = kc0 x + kc1 s1 - kc2 s2
  float wt[25];                  // omega / diag by distance class
  float g[4][2][4];              // ghost coefficients [face][layer][cell]; zero at coarse-fine edges
  float cg[4][4];                // layer-1 ghost coefficients of the coarser domain (up)
  const float *b, *xi, *xc;      // right-hand side; up: iterate in, coarse correction
  float *xo, *x2, *bcn;          // iterate out (post: += ), optional second target +=, coarse right-hand side
};

// columns of halo per open strip side and rows per open chunk side
template <int MODE>
constexpr int leg_hx() { return MODE == LEG_DOWN ? 12 : 8; }
template <int MODE>
constexpr int leg_hy() { return MODE == LEG_DOWN ? 10 : 8; }
template <int MODE>
constexpr int leg_lag() { return MODE == LEG_POST ? 6 : 8; }  // steps between reading a row and finishing it

// first useful column of strip k (k = ns: n0)
__host__ __device__ inline int leg_u(int k, int ns, int n0, int hx) {
  if (k <= 0) return 0;
  if (k >= ns) return n0;
  return (LEG_W - hx) + (k - 1) * (LEG_W - 2 * hx);
}
__host__ __device__ inline int leg_strips(int n0, int hx) {
  int ns = 1;
  while (!(ns == 1 ? n0 <= LEG_W : leg_u(ns - 1, ns, n0, hx) - hx + LEG_W >= n0)) ++ns;
  return ns;
}

namespace leg2 {
__device__ __forceinline__ float4 lin4(const float* c, float4 a, float4 b, float4 d, float4 e) {
  return make_float4(fmaf(c[3], e.x, fmaf(c[2], d.x, fmaf(c[1], b.x, c[0] * a.x))),
                     fmaf(c[3], e.y, fmaf(c[2], d.y, fmaf(c[1], b.y, c[0] * a.y))),
                     fmaf(c[3], e.z, fmaf(c[2], d.z, fmaf(c[1], b.z, c[0] * a.z))),
                     fmaf(c[3], e.w, fmaf(c[2], d.w, fmaf(c[1], b.w, c[0] * a.w))));
}
__device__ __forceinline__ float lin1(const float* c, float a, float b, float d, float e) {
  return fmaf(c[3], e, fmaf(c[2], d, fmaf(c[1], b, c[0] * a)));
}
__device__ __forceinline__ float4 ldrow(const float* __restrict__ g) {  // four cells, 8-byte aligned
  const float2 a = *reinterpret_cast<const float2*>(g), b = *reinterpret_cast<const float2*>(g + 2);
  return make_float4(a.x, a.y, b.x, b.y);
}
// asynchronous copy of four cells (8-byte aligned) into the lane's own slot; zeros where !on
__device__ __forceinline__ void cprow(float4* s, const float* g, bool on) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(s);
  const int n = on ? 8 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(g), "r"(n) : "memory");
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d + 8), "l"(g + (on ? 2 : 0)), "r"(n) : "memory");
}
template <typename V>
__device__ __forceinline__ void cpone(V* s, const float* g, bool on) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(s);
  const int n = on ? (int)sizeof(V) : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(g), "n"(sizeof(V)), "r"(n) : "memory");
}
__device__ __forceinline__ void strow(float* g, float4 v) {
  *reinterpret_cast<float2*>(g) = make_float2(v.x, v.y);
  *reinterpret_cast<float2*>(g + 2) = make_float2(v.z, v.w);
}
}  // namespace leg2

template <int MODE>
struct LegRun {
  static constexpr int HX = leg_hx<MODE>(), HY = leg_hy<MODE>(), LAG = leg_lag<MODE>();
  static constexpr int NWIN = MODE == LEG_POST ? 3 : 4;
  // shared memory of a warp, every entry private to one lane (no barriers)
  struct Smem {
    float4 f[LEG_RING][32];                                  // right-hand side rows
    float4 x[MODE == LEG_UP || MODE == LEG_POST ? 5 : 1][32];  // up: iterate rows; post: rows of xo
    float4 y[MODE == LEG_UP ? 1 : 5][32];                    // rows of the second target
    float2 c[MODE == LEG_UP ? LEG_CRING : 1][32];            // up: coarse rows
    float e[MODE == LEG_UP ? LEG_CRING : 1][2];              // up: the coarse cells beyond the strip
  };
  const Leg2D& L;
  Smem& S;
  int lane, c0, n0, n1;
  bool act, xl, xh, xface;  // lane holds cells; lane at the low / high x edge; strip touches one
  float kc0, kc1, kc2;
  float4 wI;                // factors away from the y faces
  int sy, fo;               // row pitch; offset of (c0, row 0) inside the patch
  float4 W[4][5];
  float4 hg, rp;            // ghost row held for the next step; residual of the even row
  int y0, y1, tend;         // rows this warp stores; steps end
  bool cols;                // the lane's columns are stored

  // residual of the row c between rows m1, m2 (below) and p1, p2 (above)
  __device__ __forceinline__ float4 resid(float4 m2, float4 m1, float4 c, float4 p1, float4 p2, float4 f) const {
    float lz = __shfl_up_sync(0xffffffffu, c.z, 1), lw = __shfl_up_sync(0xffffffffu, c.w, 1);
    float rx = __shfl_down_sync(0xffffffffu, c.x, 1), ry = __shfl_down_sync(0xffffffffu, c.y, 1);
    if (xface) {
      if (xl) {
        lw = leg2::lin1(L.g[0][0], c.x, c.y, c.z, c.w);
        lz = leg2::lin1(L.g[0][1], c.x, c.y, c.z, c.w);
      }
      if (xh) {
        rx = leg2::lin1(L.g[1][0], c.w, c.z, c.y, c.x);
        ry = leg2::lin1(L.g[1][1], c.w, c.z, c.y, c.x);
      }
    }
    float4 r;
    r.x = fmaf(kc2, (lz + c.z) + (m2.x + p2.x), fmaf(-kc1, (lw + c.y) + (m1.x + p1.x), fmaf(-kc0, c.x, f.x)));
    r.y = fmaf(kc2, (lw + c.w) + (m2.y + p2.y), fmaf(-kc1, (c.x + c.z) + (m1.y + p1.y), fmaf(-kc0, c.y, f.y)));
    r.z = fmaf(kc2, (c.x + rx) + (m2.z + p2.z), fmaf(-kc1, (c.y + c.w) + (m1.z + p1.z), fmaf(-kc0, c.z, f.z)));
    r.w = fmaf(kc2, (c.y + ry) + (m2.w + p2.w), fmaf(-kc1, (c.z + rx) + (m1.w + p1.w), fmaf(-kc0, c.w, f.w)));
    return r;
  }
  __device__ __forceinline__ float4 fma4(float4 w, float4 r, float4 c) const {
    return make_float4(fmaf(w.x, r.x, c.x), fmaf(w.y, r.y, c.y), fmaf(w.z, r.z, c.z), fmaf(w.w, r.w, c.w));
  }
  __device__ __forceinline__ float4 fring(int k) const { return S.f[k & (LEG_RING - 1)][lane]; }
  // factors of row k
  __device__ __forceinline__ float4 factors(int k) const {
    const int cy = face_class(L.gp.lo[1] + k, L.nd1);
    if (cy == 0) return wI;
    const int g = L.gp.lo[0] + c0;
    return make_float4(L.wt[face_class(g, L.nd0) + 5 * cy], L.wt[face_class(g + 1, L.nd0) + 5 * cy],
                       L.wt[face_class(g + 2, L.nd0) + 5 * cy], L.wt[face_class(g + 3, L.nd0) + 5 * cy]);
  }
  // a finished iterate row; sl: the slot its targets' old values wait in (-1: read them here)
  __device__ __forceinline__ void store(int k, float4 v, int sl) const {
    if (!cols || k < y0 || k >= y1) return;
    const int o = fo + k * sy;
    if (MODE == LEG_POST) {
      const float4 e = sl < 0 ? leg2::ldrow(L.xo + o) : S.x[MODE == LEG_POST && sl > 0 ? sl : 0][lane];
      leg2::strow(L.xo + o, make_float4(e.x + v.x, e.y + v.y, e.z + v.z, e.w + v.w));
    } else {
      leg2::strow(L.xo + o, v);
    }
    if (MODE != LEG_UP && L.x2 != nullptr) {
      const float4 e = sl < 0 ? leg2::ldrow(L.x2 + o) : S.y[MODE != LEG_UP && sl > 0 ? sl : 0][lane];
      leg2::strow(L.x2 + o, make_float4(e.x + v.x, e.y + v.y, e.z + v.z, e.w + v.w));
    }
  }
  // A residual row (down): rows pair up into coarse rows.  The lane's two coarse cells are stored in one
  // access where they start on an even column of the coarse patch: always on level 0, and on a refined
  // level where the box starts on an even coarse cell (boxes start on even fine cells).
  __device__ __forceinline__ void restrict_row(int k, float4 r) {
    if ((k & 1) == 0) {
      rp = r;
      return;
    }
    if (!cols || k < y0 || k >= y1) return;
    const float2 v = make_float2((((rp.x + rp.y) + r.x) + r.y) * 0.25f, (((rp.z + rp.w) + r.z) + r.w) * 0.25f);
    const PatchDesc& q = L.gcp;
    const int gy = (L.gp.lo[1] + k) >> 1, gx = (L.gp.lo[0] + c0) >> 1;
    float* o = L.bcn + (gy - q.lo[1] + NG) * (int)q.sy + gx - q.lo[0] + NG;
    if (((gx - q.lo[0]) & 1) == 0) {
      *reinterpret_cast<float2*>(o) = v;
    } else {
      o[0] = v.x;
      o[1] = v.y;
    }
  }
  // row t of the first window: down / post w f, up xi + prolongation
  __device__ __forceinline__ float4 first(int t, float4 f, float4 xrow, float2 ca, float2 cb, float ea, float eb,
                                          bool face) const {
    if (MODE != LEG_UP) {
      const float4 w = face ? factors(t) : wI;
      return make_float4(w.x * f.x, w.y * f.y, w.z * f.z, w.w * f.w);
    }
    // the tiled leg's weights and order: own, x neighbour, y neighbour, diagonal
    const int p = t >> 1, s = (t & 1) ? 1 : -1, m1 = L.gcp.n[1];
    const bool out = face && (p + s < 0 || p + s >= m1);
    const int side = s > 0, d = side ? -1 : 1, k0 = side ? m1 - 1 : 0;
    if (out) {
      // the coarse row outside the domain: the extension of the four rows next to the face
      const float* cc = L.cg[2 + side];
      cb = make_float2(0.f, 0.f);
      eb = 0.f;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float2 v = crow(k0 + m * d);
        cb.x = fmaf(cc[m], v.x, cb.x);
        cb.y = fmaf(cc[m], v.y, cb.y);
        eb = fmaf(cc[m], cedge(k0 + m * d), eb);
      }
    }
    float la = __shfl_up_sync(0xffffffffu, ca.y, 1), ra = __shfl_down_sync(0xffffffffu, ca.x, 1);
    float lb = __shfl_up_sync(0xffffffffu, cb.y, 1), rb = __shfl_down_sync(0xffffffffu, cb.x, 1);
    if (lane == 0) {
      la = ea;
      lb = eb;
    }
    if (lane == 31) {
      ra = ea;
      rb = eb;
    }
    if (xface) {
      const float nx = __shfl_down_sync(0xffffffffu, ca.x, 1), ny = __shfl_down_sync(0xffffffffu, ca.y, 1);
      const float px = __shfl_up_sync(0xffffffffu, ca.x, 1), py = __shfl_up_sync(0xffffffffu, ca.y, 1);
      const float mx = __shfl_down_sync(0xffffffffu, cb.x, 1), my = __shfl_down_sync(0xffffffffu, cb.y, 1);
      const float qx = __shfl_up_sync(0xffffffffu, cb.x, 1), qy = __shfl_up_sync(0xffffffffu, cb.y, 1);
      if (xl) {
        la = leg2::lin1(L.cg[0], ca.x, ca.y, nx, ny);
        lb = out ? corner(0, k0, d, L.cg[2 + side]) : leg2::lin1(L.cg[0], cb.x, cb.y, mx, my);
      }
      if (xh) {
        ra = leg2::lin1(L.cg[1], ca.y, ca.x, py, px);
        rb = out ? corner(1, k0, d, L.cg[2 + side]) : leg2::lin1(L.cg[1], cb.y, cb.x, qy, qx);
      }
    }
    auto mix = [](float c00, float c10, float c01, float c11) {
      return fmaf(0.0625f, c11, fmaf(0.1875f, c01, fmaf(0.1875f, c10, 0.5625f * c00)));
    };
    return make_float4(xrow.x + mix(ca.x, la, cb.x, lb), xrow.y + mix(ca.x, ca.y, cb.x, cb.y),
                       xrow.z + mix(ca.y, ca.x, cb.y, cb.x), xrow.w + mix(ca.y, ra, cb.y, rb));
  }
  // layer-1 extension beyond a corner of the coarser domain (coarse_ext2d's order)
  __device__ __forceinline__ float corner(int xside, int k0, int d, const float* cy) const {
    const float* cx = L.cg[xside];
    const int i0 = xside ? L.gcp.n[0] - 1 : 0, e = xside ? -1 : 1;
    float v = 0.f;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b)
        v = fmaf(cx[a] * cy[b], L.xc[(k0 + b * d + NG) * (int)L.gcp.sy + i0 + a * e + NG], v);
    return v;
  }
  __device__ __forceinline__ float2 crow(int k) const {
    if (!act) return make_float2(0.f, 0.f);
    return *reinterpret_cast<const float2*>(L.xc + (k + NG) * (int)L.gcp.sy + (c0 >> 1) + NG);
  }
  // the coarse cell beyond the strip (first and last lane of an open side)
  __device__ __forceinline__ float cedge(int k) const {
    if (!act || (lane != 0 && lane != 31)) return 0.f;
    const int c = lane == 0 ? max((c0 >> 1) - 1, 0) : min((c0 >> 1) + 2, L.gcp.n[0] - 1);
    return L.xc[(k + NG) * (int)L.gcp.sy + c + NG];
  }

  // Requests what step t needs, into slot PH of the five-row rings: row t of f (up: of xi, and
  // the coarse row that step t is the first to use), the old values of the row it finishes.
  template <int PH>
  __device__ __forceinline__ void request(int t) {
    if (t < n1 && t < tend) {
      const bool on = act;
      leg2::cprow(&S.f[t & (LEG_RING - 1)][lane], on ? L.b + fo + t * sy : L.b, on);
      if (MODE == LEG_UP) {
        leg2::cprow(&S.x[MODE == LEG_UP ? PH : 0][lane], on ? L.xi + fo + t * sy : L.xi, on);
        if (t & 1) request_coarse((t >> 1) + 1);
      }
    }
    const int k = t - 6;
    if (MODE != LEG_UP && cols && k >= y0 && k < y1) {
      if (MODE == LEG_POST) leg2::cprow(&S.x[MODE == LEG_POST ? PH : 0][lane], L.xo + fo + k * sy, true);
      if (L.x2 != nullptr) leg2::cprow(&S.y[MODE == LEG_UP ? 0 : PH][lane], L.x2 + fo + k * sy, true);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ __forceinline__ void request_coarse(int q) {
    if (q < 0 || q >= L.gcp.n[1]) return;
    const int sl = MODE == LEG_UP ? q & (LEG_CRING - 1) : 0;
    const float* r = L.xc + (q + NG) * (int)L.gcp.sy + NG;
    leg2::cpone(&S.c[sl][lane], act ? r + (c0 >> 1) : r, act);
    if (lane == 0) leg2::cpone(&S.e[sl][0], r + max((c0 >> 1) - 1, 0), true);
    if (lane == 31) leg2::cpone(&S.e[sl][1], act ? r + min((c0 >> 1) + 2, L.gcp.n[0] - 1) : r, act);
  }

  // One step: push row t, then every stage.  PH: physical slot of the windows' newest row.
  // FACE: some row of this step lies at a y edge of the patch.
  template <int PH, bool FACE>
  __device__ __forceinline__ void step(int t) {
    request<(PH + LEG_AHEAD) % 5>(t + LEG_AHEAD);
    asm volatile("cp.async.wait_group %0;" ::"n"(LEG_AHEAD) : "memory");
    if (!FACE || t < n1) {
      const float4 f = fring(t);
      if (MODE == LEG_UP) {
        const int p = t >> 1, q = min(max(p + ((t & 1) ? 1 : -1), 0), L.gcp.n[1] - 1), m = LEG_CRING - 1;
        const bool end = lane == 0 || lane == 31;
        const int e = lane >> 4;
        const int sp = MODE == LEG_UP ? p & m : 0, sq = MODE == LEG_UP ? q & m : 0;
        W[0][PH] = first(t, f, S.x[MODE == LEG_UP ? PH : 0][lane], S.c[sp][lane], S.c[sq][lane], end ? S.e[sp][e] : 0.f,
                         end ? S.e[sq][e] : 0.f, FACE);
      } else {
        const float2 z = make_float2(0.f, 0.f);
        W[0][PH] = first(t, f, f, z, z, 0.f, 0.f, FACE);
      }
    } else {
      push_ghost<PH>(W[0], t);
    }
#pragma unroll
    for (int s = 0; s < NWIN; ++s) {
      const int k = t - 2 * (s + 1);  // centre row of this stage
      const bool last = s == NWIN - 1;
      if (FACE && (k <= 0 || k >= n1)) {  // row 0 comes with row 1, when its ghosts are known
        if (!last && k >= n1) push_ghost<PH>(W[s + 1 < 4 ? s + 1 : 3], k);
        continue;
      }
      stage<PH, FACE>(s, last, k, W[s]);
    }
  }
  template <int PH>
  __device__ __forceinline__ void push_ghost(float4 (&V)[5], int k) {
    constexpr int N = PH, A = (PH + 4) % 5, B = (PH + 3) % 5, C = (PH + 2) % 5, D = (PH + 1) % 5;
    if (k == n1) {  // rows n1 - 1 .. n1 - 4 are A .. D
      const float4 g = leg2::lin4(L.g[3][0], V[A], V[B], V[C], V[D]);
      hg = leg2::lin4(L.g[3][1], V[A], V[B], V[C], V[D]);
      V[N] = g;
    } else {
      V[N] = hg;
    }
  }
  template <int PH, bool FACE>
  __device__ __forceinline__ void stage(int s, bool last, int k, float4 (&V)[5]) {
    constexpr int N = PH, A = (PH + 4) % 5, B = (PH + 3) % 5, C = (PH + 2) % 5, D = (PH + 1) % 5;
    // rows k - 2 .. k + 2 are D, C, B, A, N
    if (FACE && k == 1) {  // k = 1 only occurs with the patch's low edge in the region
      // rows 0 .. 3 are C, B, A, N: the two ghost rows, then row 0
      const float4 g1 = leg2::lin4(L.g[2][0], V[C], V[B], V[A], V[N]);
      const float4 g2 = leg2::lin4(L.g[2][1], V[C], V[B], V[A], V[N]);
      V[D] = g1;
      const float4 r = resid(g2, g1, V[C], V[B], V[A], fring(0));
      emit<PH, true>(s, last, 0, r, V[C], A, -1);  // its slot is taken again by now
    }
    const float4 r = resid(V[D], V[C], V[B], V[A], V[N], fring(k));
    emit<PH, FACE>(s, last, k, r, V[B], N, PH);
  }
  // the residual r of centre row k of stage s (iterate c): restricted, or swept into the next window's slot
  template <int PH, bool FACE>
  __device__ __forceinline__ void emit(int s, bool last, int k, float4 r, float4 c, int slot, int sl) {
    if (MODE == LEG_DOWN && last) {
      restrict_row(k, r);
      return;
    }
    const float4 v = fma4(FACE ? factors(k) : wI, r, c);
    if (last) {
      store(k, v, sl);
      return;
    }
    // slot is a constant after inlining
    if (s + 1 < 4) W[s + 1 < 4 ? s + 1 : 3][slot] = v;
    if (MODE == LEG_DOWN && s == 2) store(k, v, sl);  // x after four sweeps
  }

  __device__ __forceinline__ void run(int strip, int chunk) {
    n0 = L.gp.n[0];
    n1 = L.gp.n[1];
    const int u0 = leg_u(strip, L.ns, n0, HX), u1 = leg_u(strip + 1, L.ns, n0, HX);
    const int xs = strip == 0 ? 0 : min(u0 - HX, n0 - LEG_W);
    y0 = chunk * L.ch;
    y1 = min(n1, y0 + L.ch);
    tend = y1 + LAG;
    c0 = xs + 4 * lane;
    act = c0 < n0;
    cols = act && c0 >= u0 && c0 < u1;
    xl = c0 == 0;
    xh = c0 + 4 == n0;
    xface = xs == 0 || xs + LEG_W >= n0;
    sy = (int)L.gp.sy;
    fo = NG * sy + c0 + NG;
    kc0 = L.kc0;
    kc1 = L.kc1;
    kc2 = L.kc2;
    {
      const int g = L.gp.lo[0] + c0;
      wI = make_float4(L.wt[face_class(g, L.nd0)], L.wt[face_class(g + 1, L.nd0)], L.wt[face_class(g + 2, L.nd0)],
                       L.wt[face_class(g + 3, L.nd0)]);
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int q = 0; q < 5; ++q) W[s][q] = make_float4(0.f, 0.f, 0.f, 0.f);
    hg = rp = make_float4(0.f, 0.f, 0.f, 0.f);
    const int r0 = max(0, y0 - HY);  // steps r0 .. tend - 1
    if (MODE == LEG_UP) {
      const int p = r0 >> 1;
      request_coarse(p - 1);
      request_coarse(p);
    }
    static_assert(LEG_AHEAD == 4, "four rows are requested before the first step");
    request<0>(r0);
    request<1>(r0 + 1);
    request<2>(r0 + 2);
    request<3>(r0 + 3);
    // groups of five steps (the windows' slots are then constants); the last group may run past
    // tend: its extra rows are not stored
    for (int t = r0; t < tend; t += 5) {
      // rows t + 4 - LAG .. t + 4: none within two rows of a y edge that this region contains
      const bool face = (r0 == 0 && t - LAG <= 1) || t + 5 > n1 - 3;
      if (!face) {
        group<false>(t);
      } else {
        group<true>(t);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  template <bool FACE>
  __device__ __forceinline__ void group(int t) {
    step<0, FACE>(t);
    step<1, FACE>(t + 1);
    step<2, FACE>(t + 2);
    step<3, FACE>(t + 3);
    step<4, FACE>(t + 4);
  }
};

template <int MODE>
constexpr size_t leg_smem_bytes() { return LEG_WARPS * sizeof(typename LegRun<MODE>::Smem); }

template <int MODE>
__global__ void __launch_bounds__(32 * LEG_WARPS, 3) k_leg2d(const __grid_constant__ Leg2D d) {
  extern __shared__ float4 leg_smem[];
  auto* ring = reinterpret_cast<typename LegRun<MODE>::Smem*>(leg_smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = blockIdx.x * LEG_WARPS + warp;
  pdl_wait();
  if (w >= d.ns * d.nch) return;
  LegRun<MODE> r{d, ring[warp], lane};
  r.run(w % d.ns, w / d.ns);
}

// batches: entry blockIdx.y of a descriptor list, skipped once its problem has converged
template <int MODE>
__global__ void __launch_bounds__(32 * LEG_WARPS, 3) k_leg2d_b(const Leg2D* __restrict__ list, const int* __restrict__ active) {
  extern __shared__ float4 leg_smem[];
  auto* ring = reinterpret_cast<typename LegRun<MODE>::Smem*>(leg_smem);
  __shared__ Leg2D d;
  pdl_wait();
  const Leg2D* e = list + blockIdx.y;
  if (!active[e->p] || blockIdx.x * LEG_WARPS >= e->ns * e->nch) return;
  for (int q = threadIdx.x; q < (int)(sizeof(Leg2D) / 4); q += 32 * LEG_WARPS)
    reinterpret_cast<int*>(&d)[q] = reinterpret_cast<const int*>(e)[q];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = blockIdx.x * LEG_WARPS + warp;
  if (w >= d.ns * d.nch) return;
  LegRun<MODE> r{d, ring[warp], lane};
  r.run(w % d.ns, w / d.ns);
}

}  // namespace amr4
