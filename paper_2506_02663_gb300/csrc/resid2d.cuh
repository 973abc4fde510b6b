// resid2d.cuh -- FP64 residual of a large 2-D level-0 grid with exact fixed-point sums.
//
// The refinement loop's residual f - (alpha x + beta L x) takes nine FP64 operations a cell in
// floating point and is bound by their rate (377 us on 4096^2, whose bytes take 60 us).  As in
// the 3-D residual (k_resid3d_fx) every value of x is rounded once to a 64-bit fixed-point
// frame set by the grid's largest |x| (k_absmax_patch), T = 16 s1 - s2 - 60 x = 12 h^2 L x is
// exact in int64, and two FP64 multiply-adds remain (one for alpha = 0).  What bounds it now is
// the integer work, most of it the two conversions, and the FP64 rate: 189 us and 25 us for the
// frame (alpha not zero).
//
// One warp owns a strip of 128 columns, four per lane, and marches up the rows: each row is
// converted once, five rows of integers sit in registers, x neighbours come by shuffle, and
// the strips overlap by one lane per side.  The grid is the whole domain, so every ghost is a
// physical one: in x the face lanes evaluate it from their own four cells, in y the ghost rows
// are formed from the four rows next to the face when the march reaches them.
//
// The frame holds 56 bits, three more than a double: values within a factor 8 of the largest
// enter exactly.  Away from the faces |T| < (16 4 + 4 + 60) 2^56 = 2^63.  Next to a face the
// ghosts (at most 11.7 and 84.4 times the largest value) could carry T out of int64, so its
// parts, |s1| < 2^61 and two halves of s2 below 2^63, are combined in FP64 there.  A grid
// without a frame (a non-finite value, or all values tiny) takes plain FP64 in the same launch.
#pragma once

#include "stream2d.cuh"

namespace amr4 {

constexpr int RX_W = 120;     // columns a strip finishes (128 less one lane per side)
constexpr int RX_WARPS = 4;

struct I4 {
  long long v[4];
};

// x in the frame of exponent emax: significand << 3 at e = emax, rounded to nearest below
__device__ __forceinline__ long long fx56_of(double x, int emax) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned bh = (unsigned)(b >> 32), bl = (unsigned)b;
  const int e = (int)((bh >> 20) & 0x7ffu), s = emax - e;
  unsigned long long u;
  if (s < 32 && e != 0) {
    const unsigned mh = __funnelshift_l(bl, (bh & 0xfffffu) | 0x100000u, 3), ml = bl << 3;
    const unsigned lo = ml + ((1u << s) >> 1);
    const unsigned hi = mh + (lo < ml ? 1u : 0u);
    u = ((unsigned long long)(hi >> s) << 32) | __funnelshift_r(lo, hi, s);
  } else {
    const unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 3;
    u = e != 0 && s < 58 ? (m + (1ull << (s - 1))) >> s : 0ull;  // subnormal values lie below any frame's unit
  }
  return (bh >> 31) ? -(long long)u : (long long)u;
}

struct Resid2dFx {
  const LevelView& lv;
  const double* __restrict__ xb;  // patch base
  int n0, n1, sy, c0, emax;
  bool act;

  __device__ __forceinline__ void load(int k, double d[4]) const {
    if (!act) {
      d[0] = d[1] = d[2] = d[3] = 0.0;
      return;
    }
    const double* r = xb + (k + NG) * sy + c0 + NG;
    const double2 a = *reinterpret_cast<const double2*>(r), b = *reinterpret_cast<const double2*>(r + 2);
    d[0] = a.x;
    d[1] = a.y;
    d[2] = b.x;
    d[3] = b.y;
  }
  __device__ __forceinline__ I4 convert(const double d[4]) const {
    I4 r;
#pragma unroll
    for (int q = 0; q < 4; ++q) r.v[q] = fx56_of(d[q], emax);
    return r;
  }
  // physical ghost of layer l from four integers inward of the face
  __device__ __forceinline__ long long ghost(int type, int l, long long a, long long b, long long c, long long d) const {
    double v = 0.0;
    v += gcoef<double>(type, l, 0) * (double)a;
    v += gcoef<double>(type, l, 1) * (double)b;
    v += gcoef<double>(type, l, 2) * (double)c;
    v += gcoef<double>(type, l, 3) * (double)d;
    return __double2ll_rn(v);
  }
  // row k of the march: a stored row (values d, loaded ahead), or a ghost row
  __device__ __forceinline__ I4 row(int k, const double d[4]) const {
    if (k >= 0 && k < n1) return convert(d);
    const int side = k < 0 ? 0 : 1, l = side == 0 ? -k - 1 : k - n1, type = lv.bc[2 + side];
    const int k0 = side == 0 ? 0 : n1 - 1, s = side == 0 ? 1 : -1;
    I4 q[4], r;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      double e[4];
      load(k0 + m * s, e);
      q[m] = convert(e);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) r.v[c] = ghost(type, l, q[0].v[c], q[1].v[c], q[2].v[c], q[3].v[c]);
    return r;
  }
};

// Residual of rows [chunk ch, ...) of one strip; see above.  HASA: alpha is not zero.
template <bool HASA>
__device__ __forceinline__ void resid2d_fx_strip(const LevelView& lv, const PatchDesc& p, unsigned long long frame, int strip,
                                                 int chunk, int ch, const double* __restrict__ x,
                                                 const double* __restrict__ f, double* __restrict__ out, double alpha,
                                                 double beta) {
  const int lane = threadIdx.x & 31;
  const int n0 = p.n[0], n1 = p.n[1], sy = (int)p.sy;
  const int u0 = strip * RX_W, u1 = min(n0, u0 + RX_W);
  const int xs = strip == 0 ? 0 : u0 - 4;
  const int c0 = xs + 4 * lane;
  const int y0 = chunk * ch, y1 = min(n1, y0 + ch);
  if (y0 >= y1) return;
  const bool act = c0 < n0, cols = act && c0 >= u0 && c0 < u1;
  const int emax = (int)((frame >> 52) & 0x7ffull);
  const double* __restrict__ xb = x + p.off;
  const double* __restrict__ fb = f + p.off;
  double* __restrict__ ob = out + p.off;
  if (emax == 0x7ff || (emax != 0 && emax < 56)) {
    // no frame: plain FP64, cell by cell
    const double inv = lv.inv12h2, kc2 = beta * inv, kc1 = 16.0 * kc2, kc0 = alpha - 60.0 * kc2;
    if (!cols) return;
    for (int k = y0; k < y1; ++k)
      for (int q = 0; q < 4; ++q) {
        const int i = c0 + q, o = (k + NG) * sy + i + NG;
        double a1, a2, b1, b2;
        line_sums<double>(xb, o, 1, face_class(i, n0) == 0, i, n0, lv.bc[0], lv.bc[1], a1, a2);
        line_sums<double>(xb, o, sy, face_class(k, n1) == 0, k, n1, lv.bc[2], lv.bc[3], b1, b2);
        ob[o] = fma(kc2, a2 + b2, fma(-kc1, a1 + b1, fma(-kc0, xb[o], fb[o])));
      }
    return;
  }
  const double kT = emax == 0 ? 0.0 : beta * lv.inv12h2 * __longlong_as_double((long long)(emax - 55) << 52);
  const bool xl = c0 == 0, xh = c0 + 4 == n0, xface = xs == 0 || xs + 128 >= n0;
  const Resid2dFx R{lv, xb, n0, n1, sy, c0, emax, act};
  I4 w[5];
  double d[4], dn[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int k = y0 - 2 + m;
    if (k >= 0 && k < n1) R.load(k, d);
    w[m] = R.row(k, d);
  }
  if (y0 + 2 < n1) R.load(y0 + 2, d);
  auto rows4 = [&](const double* g, int k, double v[4]) {
    const double* r = g + (k + NG) * sy + c0 + NG;
    const double2 a = *reinterpret_cast<const double2*>(r), b = *reinterpret_cast<const double2*>(r + 2);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
  };
  double fk[4] = {0, 0, 0, 0};
  if (cols) rows4(fb, y0, fk);
  // one row; FACE: some cell of the strip's row lies next to a face (uniform in the warp), so that
  // the FP64 conversions stay off the other rows' path
  auto step = [&](int k, auto facec) {
    constexpr bool FACE = decltype(facec)::value;
    // the next row of x and of f, one step ahead; x of this row again (read two steps ago, in L1)
    double fn[4] = {0, 0, 0, 0}, xk[4] = {0, 0, 0, 0};
    if (k + 3 < n1) R.load(k + 3, dn);
    if (cols && k + 1 < y1) rows4(fb, k + 1, fn);
    if (HASA && cols) rows4(xb, k, xk);
    w[4] = R.row(k + 2, d);
    const I4& c = w[2];
    long long lz = __shfl_up_sync(0xffffffffu, c.v[2], 1), lw = __shfl_up_sync(0xffffffffu, c.v[3], 1);
    long long rx = __shfl_down_sync(0xffffffffu, c.v[0], 1), ry = __shfl_down_sync(0xffffffffu, c.v[1], 1);
    if (FACE && xface) {
      if (xl) {
        lw = R.ghost(lv.bc[0], 0, c.v[0], c.v[1], c.v[2], c.v[3]);
        lz = R.ghost(lv.bc[0], 1, c.v[0], c.v[1], c.v[2], c.v[3]);
      }
      if (xh) {
        rx = R.ghost(lv.bc[1], 0, c.v[3], c.v[2], c.v[1], c.v[0]);
        ry = R.ghost(lv.bc[1], 1, c.v[3], c.v[2], c.v[1], c.v[0]);
      }
    }
    double r[4];
    auto sums = [&](int q, long long& s1, long long& sx, long long& sy2) {
      const long long m1 = q > 0 ? c.v[q > 0 ? q - 1 : 0] : lw, m2 = q > 1 ? c.v[q > 1 ? q - 2 : 0] : (q == 1 ? lw : lz);
      const long long p1 = q < 3 ? c.v[q < 3 ? q + 1 : 3] : rx, p2 = q < 2 ? c.v[q < 2 ? q + 2 : 3] : (q == 2 ? rx : ry);
      s1 = (m1 + p1) + (w[1].v[q] + w[3].v[q]);
      sx = m2 + p2;
      sy2 = w[0].v[q] + w[4].v[q];
    };
    if constexpr (FACE) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        long long s1, sx, sy2;
        sums(q, s1, sx, sy2);
        r[q] = fma(16.0, (double)s1, -fma(60.0, (double)c.v[q], (double)sx + (double)sy2));
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        long long s1, sx, sy2;
        sums(q, s1, sx, sy2);
        r[q] = fx_to_double(s1 * 16 - (sx + sy2) - c.v[q] * 60);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) r[q] = fma(-kT, r[q], HASA ? fma(-alpha, xk[q], fk[q]) : fk[q]);
    if (cols) {
      double* o = ob + (k + NG) * sy + c0 + NG;
      *reinterpret_cast<double2*>(o) = make_double2(r[0], r[1]);
      *reinterpret_cast<double2*>(o + 2) = make_double2(r[2], r[3]);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) w[m] = w[m + 1];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      d[q] = dn[q];
      fk[q] = fn[q];
    }
  };
#pragma unroll 1
  for (int k = y0; k < y1; ++k) {
    if (xface || k < 2 || k >= n1 - 2) step(k, std::true_type{});
    else step(k, std::false_type{});
  }
}

template <bool HASA>
__global__ void __launch_bounds__(32 * RX_WARPS, 4) k_resid2d_fx(LevelView lv, int ns, int nch, int ch,
                                                                 const double* __restrict__ x, const double* __restrict__ f,
                                                                 double* __restrict__ out, double alpha, double beta) {
  const int w = blockIdx.x * RX_WARPS + (threadIdx.x >> 5);
  pdl_wait();  // the frame is written by the preceding kernel
  if (w >= ns * nch) return;
  resid2d_fx_strip<HASA>(lv, lv.p0, lv.fxs[0], w % ns, w / ns, ch, x, f, out, alpha, beta);
}

}  // namespace amr4
