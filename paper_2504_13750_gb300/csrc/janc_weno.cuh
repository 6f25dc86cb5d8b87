// WENO5-JS reconstruction along a line of split fluxes, shared by the
// single-grid, the block (AMR) and the adjoint face kernels.
//
// The reconstruction costs the FP64 pipe little: with D_j = F_j - F_{j-1} the
// differences of the five values of a window, the face value is
//   F_2 + c1 D1 + c2 D2 + c3 D3 + c4 D4,
//   c1 = -w0/3, c2 = (w1 + 5 w0)/6, c3 = (w1 + 2 w2)/3, c4 = -w2/6
// with the nonlinear weights w_k of the three substencils. Only D_j, the
// products with c_m and their sum are FP64 operations (14 per face for both
// split signs). The weights are formed on 64-bit integers (janc_soft.cuh),
// accurate to about 2^-55, which the FP64 pipe's own evaluation (about 2^-51)
// does not reach.
//
// The smoothness indicators are quadratic forms of adjacent differences,
//   3 beta_0 = 4 D1^2 - 11 D1 D2 + 10 D2^2,
//   3 beta_1 = 4 D2^2 -  5 D2 D3 +  4 D3^2,
//   3 beta_2 = 10 D3^2 - 11 D3 D4 + 4 D4^2,
// so each adjacent pair of differences gives the three forms it will be used
// in (as substencil 0, 1 and 2 of three consecutive windows) from one new
// square and one product. Terms are aligned to the larger difference of the
// pair (or to epsilon where that is larger), where a form is at least 0.7
// times its square, so no form loses relative accuracy to cancellation.
#pragma once

#include "janc_soft.cuh"

#ifdef __CUDACC__
#include "janc_device.cuh"
#endif

namespace janc {
namespace weno {

using namespace soft;

// Sums and products that the compiler must not contract: a line's values are
// the same bits in every kernel that slides along it.
JANC_HD double mul_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dmul_rn(a, b);
#else
  return a * b;
#endif
}
JANC_HD double sub_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dadd_rn(a, -b);
#else
  return a - b;
#endif
}

// 3 epsilon in the unit of a pair's forms at exponent e_min, the smallest a
// pair is aligned to.
struct Eps {
  u64 n;
  int e_min;
  JANC_HD explicit Eps(double eps4) {
    // |D| = M 2^(e - 1086) with M in [2^63, 2^64), so (M^2 / 2^64) 2^-5 counts
    // units of 2^(2e - 2103): 3 eps = m 2^(x - 1075) gives n in [2^59, 2^61).
    const u64 b = bits_of(0.75 * eps4);
    const int x = (int)(b >> 52);
    e_min = (x + 1021) >> 1;
    n = ((b & 0xfffffffffffffull) | (1ull << 52)) << (x + 1028 - 2 * e_min);
  }
};

// One difference: its mantissa in [2^63, 2^64), exponent field and square.
struct Diff {
  u64 m, sq;
  int e;
  JANC_HD void set(double D) {
    const u64 b = bits_of(D);
    e = (int)(hi32(b) >> 20) & 0x7ff;
    m = (b << 11) | (1ull << 63);
    sq = sqhi(m);
  }
};

// 3 (beta + epsilon) of the pair (a, b) as substencil 0, 1 and 2, in units of
// 2^-2103.
struct Forms {
  Num c0, c1, c2;
};
JANC_HD Forms pair_forms(double Da, double Db, const Diff& a, const Diff& b, const Eps& eps) {
  int e = a.e > b.e ? a.e : b.e;
  e = e > eps.e_min ? e : eps.e_min;
  const int da = e - a.e, db = e - b.e;
  const u64 A = shr(a.sq, 2 * da + 5), B = shr(b.sq, 2 * db + 5);
  const u64 C = shr(mulhi(a.m, b.m), da + db + 5);
  const bool opposite = (int)(hi32(bits_of(Da)) ^ hi32(bits_of(Db))) < 0;
  const u64 X = opposite ? C : 0ull - C;  // -D_a D_b
  const u64 t = ((A + B) << 2) + shr(eps.n, 2 * (e - eps.e_min));
  const u64 u = t + 11 * X;
  return Forms{normal(u + 6 * B, 2 * e), normal(t + 5 * X, 2 * e), normal(u + 6 * A, 2 * e)};
}

// Weights of substencils with indicators s0, s1, s2 and linear weights
// 1 : 6 : 3, a sixth of each: w0 = u0 2^(x - 5 - 2 d0), w1 = 3 u1 2^(x - 4 - 2 d1),
// w2 = 3 u2 2^(x - 5 - 2 d2), all times 2^-64, with u_k in [2^59, 2^64): each
// weight keeps its relative accuracy however small it is. The weights are
// 1/s_k^2 up to a common factor; with s0^2 s1^2 s2^2 as that factor they are
// the squares of the products p12 = s1 s2 and so on (upper halves).
struct Weights {
  u64 u0, u1, u2, p12, p02, p01;
  int x, d0, d1, d2;
  JANC_HD Weights(const Num& s0, const Num& s1, const Num& s2) {
    p12 = mulhi(s1.n, s2.n);
    p02 = mulhi(s0.n, s2.n);
    p01 = mulhi(s0.n, s1.n);
    int e = s0.e < s1.e ? s0.e : s1.e;
    e = e < s2.e ? e : s2.e;
    d0 = s0.e - e;
    d1 = s1.e - e;
    d2 = s2.e - e;
    u0 = sqhi(p12);
    u1 = sqhi(p02);
    u2 = sqhi(p01);
    const u64 s = shr(u0, 2 * d0 + 4) + 3 * (shr(u1, 2 * d1 + 3) + shr(u2, 2 * d2 + 4));
    const u64 y = recip(s + (s >> 1), &x);  // 2^127 / (1.5 s 2^x)
    u0 = mulhi(u0, y);
    u1 = mulhi(u1, y);
    u2 = mulhi(u2, y);
  }
};

// The sizes |c1|, c2, c3, |c4| of the coefficients in the stencil's own
// direction. c2 and c3 are sums of two weights aligned to the larger one.
struct Coef {
  double k1, k2, k3, k4;
  JANC_HD explicit Coef(const Weights& w) {
    const u64 v1 = w.u1 >> 3, v2 = w.u2 >> 3;
    const int m = w.d0 < w.d1 ? w.d0 : w.d1, n = w.d1 < w.d2 ? w.d1 : w.d2;
    k1 = to_double(w.u0, w.x - 4 - 2 * w.d0);
    k2 = to_double(3 * shr(v1, 2 * (w.d1 - m)) + 5 * shr(w.u0, 2 * (w.d0 - m) + 4), w.x - 1 - 2 * m);
    k3 = to_double(3 * (shr(v1, 2 * (w.d1 - n)) + shr(v2, 2 * (w.d2 - n))), w.x - 2 * n);
    k4 = to_double(3 * (w.u2 >> 2), w.x - 3 - 2 * w.d2);
  }
};

// Sliding window of one split sign along a line: values F_2..F_4, differences
// D1..D4 and the forms of the pairs (1 2), (2 3), (3 4) that the current and
// the next two windows use.
struct Win {
  double F2, F3, F4, D1, D2, D3, D4;
  Diff d4;
  Num a0, b0, c0, b1, c1, c2;  // pair (1 2) a, (2 3) b, (3 4) c
  JANC_HD void init(double F0, double F1, double f2, double f3, double f4, const Eps& eps) {
    F2 = f2; F3 = f3; F4 = f4;
    D1 = sub_rn(F1, F0); D2 = sub_rn(F2, F1); D3 = sub_rn(F3, F2); D4 = sub_rn(F4, F3);
    Diff d1, d2, d3;
    d1.set(D1); d2.set(D2); d3.set(D3); d4.set(D4);
    a0 = pair_forms(D1, D2, d1, d2, eps).c0;
    const Forms b = pair_forms(D2, D3, d2, d3, eps);
    b0 = b.c0; b1 = b.c1;
    const Forms c = pair_forms(D3, D4, d3, d4, eps);
    c0 = c.c0; c1 = c.c1; c2 = c.c2;
  }
  JANC_HD void push(double Fn, const Eps& eps) {
    const double Dn = sub_rn(Fn, F4);
    F2 = F3; F3 = F4; F4 = Fn;
    Diff dn;
    dn.set(Dn);
    const Forms f = pair_forms(D4, Dn, d4, dn, eps);
    D1 = D2; D2 = D3; D3 = D4; D4 = Dn;
    d4 = dn;
    a0 = b0; b0 = c0; c0 = f.c0;
    b1 = c1; c1 = f.c1;
    c2 = f.c2;
  }
  // F+ at the right face of cell 2: substencils 0, 1, 2 from the left.
  JANC_HD Weights weights_plus() const { return Weights(a0, b1, c2); }
  // F- at the left face of cell 2: the mirror image.
  JANC_HD Weights weights_minus() const { return Weights(c2, b1, a0); }
};

// c1 D1 + .. + c4 D4 added to r.
JANC_HD double offset_plus(const Win& P, const Coef& p) {
  return fma(-p.k4, P.D4, fma(-p.k1, P.D1, fma(p.k3, P.D3, mul_rn(p.k2, P.D2))));
}
JANC_HD double offset_minus(const Win& M, const Coef& m, double r) {
  return fma(m.k4, M.D1, fma(m.k1, M.D4, fma(-m.k3, M.D2, fma(-m.k2, M.D3, r))));
}
// F+ of window P plus F- of window M at their common face: the eight small
// terms first, then the two centre values.
JANC_HD double face_sum(const Win& P, const Coef& p, const Win& M, const Coef& m) {
  return sub_rn(sub_rn(P.F2, -M.F2), -offset_minus(M, m, offset_plus(P, p)));
}

// The derivative of one reconstruction with respect to its window's
// differences D1..D4 in the stencil's own direction (for F-: D4..D1 with the
// sign changed): with q_k the substencils' offsets and r their weighted mean,
// both less F_2,
//   dr/dD_m = c_m + sum_k h_k dC_k/dD_m, h_k = -2 (w_k / C_k) (q_k - r),
// C_k = 3 (beta_k + eps) and dC_k/dD_m linear in the pair's differences.
// w_k / C_k comes from the products of the weights and one more reciprocal,
// that of C_0 C_1 C_2.
JANC_HD void derivative(const Num& s0, const Num& s1, const Num& s2, const Weights& w, const Coef& c, double D1,
                        double D2, double D3, double D4, double r, double* g) {
  int z;
  const u64 y = recip(mulhi(w.p12, s0.n), &z);
  // 1 / C_0 = mulhi(p12, y) 2^(z - 127 + 2103 - e_0); twice the sixth of the weight over C_k
  const int b = w.x + z + 1 - 127 + 2103;
  const double G0 = to_double(mulhi(w.u0, mulhi(w.p12, y)), b - 5 - 2 * w.d0 - s0.e + 64);
  const double G1 = to_double(3 * (mulhi(w.u1, mulhi(w.p02, y)) >> 2), b - 2 - 2 * w.d1 - s1.e + 64);
  const double G2 = to_double(3 * (mulhi(w.u2, mulhi(w.p01, y)) >> 2), b - 3 - 2 * w.d2 - s2.e + 64);
  // 6 (r - q_k)
  const double h0 = G0 * fma(6.0, r, fma(-5.0, D2, 2.0 * D1));
  const double h1 = G1 * fma(6.0, r, fma(-2.0, D3, -D2));
  const double h2 = G2 * fma(6.0, r, fma(-4.0, D3, D4));
  double a = h0 * D1, t = h0 * D2;
  g[0] = fma(8.0, a, fma(-11.0, t, -c.k1));
  g[1] = fma(20.0, t, fma(-11.0, a, c.k2));
  a = h1 * D2; t = h1 * D3;
  g[1] = fma(8.0, a, fma(-5.0, t, g[1]));
  g[2] = fma(8.0, t, fma(-5.0, a, c.k3));
  a = h2 * D3; t = h2 * D4;
  g[2] = fma(20.0, a, fma(-11.0, t, g[2]));
  g[3] = fma(8.0, t, fma(-11.0, a, -c.k4));
}
// The derivatives of the F+ and the F- reconstruction with respect to the
// window's D1..D4.
JANC_HD void derivative_plus(const Win& P, const Weights& w, const Coef& c, double* g) {
  derivative(P.a0, P.b1, P.c2, w, c, P.D1, P.D2, P.D3, P.D4, offset_plus(P, c), g);
}
JANC_HD void derivative_minus(const Win& M, const Weights& w, const Coef& c, double* g) {
  // with the differences D'_1 = -D4 .. D'_4 = -D1; all of them negated below,
  // which turns r - q and the products h D' but not the derivatives' values
  double t[4];
  derivative(M.c2, M.b1, M.a0, w, c, M.D4, M.D3, M.D2, M.D1, -offset_minus(M, c, 0.0), t);
  g[0] = -t[3]; g[1] = -t[2]; g[2] = -t[1]; g[3] = -t[0];
}

}  // namespace weno

#ifdef __CUDACC__
// The split fluxes of one (variable, line) from its staged cells: value w of
// lp U (+ pt), lm U (+ pt).
struct SplitLine {
  const double *U, *lp, *lm, *pt;
  __device__ __forceinline__ double plus(int w) const { return pt ? fma(lp[w], U[w], pt[w]) : __dmul_rn(lp[w], U[w]); }
  __device__ __forceinline__ double minus(int w) const { return pt ? fma(lm[w], U[w], pt[w]) : __dmul_rn(lm[w], U[w]); }
  __device__ __forceinline__ void init(weno::Win& P, weno::Win& M, const weno::Eps& eps) const {
    P.init(plus(0), plus(1), plus(2), plus(3), plus(4), eps);
    M.init(minus(1), minus(2), minus(3), minus(4), minus(5), eps);
  }
};

// One (variable, line): reconstructs F+ (window starting at cell w = 0) and
// F- (window starting at w = 1) at every face of the line, two independent
// dependency chains per thread, and stores F^ = F+^ + F-^ at out[t * stride].
__device__ __forceinline__ void slide_line2(const SplitLine& L, double eps4, int nf, double* __restrict__ out,
                                            long long stride) {
  const weno::Eps eps(eps4);
  weno::Win P, M;
  L.init(P, M, eps);
  for (int t = 0; t < nf; ++t) {
    const weno::Coef cp(P.weights_plus()), cm(M.weights_minus());
    out[(long long)t * stride] = weno::face_sum(P, cp, M, cm);
    if (t + 1 < nf) {
      P.push(L.plus(t + 5), eps);
      M.push(L.minus(t + 6), eps);
    }
  }
}

// slide_line2 that also stores, per face, the derivatives of both
// reconstructions with respect to their window differences: component c (0..3:
// F+ window D1..D4, 4..7: F- window) of face t at lin[c * cstride + t * fstride].
// The face values are slide_line2's bit for bit.
__device__ __forceinline__ void slide_line2_lin(const SplitLine& L, double eps4, int nf, double* __restrict__ out,
                                                long long stride, double* __restrict__ lin, long long fstride,
                                                long long cstride) {
  const weno::Eps eps(eps4);
  weno::Win P, M;
  L.init(P, M, eps);
  for (int t = 0; t < nf; ++t) {
    double g[4];
    double* l = lin + (long long)t * fstride;
    const weno::Weights wp = P.weights_plus();
    const weno::Coef cp(wp);
    weno::derivative_plus(P, wp, cp, g);
#pragma unroll
    for (int c = 0; c < 4; ++c) l[c * cstride] = g[c];
    const weno::Weights wm = M.weights_minus();
    const weno::Coef cm(wm);
    weno::derivative_minus(M, wm, cm, g);
#pragma unroll
    for (int c = 0; c < 4; ++c) l[(4 + c) * cstride] = g[c];
    out[(long long)t * stride] = weno::face_sum(P, cp, M, cm);
    if (t + 1 < nf) {
      P.push(L.plus(t + 5), eps);
      M.push(L.minus(t + 6), eps);
    }
  }
}
#endif

}  // namespace janc
