// WENO5-JS reconstruction along a line of split fluxes, shared by the
// single-grid, the block (AMR) and the adjoint face kernels.
//
// The reconstruction costs the FP64 pipe little: with D_j = F_j - F_{j-1} the
// differences of the five values of a window, the face value is F_2 plus
//   r = (w0 Q0 + w1 Q1 + w2 Q2) / 6,
//   Q0 = 5 D2 - 2 D1, Q1 = D2 + 2 D3, Q2 = 4 D3 - D4
// with the nonlinear weights w_k of the three substencils. Only the split
// fluxes, D_j, and the final products and sums are FP64 operations (8 per face
// for both split signs). The weights and the weighted sum of the Q_k are formed
// on 64-bit integers (janc_soft.cuh): weights accurate to about 2^-55, the sum
// to 2^-51 or better of its largest term, which the FP64 pipe's own evaluation
// (about 2^-51) does not reach. 2048 x 256, 12 variables, both directions:
// 0.597 ms with the coefficients of the D_j as doubles (14 FP64 instructions a
// face), 0.557 ms with the sum on integers; with the derivatives (1000 x 400,
// 6 variables) 1.05 and 0.56 ms.
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

// One difference: its mantissa in [2^63, 2^64), exponent field, sign (all ones
// if negative) and square.
struct Diff {
  u64 m, sq;
  int e, neg;
  JANC_HD void set(double D) {
    const u64 b = bits_of(D);
    e = (int)(hi32(b) >> 20) & 0x7ff;
    neg = (int)hi32(b) >> 31;
    m = (b << 11) | (1ull << 63);
    sq = sqhi(m);
  }
};
JANC_HD long long with_sign(u64 x, int neg) {
  const u64 s = ((u64)(u32)neg << 32) | (u32)neg;
  return (long long)((x ^ s) - s);
}

// An adjacent pair of differences as signed integers below 2^58 in units of
// 2^(e - 1080), e the larger exponent field.
struct Pair {
  long long a, b;
  int e;
};

// 3 (beta + epsilon) of the pair (a, b) as substencil 0, 1 and 2, in units of
// 2^-2103.
struct Forms {
  Num c0, c1, c2;
};
JANC_HD Forms pair_forms(const Diff& a, const Diff& b, const Eps& eps, Pair& p) {
  p.e = a.e > b.e ? a.e : b.e;
  p.a = with_sign(shr(a.m, p.e - a.e + 6), a.neg);
  p.b = with_sign(shr(b.m, p.e - b.e + 6), b.neg);
  const int e = p.e > eps.e_min ? p.e : eps.e_min;
  const int da = e - a.e, db = e - b.e;
  const u64 A = shr(a.sq, 2 * da + 5), B = shr(b.sq, 2 * db + 5);
  const u64 C = shr(mulhi(a.m, b.m), da + db + 5);
  const u64 X = (u64)with_sign(C, ~(a.neg ^ b.neg));  // -D_a D_b
  const u64 t = ((A + B) << 2) + shr(eps.n, 2 * (e - eps.e_min));
  const u64 u = t + 11 * X;
  return Forms{normal(u + 6 * B, 2 * e), normal(t + 5 * X, 2 * e), normal(u + 6 * A, 2 * e)};
}

// Weights of substencils with indicators s0, s1, s2 and linear weights
// 1 : 6 : 3. The weights are 1/s_k^2 up to a common factor; with s0^2 s1^2 s2^2
// as that factor they are the squares u_k 2^(-2 d_k) of the products
// p12 = s1 s2 and so on (upper halves), each with its own exponent, so that a
// weight keeps its relative accuracy however small it is. y 2^x is 2^127 over
// 1.5 times their sum / 16.
struct Weights {
  u64 u0, u1, u2, p12, p02, p01, y;
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
    y = recip(s + (s >> 1), &x);
  }
};

// The weighted mean r = n y of the substencils' offsets (Q_k / 6): Q_k as
// integers in units of 2^(e_k - 1080) below 7 2^58, 3 2^58, 5 2^58. Their
// products with the weights are aligned to the largest and summed below 2^63.
// Not finite where a difference was not. s, t: the sum and its exponent,
// r = s y 2^(t + x - 1149) with y and x of the weights.
struct Mean {
  double n, y;
  long long s;
  int t;
  bool bad;
  JANC_HD Mean(const Weights& w, long long q0, int e0, long long q1, int e1, long long q2, int e2) {
    const int t0 = e0 - 2 * w.d0, t1 = e1 - 2 * w.d1 + 2, t2 = e2 - 2 * w.d2 + 1;  // weights 1, 4 (1.5), 2 (1.5)
    t = t0 > t1 ? t0 : t1;
    t = t > t2 ? t : t2;
    const long long v = sar(mulhi_signed(w.u1, q1), t - t1) + sar(mulhi_signed(w.u2, q2), t - t2);
    s = sar(mulhi_signed(w.u0, q0), t - t0) + v + (v >> 1);
    n = scaled_double(s, t + w.x - 1085);
    int e = e0 > e1 ? e0 : e1;
    e = e > e2 ? e : e2;
    bad = e > 2000;
    if (bad) n = double_of(0x7ff8000000000000ull);
    y = round_double(w.y, -1);
  }
};

// The sizes |c1|, c2, c3, |c4| of the derivatives of r at fixed weights
// (r = -c1 D1 + c2 D2 + c3 D3 - c4 D4), in the stencil's own direction, and a
// sixth of each weight: w0 = u0 2^(x - 5 - 2 d0), w1 = 3 u1 2^(x - 4 - 2 d1),
// w2 = 3 u2 2^(x - 5 - 2 d2), all times 2^-64. c2 and c3 are sums of two
// weights aligned to the larger one.
struct Coef {
  u64 u0, u1, u2;
  double k1, k2, k3, k4;
  JANC_HD explicit Coef(const Weights& w) : u0(mulhi(w.u0, w.y)), u1(mulhi(w.u1, w.y)), u2(mulhi(w.u2, w.y)) {
    const u64 v1 = u1 >> 3, v2 = u2 >> 3;
    // a weight below 2^-960 as one of that size: its exponent stays that of a double
    const int d0 = w.d0 < 480 ? w.d0 : 480, d1 = w.d1 < 480 ? w.d1 : 480, d2 = w.d2 < 480 ? w.d2 : 480;
    const int m = d0 < d1 ? d0 : d1, n = d1 < d2 ? d1 : d2;
    k1 = to_double(u0, w.x - 4 - 2 * d0);
    k2 = to_double(3 * shr(v1, 2 * (d1 - m)) + 5 * shr(u0, 2 * (d0 - m) + 4), w.x - 1 - 2 * m);
    k3 = to_double(3 * (shr(v1, 2 * (d1 - n)) + shr(v2, 2 * (d2 - n))), w.x - 2 * n);
    k4 = to_double(3 * (u2 >> 2), w.x - 3 - 2 * d2);
  }
};

// Sliding window of one split sign along a line: values F_2..F_4, the last
// difference, the pairs (1 2) A, (2 3) B, (3 4) C of differences and the forms
// that the current and the next two windows use of them.
struct Win {
  double F2, F3, F4;
  Diff d4;
  Pair A, B, C;
  Num a0, b0, c0, b1, c1, c2;  // pair A: a, B: b, C: c
  JANC_HD void init(double F0, double F1, double f2, double f3, double f4, const Eps& eps) {
    F2 = f2; F3 = f3; F4 = f4;
    Diff d1, d2, d3;
    d1.set(sub_rn(F1, F0)); d2.set(sub_rn(F2, F1)); d3.set(sub_rn(F3, F2)); d4.set(sub_rn(F4, F3));
    a0 = pair_forms(d1, d2, eps, A).c0;
    const Forms b = pair_forms(d2, d3, eps, B);
    b0 = b.c0; b1 = b.c1;
    const Forms c = pair_forms(d3, d4, eps, C);
    c0 = c.c0; c1 = c.c1; c2 = c.c2;
  }
  JANC_HD void push(double Fn, const Eps& eps) {
    Diff dn;
    dn.set(sub_rn(Fn, F4));
    F2 = F3; F3 = F4; F4 = Fn;
    A = B; B = C;
    const Forms f = pair_forms(d4, dn, eps, C);
    d4 = dn;
    a0 = b0; b0 = c0; c0 = f.c0;
    b1 = c1; c1 = f.c1;
    c2 = f.c2;
  }
  // F+ at the right face of cell 2: substencils 0, 1, 2 from the left.
  JANC_HD Weights weights_plus() const { return Weights(a0, b1, c2); }
  JANC_HD Mean mean_plus(const Weights& w) const {
    return Mean(w, 5 * A.b - 2 * A.a, A.e, B.a + 2 * B.b, B.e, 4 * C.a - C.b, C.e);
  }
  // F- at the left face of cell 2: the mirror image, whose differences run
  // backwards with the sign changed. The mean is that of the unchanged signs.
  JANC_HD Weights weights_minus() const { return Weights(c2, b1, a0); }
  JANC_HD Mean mean_minus(const Weights& w) const {
    return Mean(w, 5 * C.a - 2 * C.b, C.e, B.b + 2 * B.a, B.e, 4 * A.b - A.a, A.e);
  }
};

// F+ of window P plus F- of window M at their common face: the two small
// terms first, then the two centre values.
JANC_HD double face_sum(const Win& P, const Mean& p, const Win& M, const Mean& m) {
  return sub_rn(sub_rn(P.F2, -M.F2), -fma(-m.n, m.y, mul_rn(p.n, p.y)));
}

// The derivative of one reconstruction with respect to its window's
// differences in the stencil's own direction, d_1..d_4: with r their weighted
// mean of the substencils' offsets q_k = Q_k / 6,
//   dr/dd_m = c_m + sum_k h_k dC_k/dd_m, h_k = -2 (w_k / C_k) (q_k - r),
// C_k = 3 (beta_k + eps) and dC_k/dd_m linear in the pair's differences.
// w_k / C_k comes from the products of the weights and one more reciprocal,
// that of C_0 C_1 C_2. (a_k, b_k): the pair of substencil k, first difference
// first, in units of 2^(e_k - 1080): Q_k and dC_k/dd_m are small integer
// combinations of them, and h_k is formed on integers too, so that six FP64
// instructions are left of 30 (1000 x 400, 6 variables: 0.51 ms a launch, 0.56 with
// h_k as doubles, 1.05 with all of it).

// 2 (w_k / C_k) 6 (r - q_k) = g (6 r - Q_k) 2^x, g 2^64 at least 2^55: 6 r = v
// 2^(ev - 1080), Q_k = q 2^(e - 1080), aligned to the larger.
JANC_HD double weighted_gap(u64 g, int x, long long v, int ev, long long q, int e) {
  const int top = ev > e ? ev : e;
  const long long d = sar(v, top - ev) - sar(q, top - e);
  u64 m = d < 0 ? 0ull - (u64)d : (u64)d;
  x += top - 1080;
  if (hi32(m) == 0) {
    m <<= 32;
    x -= 32;
  }
  int z = leading_zeros(hi32(m));  // 158 for 0
  const u64 p = mulhi(g, shl(m, z));
  const int f = 1085 + x - z;
  z = leading_zeros(hi32(p));
  const u64 b = (shl(p, z) >> 11) + ((u64)((u32)(f - z) << 20 | (hi32((u64)d) & 0x80000000u)) << 32);
  return double_of(f - z < 0 || p == 0 ? 0ull : b);
}
JANC_HD void derivative(const Num& s0, const Num& s1, const Num& s2, const Weights& w, const Coef& c, const Mean& r,
                        long long a0, long long b0, int e0, long long a1, long long b1, int e1, long long a2,
                        long long b2, int e2, double* g) {
  int z;
  const u64 y = recip(mulhi(w.p12, s0.n), &z);
  // 1 / C_0 = mulhi(p12, y) 2^(z - 127 + 2103 - e_0); twice the sixth of the weight over C_k
  const int b = w.x + z + 1 - 127 + 2103;
  const long long ri = mulhi_signed(w.y, r.s);
  const long long v = (ri + (ri >> 1)) >> 1;  // 6 r in units of 2^(ev - 1080), below 2^62
  const int ev = r.t + w.x - 2;
  double h0 = weighted_gap(mulhi(c.u0, mulhi(w.p12, y)), b - 5 - 2 * w.d0 - s0.e + 64, v, ev, 5 * b0 - 2 * a0, e0);
  double h1 = weighted_gap(3 * (mulhi(c.u1, mulhi(w.p02, y)) >> 2), b - 2 - 2 * w.d1 - s1.e + 64, v, ev, a1 + 2 * b1, e1);
  double h2 = weighted_gap(3 * (mulhi(c.u2, mulhi(w.p01, y)) >> 2), b - 3 - 2 * w.d2 - s2.e + 64, v, ev, 4 * a2 - b2, e2);
  if (r.bad) h0 = h1 = h2 = double_of(0x7ff8000000000000ull);
  e0 -= 1080;
  e1 -= 1080;
  e2 -= 1080;
  g[0] = fma(h0, scaled_double(8 * a0 - 11 * b0, e0), -c.k1);
  g[1] = fma(h1, scaled_double(8 * a1 - 5 * b1, e1), fma(h0, scaled_double(20 * b0 - 11 * a0, e0), c.k2));
  g[2] = fma(h2, scaled_double(20 * a2 - 11 * b2, e2), fma(h1, scaled_double(8 * b1 - 5 * a1, e1), c.k3));
  g[3] = fma(h2, scaled_double(8 * b2 - 11 * a2, e2), -c.k4);
}
// The derivatives of the F+ and the F- reconstruction with respect to the
// window's D1..D4.
JANC_HD void derivative_plus(const Win& P, const Weights& w, const Mean& r, double* g) {
  derivative(P.a0, P.b1, P.c2, w, Coef(w), r, P.A.a, P.A.b, P.A.e, P.B.a, P.B.b, P.B.e, P.C.a, P.C.b, P.C.e, g);
}
JANC_HD void derivative_minus(const Win& M, const Weights& w, const Mean& r, double* g) {
  // the stencil's differences are -D4..-D1: the signs of r and q_k change, h_k
  // times a difference does not, and neither do the derivatives' values but for
  // the sign of dd/dD
  double t[4];
  derivative(M.c2, M.b1, M.a0, w, Coef(w), r, M.C.b, M.C.a, M.C.e, M.B.b, M.B.a, M.B.e, M.A.b, M.A.a, M.A.e, t);
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
    const weno::Mean rp = P.mean_plus(P.weights_plus()), rm = M.mean_minus(M.weights_minus());
    out[(long long)t * stride] = weno::face_sum(P, rp, M, rm);
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
    const weno::Mean rp = P.mean_plus(wp);
    weno::derivative_plus(P, wp, rp, g);
#pragma unroll
    for (int c = 0; c < 4; ++c) l[c * cstride] = g[c];
    const weno::Weights wm = M.weights_minus();
    const weno::Mean rm = M.mean_minus(wm);
    weno::derivative_minus(M, wm, rm, g);
#pragma unroll
    for (int c = 0; c < 4; ++c) l[(4 + c) * cstride] = g[c];
    out[(long long)t * stride] = weno::face_sum(P, rp, M, rm);
    if (t + 1 < nf) {
      P.push(L.plus(t + 5), eps);
      M.push(L.minus(t + 6), eps);
    }
  }
}
#endif

}  // namespace janc
