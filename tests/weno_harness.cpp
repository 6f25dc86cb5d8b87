// Test harness: the WENO5 reconstruction of the face kernels (janc_weno.cuh,
// 64-bit integer weights) compiled for the host behind a C ABI, so that the
// CPU tests can compare it with exact arithmetic. Built by the tests with the
// host C++ compiler; not part of the library.
#include "../paper_2504_13750_gb300/csrc/janc_weno.cuh"

using namespace janc;

extern "C" {

// n windows of 6 values each: sum[i] = F+ of values 0..4 plus F- of values
// 1..5 at their common face, reached by `slide` pushes from a window of
// 6 + slide values (F: n x (6 + slide)); d[8 i ..] the derivatives with respect
// to the differences of the F+ and the F- window.
void wh_faces(int n, int slide, const double* Fp, const double* Fm, double eps, double* sum, double* d) {
  const weno::Eps e(4.0 * eps);
  const int len = 6 + slide;
  for (int i = 0; i < n; ++i) {
    const double *p = Fp + (long)i * len, *m = Fm + (long)i * len;
    weno::Win P, M;
    P.init(p[0], p[1], p[2], p[3], p[4], e);
    M.init(m[1], m[2], m[3], m[4], m[5], e);
    for (int t = 0; t < slide; ++t) {
      P.push(p[t + 5], e);
      M.push(m[t + 6], e);
    }
    const weno::Weights wp = P.weights_plus(), wm = M.weights_minus();
    const weno::Mean rp = P.mean_plus(wp), rm = M.mean_minus(wm);
    sum[i] = weno::face_sum(P, rp, M, rm);
    weno::derivative_plus(P, wp, rp, d + 8 * i);
    weno::derivative_minus(M, wm, rm, d + 8 * i + 4);
  }
}

// e^x, ln x and 1/x, elementwise.
void wh_functions(int n, const double* x, double* e, double* l, double* r) {
  for (int i = 0; i < n; ++i) {
    e[i] = soft::exp_double(x[i]);
    l[i] = soft::log_double(x[i]);
    r[i] = soft::rcp_double(x[i]);
  }
}
// sqrt(d / 2^64) in units of 2^-64, and a 2^e as a double.
void wh_sqrt(int n, const unsigned long long* d, unsigned long long* s) {
  for (int i = 0; i < n; ++i) s[i] = soft::sqrt_q(d[i]);
}
void wh_signed(int n, const long long* a, int e, double* x) {
  for (int i = 0; i < n; ++i) x[i] = soft::signed_double(a[i], e);
}

// a 2^e as a double, 0 below the normal range; 2^(a 2^-54); x cut to a float and back.
void wh_scaled(int n, const long long* a, int e, double* x) {
  for (int i = 0; i < n; ++i) x[i] = soft::scaled_double(a[i], e);
}
void wh_exp2(int n, const long long* a, double* x) {
  for (int i = 0; i < n; ++i) x[i] = soft::exp2_fixed(a[i]);
}
void wh_float(int n, const double* x, double* y) {
  for (int i = 0; i < n; ++i) y[i] = soft::widen(soft::cut_float(x[i]));
}

// y[i] = 2^127 / (x[i] 2^z[i]) and b[i] = x[i] 2^-64 as a double.
void wh_soft(int n, const unsigned long long* x, unsigned long long* y, int* z, double* b) {
  for (int i = 0; i < n; ++i) {
    y[i] = soft::recip(x[i], z + i);
    b[i] = soft::to_double(x[i], 0);
  }
}

}  // extern "C"
