// Device-side data layout and helpers shared by the kernels of the reacting-
// flow step (arXiv 2504.13750, Sec. 4). State and results are FP64; arithmetic is FP64
// or 64-bit integer, but for the start of the Newton recovery (newton_cell).
//
// GB300 notes that shape this code: the FP64 pipe issues about 2 DFMA per
// clock per SM (roughly 1/64 of the FP32 rate), while integer, FP32, load and
// shuffle instructions issue at full rate. So every operation that can be
// done exactly outside the FP64 pipe is done there: maxima of non-negative
// doubles compare their bit patterns as integers, absolute values clear the
// sign bit, pivot searches and row swaps are integer compares and selects,
// and reciprocals, exponentials, logarithms, square roots and the mixture sums
// are formed on 64-bit integers (janc_soft.cuh).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "janc_soft.cuh"

namespace janc {

constexpr double RU = 8.314472;     // universal gas constant (text after Eq. 4.5)
constexpr double P_REF = 101325.0;  // reference pressure of Eq. 4.9
constexpr int MAX_NS = 9;
constexpr int MAX_NR = 32;
constexpr int MAX_SIDE = 3;  // distinct species per reaction side

enum : int { ST_NONFINITE = 1, ST_NONPOSITIVE = 2, ST_NEWTON_FAIL = 4, ST_SINGULAR = 8 };
// BC_HALO marks an x side shared with the neighbouring slab of an x-slab
// decomposition (Sec. 4.4): its 3 ghost columns are read from a halo buffer
// that the exchange fills, not derived from the slab's own cells.
enum : int { BC_WALL = 0, BC_ZEROGRAD = 1, BC_PERIODIC = 2, BC_HALO = 3 };

// Mechanism in the form the kernels consume (built on the host from the
// user's table, copied once to device memory).
struct MechDev {
  int ns, nr;
  double M[MAX_NS];
  double invM[MAX_NS];
  // Enthalpy polynomial h_k/(Ru/M_k) = sum_{m<5} hc[k][m] T^{m+1} + hc[k][5]
  // with hc[k][m] = a_m/(m+1) (Eq. 4.4).
  double hc[MAX_NS][6];
  // Dimensionless Gibbs term of Eq. 4.9, G_k = s_k/R - h_k/(RT) (Eq. 4.4-4.5):
  // G = gc0 ln T + gc6 + T (gc1 + T (gc2 + T (gc3 + T gc4))) + gc5 / T with
  // gc0 = a0, gc1 = a1/2, gc2 = a2/6, gc3 = a3/12, gc4 = a4/20, gc5 = -a5,
  // gc6 = a6 - a0.
  double gc[MAX_NS][7];
  // Reactions (Eq. 4.6-4.8): ln k_f = lnA + b ln T - EaR / T.
  double lnA[MAX_NR], b[MAX_NR], EaR[MAX_NR];
  int nre[MAX_NR], rsp[MAX_NR][MAX_SIDE], rnu[MAX_NR][MAX_SIDE];
  int npr[MAX_NR], psp[MAX_NR][MAX_SIDE], pnu[MAX_NR][MAX_SIDE];
  int dnu[MAX_NR];  // sum of (nu_b - nu_f)
  int tb[MAX_NR];
  double rnud[MAX_NR][MAX_SIDE], pnud[MAX_NR][MAX_SIDE];  // the coefficients as doubles
  // Third-body factor as sum_j X_j + sum over the few species whose
  // coefficient differs from one: neff entries of (species, eff - 1).
  int neff[MAX_NR], effsp[MAX_NR][MAX_NS];
  double effv[MAX_NR][MAX_NS];
  double effm1[MAX_NR][MAX_NS];  // third-body coefficient minus one
  // Column factor for the Jacobian in carried variables (text after Eq. 4.13):
  // eff_il - (M_l / M_ns) eff_i,ns for l < ns - 1.
  double ceff[MAX_NR][MAX_NS];
  double mratio[MAX_NS];  // M_l / M_ns
  double third[MAX_NS];   // 1 - M_l / M_ns: ceff of a reaction whose coefficients are all one
  // Mixture sums in the carried variables: since rho Y_ns = rho - sum_{k<ns-1}
  // rho Y_k, sum_k (rho Y_k / M_k) c_k = rho cN + sum_{k<ns-1} rho Y_k cd_k
  // with cN = c_ns / M_ns and cd_k = c_k / M_k - cN. For the enthalpy
  // coefficients (hcN, hcd) and for c = 1 (WN, Wd: W = sum_k z_k).
  double hcN[6];
  double hcd[MAX_NS][6];
  double WN;
  double Wd[MAX_NS];
  // The same sums on integers: row 0 is W, row 1 + q coefficient q; entry 0
  // multiplies rho, entry 1 + k rho Y_k. A coefficient is +-n 2^(mixe - 64)
  // 2^mixp (mixs: the sign as a mask); 2^mixp is 1/M_k over 1/M_ns to a power
  // of two, moved over to the variable so that a light species' large
  // coefficients do not cost the others their low bits.
  unsigned long long mixn[7][MAX_NS];
  unsigned mixs[7][MAX_NS];
  int mixe[7], mixp[MAX_NS];
  int mix_ok;  // every mixe within +-400
  // G_k and ln k_f as base-2 logarithms in fixed point (fixed_T and below): gq in the
  // order of gc, the factor of log2 T in units of 2^-58, those of (T / 8192)^m and
  // the constant of 2^-54, that of 1/T of 2^-46; kq: ln A, b, -Ea/R likewise;
  // lref = log2(Ru / P_ref) in units of 2^-54. rate_ok: the numbers fit, and every
  // log2 k_f and log2 k_b stays within +-440 for T in [256, 8192).
  long long gq[MAX_NS][7], kq[MAX_NR][3], lref;
  int rate_ok;
};

// Grid constants passed by value to every kernel.
struct GridDev {
  int nx, ny;
  long long n;  // nx * ny
  double dx, dy, rdx, rdy;
  int bc[4];  // left, right, bottom, top
  double eps4;  // 4 * WENO epsilon (smoothness indicators are carried scaled by 4)
  double newton_tol;
  int newton_maxit;
  // Halo buffers of the x sides whose bc is BC_HALO: [nv + 4][ny][3] each,
  // the 3 columns nearest the side, plane by plane like the state (column c
  // of the low halo is ghost cell c - 3, of the high halo cell nx + c).
  const double* halo_lo;
  const double* halo_hi;
  // 1: the mechanism has the reaction structure compiled into the fixed
  // chemistry kernels (the same operations, every index a constant)
  int chem_fixed;
};

// One state buffer: planes 0..nv-1 conserved, nv: T, nv+1: u, nv+2: v, nv+3: p.
struct StateView {
  double* base;
  __host__ __device__ double* plane(int k, long long n) const { return base + (long long)k * n; }
};

// Per-step control: fixed dt (> 0) or CFL; alpha slots hold max(|u|+c),
// max(|v|+c) as the bit patterns of non-negative doubles.
struct StepCtl {
  double dt_fixed;
  double cfl;
  double hmin;       // min(dx, dy)
  double chem_frac;  // share of the step's dt taken by one chemistry launch: 1, or 1/2 in the Strang order
  int source;        // 1: the production rates are an explicit source of every RK stage
};

// One request of a batched (serving) launch: its grid constants and buffers.
// Alpha slots (2 x u64 each): 0 = U^n, 1 = U^1, 2 = U^2, 3 = U^*, 4 = U^{n+1}.
struct BatchReq {
  GridDev g;
  StateView S[3];
  double* Fx;
  double* Gy;
  unsigned long long* alpha;
  double* clock2;
  int* status;
  const MechDev* mech;
  StepCtl ctl;
  int nbx, ntx_x, ntx_y;  // face-flux tiling
  int ubx, uby;           // update-kernel blocks in x and y
  int fresh;              // 1 until the first batched step after admission
};

// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long dbits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ double bitsd(unsigned long long b) { return __longlong_as_double((long long)b); }
// |x| by clearing the sign bit (integer pipe).
__device__ __forceinline__ double dabs(double x) { return bitsd(dbits(x) & 0x7fffffffffffffffull); }
__device__ __forceinline__ bool finite_bits(double x) {
  return ((dbits(x) >> 52) & 0x7ff) != 0x7ff;
}

// x > 0 (false for NaN), on the bits.
__device__ __forceinline__ bool positive_bits(double x) {
  return dbits(x) - 1ull < 0x7ff0000000000000ull;
}

// Reciprocal, exponential and logarithm on integers (janc_soft.cuh). As FP64
// sequences they were 3, 10 and about 25 FP64 instructions (16 clocks each),
// here 30, 70 and 75 instructions of which the SM starts four a clock.
__device__ __forceinline__ double rcp(double d) { return soft::rcp_double(d); }

// e^x; results that would overflow give +inf, results below the normal range
// 0, NaN stays NaN.
__device__ __forceinline__ double exp_t(double x) {
  if ((__double2hiint(x) & 0x7fffffff) < 0x40862000) return soft::exp_double(x);  // |x| < 708
  const double r = exp(x);
  return r < 0x1p-1022 ? 0.0 : r;
}

__device__ __forceinline__ double log_t(double x) {
  const int h = __double2hiint(x);
  if (h >= 0x40000000 && h < 0x7fd00000) return soft::log_double(x);  // [2, 2^1022)
  return log(x);
}

// dt of the step from the alpha slot of its starting state (cfl() of Sec. 4.3).
__device__ __forceinline__ double step_dt(const StepCtl& c, const unsigned long long* a0) {
  if (c.dt_fixed > 0.0) return c.dt_fixed;
  unsigned long long ax = a0[0], ay = a0[1];
  double amax = bitsd(ax > ay ? ax : ay);
  return c.cfl * c.hmin / amax;
}

// W = sum_k z_k and the first NH mixture enthalpy coefficients
// h[q] = sum_k z_k hc_k[q] (z_k = rho Y_k / M_k) from the carried variables,
// through the folded tables of MechDev. On integers: the variables aligned to
// the largest one, 62 bits each, products kept to their upper halves; an
// error of 2^-58 of the largest term of a sum, with ns terms about 10
// instructions each (an FP64 term is one, but of 16 clocks). Variables that
// are not finite, extreme (beyond about 2^+-500), or whose sizes add up to more
// than a word holds, take the FP64 sums.
template <int NS, int NH>
__device__ __forceinline__ void mixture_sums(const double* u, const MechDev& m, double& W, double* h) {
  using namespace soft;
  if (NS > 1) {
    u64 x[NS];
    unsigned neg[NS];
    int e[NS], E = 0;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const Parts p(k ? u[3 + k] : u[0]);
      x[k] = p.m;
      neg[k] = p.neg ? 0xffffffffu : 0u;
      e[k] = p.e + (k ? m.mixp[k] : 0);
      E = e[k] > E ? e[k] : E;
    }
    unsigned total = 0;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      x[k] = shr(x[k], E - e[k] + 2);
      total += hi32(x[k]) >> 3;
    }
    if (m.mix_ok && E >= 512 && E < 1536 && total < (1u << 28) - NS) {
#pragma unroll
      for (int q = 0; q <= NH; ++q) {
        u64 s = 0;
#pragma unroll
        for (int k = 0; k < NS; ++k) {
          const unsigned f = neg[k] ^ m.mixs[q][k];
          const u64 t = mulhi(x[k], m.mixn[q][k]);
          s += (t ^ (((u64)f << 32) | f)) + (f & 1u);
        }
        const double v = signed_double((long long)s, E - 1084 + m.mixe[q]);
        if (q == 0) W = v; else h[q - 1] = v;
      }
      return;
    }
  }
  const double rho = u[0];
  W = rho * m.WN;
#pragma unroll
  for (int k = 0; k < NS - 1; ++k) W = fma(u[4 + k], m.Wd[k], W);
#pragma unroll
  for (int q = 0; q < NH; ++q) {
    double s = rho * m.hcN[q];
#pragma unroll
    for (int k = 0; k < NS - 1; ++k) s = fma(u[4 + k], m.hcd[k][q], s);
    h[q] = s;
  }
}

// sqrt(a b r / d), r a reciprocal: on integers for positive normal factors.
__device__ __forceinline__ double speed(double a, double b, double r, double d) {
  using namespace soft;
  const Parts pa(a), pb(b), pr(r), pd(d);
  const int lo = min(min(pa.e, pb.e), min(pr.e, pd.e)), hi = max(max(pa.e, pb.e), max(pr.e, pd.e));
  if (lo >= 512 && hi < 1536 && !(pa.neg | pb.neg | pr.neg | pd.neg)) {
    // a b r / d = n 2^(e - 64) with e even and n in [2^62, 2^64)
    const u64 t = mulhi(mulhi(pa.m, pb.m), mulhi(pr.m, recip_normal(pd.m)));
    int e = pa.e + pb.e + pr.e - 1086 * 3 + 959 - pd.e + 64 * 3 + 64;
    const Num n = normal(t, e);
    e = n.e;
    const u64 s = sqrt_q((e & 1) ? n.n >> 1 : n.n);  // in [2^63, 2^64)
    e += e & 1;
    return round_double(s, e / 2 - 1);
  }
  return sqrt(a * b * r * rcp(d));
}

// Sound speed exactly as newton_cell finishes it, from the stored T.
template <int NS>
__device__ __forceinline__ double sound_speed(const double* u, double t, const MechDev& m) {
  const double rrho = rcp(u[0]);
  double W, h[5];
  mixture_sums<NS, 5>(u, m, W, h);
  const double c1 = 2.0 * h[1], c2 = 3.0 * h[2], c3 = 4.0 * h[3], c4 = 5.0 * h[4];
  const double K1 = h[0] - W;
  const double Cv = fma(t, fma(t, fma(t, fma(t, c4, c3), c2), c1), K1);
  const double Cp = Cv + W;
  const double p = RU * W * t;
  return speed(Cp, p, rrho, Cv);
}

// G_k of Eq. 4.9.
__device__ __forceinline__ double gibbs(const MechDev& m, int k, double T, double lnT, double rT) {
  const double* c = m.gc[k];
  return fma(c[0], lnT, fma(c[5], rT, fma(T, fma(T, fma(T, fma(T, c[4], c[3]), c[2]), c[1]), c[6])));
}

// T in [256, 8192) = 2^e (1 + ..) for the fixed-point logarithms of the rate
// constants: L = log2 T in units of 2^-60, y = 2^(64 + e) / T, x = T / 8192 in units
// of 2^-64, lref = log2(Ru T / P_ref) in units of 2^-54. False where T is outside
// or the mechanism's numbers do not fit (MechDev::rate_ok).
struct FixedT {
  soft::u64 L, y, x;
  int e;
  long long lref;
};
__device__ __forceinline__ bool fixed_T(const MechDev& m, double T, FixedT& t) {
  const soft::Parts p(T);
  if (!m.rate_ok || p.neg || p.e < 1031 || p.e >= 1036) return false;
  t.e = p.e - 1023;
  t.L = ((soft::u64)t.e << 60) + (soft::log2_frac(p.m) >> 4);
  t.y = soft::recip_normal(p.m);
  t.x = soft::shr(p.m, 12 - t.e);
  t.lref = m.lref + (long long)(t.L >> 6);
  return true;
}
// c0 log2 T + c5 / T + c6 in units of 2^-54, the factors as in MechDev::kq.
__device__ __forceinline__ long long fixed_arrhenius(long long c6, long long c0, long long c5, const FixedT& t) {
  return c6 + soft::mulhi_signed(t.L, c0) + soft::sar(soft::mulhi_signed(t.y, c5), t.e - 8);
}
// G_k log2 e in units of 2^-54.
__device__ __forceinline__ long long fixed_gibbs(const MechDev& m, int k, const FixedT& t) {
  const long long* c = m.gq[k];
  long long p = soft::mulhi_signed(t.x, c[4]);
#pragma unroll
  for (int q = 3; q > 0; --q) p = soft::mulhi_signed(t.x, c[q] + p);
  return p + fixed_arrhenius(c[6], c[0], c[5], t);
}
// ln k_f and ln k_b of reaction i in FP64, lcr = ln(Ru T / P_ref).
__device__ __forceinline__ void log_rates(const MechDev& m, int i, double T, double lnT, double rT, double lcr,
                                          double& f, double& b) {
  f = fma(m.b[i], lnT, fma(-m.EaR[i], rT, m.lnA[i]));
  b = fma((double)m.dnu[i], lcr, f);
#pragma unroll 1
  for (int r = 0; r < m.nre[i]; ++r) b = fma(m.rnud[i][r], gibbs(m, m.rsp[i][r], T, lnT, rT), b);
#pragma unroll 1
  for (int r = 0; r < m.npr[i]; ++r) b = fma(-m.pnud[i][r], gibbs(m, m.psp[i][r], T, lnT, rT), b);
}

// Molar production rates (Eq. 4.7-4.9) of the carried species k < ns - 1 at
// (T, X(u)), for the explicit source-term form of the step.
template <int NS>
// keep (the discrete adjoint's store): k_f and k_b of reaction i go to
// keep[2i n + idx] and keep[(2i+1) n + idx].
__device__ __forceinline__ void carried_rates(const double* u, double T, const MechDev& m, double* wd,
                                              double* __restrict__ keep = nullptr, long long n = 0,
                                              long long idx = 0) {
  constexpr int NSP = NS - 1;
  double X[NS];
  double rest = u[0];
#pragma unroll
  for (int k = 0; k < NSP; ++k) {
    X[k] = u[4 + k] * m.invM[k];
    rest -= u[4 + k];
    wd[k] = 0.0;
  }
  X[NSP] = rest * m.invM[NSP];
  double Ctot = X[0];
#pragma unroll
  for (int k = 1; k < NS; ++k) Ctot += X[k];
  // the rate constants from their logarithms: fixed point, else FP64
  FixedT t;
  const bool fixed = fixed_T(m, T, t);
  long long G[NS];
  double lnT = 0.0, rT = 0.0, lcr = 0.0;
  if (fixed) {
#pragma unroll
    for (int k = 0; k < NS; ++k) G[k] = fixed_gibbs(m, k, t);
  } else {
    lnT = log_t(T);
    rT = rcp(T);
    lcr = log_t((RU / P_REF) * T);
  }
  for (int i = 0; i < m.nr; ++i) {
    const int nre = m.nre[i], npr = m.npr[i];
    double kf, kb;
    if (fixed) {
      const long long f = fixed_arrhenius(m.kq[i][0], m.kq[i][1], m.kq[i][2], t);
      long long b = f + m.dnu[i] * t.lref;
      for (int r = 0; r < nre; ++r) b += m.rnu[i][r] * G[m.rsp[i][r]];
      for (int r = 0; r < npr; ++r) b -= m.pnu[i][r] * G[m.psp[i][r]];
      kf = soft::exp2_fixed(f);
      kb = soft::exp2_fixed(b);
    } else {
      log_rates(m, i, T, lnT, rT, lcr, kf, kb);
      kf = exp_t(kf);
      kb = exp_t(kb);
    }
    if (keep) {
      keep[(2LL * i) * n + idx] = kf;
      keep[(2LL * i + 1) * n + idx] = kb;
    }
    double fwd = kf, bwd = kb;
    for (int r = 0; r < nre; ++r)
      for (int q = 0; q < m.rnu[i][r]; ++q) fwd *= X[m.rsp[i][r]];
    for (int r = 0; r < npr; ++r)
      for (int q = 0; q < m.pnu[i][r]; ++q) bwd *= X[m.psp[i][r]];
    double Mi = 1.0;
    if (m.tb[i]) {
      Mi = Ctot;
      for (int e = 0; e < m.neff[i]; ++e) Mi = fma(m.effv[i][e], X[m.effsp[i][e]], Mi);
    }
    const double q = Mi * (fwd - bwd);
    for (int r = 0; r < nre; ++r)
      if (m.rsp[i][r] < NSP) wd[m.rsp[i][r]] = fma(-m.rnud[i][r], q, wd[m.rsp[i][r]]);
    for (int r = 0; r < npr; ++r)
      if (m.psp[i][r] < NSP) wd[m.psp[i][r]] = fma(m.pnud[i][r], q, wd[m.psp[i][r]]);
  }
}

// Ghost-cell source index along one axis (3 layers, text after Eq. 4.11).
__device__ __forceinline__ int ghost_src(int i, int n, int bc_lo, int bc_hi, bool& flip) {
  flip = false;
  if (i < 0) {
    if (bc_lo == BC_WALL) { flip = true; return -1 - i; }
    if (bc_lo == BC_ZEROGRAD) return 0;
    return i + n;
  }
  if (i >= n) {
    if (bc_hi == BC_WALL) { flip = true; return 2 * n - 1 - i; }
    if (bc_hi == BC_ZEROGRAD) return n - 1;
    return i - n;
  }
  return i;
}

// Request that owns entry e of a flattened list with per-request starts
// first[0..nreq] (first[0] = 0): the last r with first[r] <= e.
__device__ __forceinline__ int batch_owner(const int* __restrict__ first, int nreq, int e) {
  int lo = 0, hi = nreq - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Block-wide max of two non-negative doubles (as bits) and OR of a status
// word, then one atomic per block. blockDim.x * blockDim.y <= 1024.
__device__ __forceinline__ void block_reduce_alpha_status(unsigned long long sx, unsigned long long sy, int st,
                                                          unsigned long long* alpha_out, int* status) {
  __shared__ unsigned long long red_x[32], red_y[32];
  __shared__ int red_s[32];
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  const int nthr = blockDim.x * blockDim.y;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long ox = __shfl_xor_sync(0xffffffffu, sx, o);
    unsigned long long oy = __shfl_xor_sync(0xffffffffu, sy, o);
    int os = __shfl_xor_sync(0xffffffffu, st, o);
    sx = ox > sx ? ox : sx;
    sy = oy > sy ? oy : sy;
    st |= os;
  }
  const int w = tid >> 5, lane = tid & 31;
  if (lane == 0) { red_x[w] = sx; red_y[w] = sy; red_s[w] = st; }
  __syncthreads();
  if (w == 0) {
    const int nw = (nthr + 31) >> 5;
    sx = lane < nw ? red_x[lane] : 0ull;
    sy = lane < nw ? red_y[lane] : 0ull;
    st = lane < nw ? red_s[lane] : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      unsigned long long ox = __shfl_xor_sync(0xffffffffu, sx, o);
      unsigned long long oy = __shfl_xor_sync(0xffffffffu, sy, o);
      int os = __shfl_xor_sync(0xffffffffu, st, o);
      sx = ox > sx ? ox : sx;
      sy = oy > sy ? oy : sy;
      st |= os;
    }
    if (lane == 0) {
      if (alpha_out) {
        atomicMax(alpha_out, sx);
        atomicMax(alpha_out + 1, sy);
      }
      if (st) atomicOr(status, st);
    }
  }
}

// Newton-Raphson T recovery (end of Sec. 4.2) from the energy, warm-started
// at Tw, followed by p (Eq. 4.2) and the frozen sound speed. The mixture is
// reduced to polynomial coefficients once per cell (mixture_sums):
//   H(T) = sum_k z_k h_k(T)/Ru with z_k = rho Y_k / M_k,
//   F(T) = H(T) - W T - rho e / Ru  (W = sum_k z_k, rho e = E - |rho u|^2 / (2 rho)),
//   F'(T) = sum_k z_k cv_k / Ru.
// Stops when |dT| <= tol * T after the update, or, with another iteration
// allowed to confirm it, at |dT| <= 2^-28 T: the next correction would be
// below T dT^2 F''/2F' < 2^-54 T. Returns status bits.
//
// Three iterations in single precision, then one in double with the second-order
// term of the root (Chebyshev's iteration; that term only, a 2^-36th of T at
// most, is formed in single precision), give the same T: accepted where that one
// step is below 2^-18 T and s, the term's share of it, below 2^-19. The third-order
// rest is then below 2^-55 T (2 s^2 of the step, and the third derivative's for heat
// capacities that vary on the scale of T); the rounding of F remains, as after any
// Newton step. 12 FP64 instructions instead of
// three iterations' 33 (of 143 in a stage update of 12 variables: 16.4 us at
// 512 x 64 then, 14.6 now; one variable's gas at 1021 x 257: 50.9 and 43.5 us). Anything
// else, so every state that does not converge at once, takes the iterations from
// Tw.
template <int NS>
__device__ __forceinline__ int newton_cell(const double* u, double Tw, const MechDev& m, double tol, int maxit,
                                           double& T, double& p, double& c, double& rrho) {
  const double rho = u[0];
  rrho = rcp(rho);
  double W, h[6];
  mixture_sums<NS, 6>(u, m, W, h);
  const double c1 = 2.0 * h[1], c2 = 3.0 * h[2], c3 = 4.0 * h[3], c4 = 5.0 * h[4];
  const double ke = fma(u[1], u[1], u[2] * u[2]);
  const double K0 = fma(-fma(-0.5 * rrho, ke, u[3]), 1.0 / RU, h[5]);
  const double K1 = h[0] - W;
  const bool early = tol >= 0x1p-50 && tol <= 0x1p-28;
  double t = Tw;
  int st = 0;
  int it = 0;
  bool found = false;
  // maxit: so that the iterations would have converged too; Tw positive, below 2^100: no
  // other has a float (NaN or infinity would come out as an ordinary number)
  if (early && maxit >= 8 && (unsigned)(__double2hiint(Tw) >> 20) - 923u < 200u) {
    const float f4 = soft::cut_float(h[4]), f3 = soft::cut_float(h[3]), f2 = soft::cut_float(h[2]),
                f1 = soft::cut_float(h[1]), k1 = soft::cut_float(K1), k0 = soft::cut_float(K0);
    float x = soft::cut_float(Tw);
    const float g1 = 2.0f * f1, g2 = 3.0f * f2, g3 = 4.0f * f3, g4 = 5.0f * f4;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float F = fmaf(x, fmaf(x, fmaf(x, fmaf(x, fmaf(x, f4, f3), f2), f1), k1), k0);
      const float Fp = fmaf(x, fmaf(x, fmaf(x, fmaf(x, g4, g3), g2), g1), k1);
      x -= __fdividef(F, Fp);
    }
    if (x > 1e-3f && x < 1e6f) {
      const double y = soft::widen(x);
      const double F = fma(y, fma(y, fma(y, fma(y, fma(y, h[4], h[3]), h[2]), h[1]), K1), K0);
      const double Fp = fma(y, fma(y, fma(y, fma(y, c4, c3), c2), c1), K1);
      const double dT = -F * rcp(Fp);
      const float Fpp = fmaf(x, fmaf(x, fmaf(x, 4.0f * g4, 3.0f * g3), 2.0f * g2), g1);
      const float s = 0.5f * __fdividef(Fpp, soft::cut_float(Fp)) * soft::cut_float(dT);
      // F' within 2^+-100 (positive): its float and the quotient are sound
      found = dbits(dabs(dT)) + (18ull << 52) <= dbits(y) && fabsf(s) < 0x1p-19f &&
              (unsigned)(__double2hiint(Fp) >> 20) - 923u < 200u;
      if (found) t = y + fma(-dT, soft::widen(s), dT);
    }
  }
  for (; !found && it < maxit; ++it) {
    double F = fma(t, fma(t, fma(t, fma(t, fma(t, h[4], h[3]), h[2]), h[1]), K1), K0);
    double Fp = fma(t, fma(t, fma(t, fma(t, c4, c3), c2), c1), K1);
    double dT = -F * rcp(Fp);
    t = __dadd_rn(t, dT);
    // the early test on integers: 2^28 |dT| by its exponent field
    const bool done = early && it + 1 < maxit
                          ? dbits(dabs(dT)) + (28ull << 52) <= dbits(dabs(t)) || !finite_bits(dT)
                          : !(dabs(dT) > tol * dabs(t));
    if (done) break;
  }
  if (!found && it == maxit) st |= ST_NEWTON_FAIL;
  T = t;
  const double Cv = fma(t, fma(t, fma(t, fma(t, c4, c3), c2), c1), K1);
  const double Cp = Cv + W;
  p = RU * W * t;
  c = speed(Cp, p, rrho, Cv);
  if (!positive_bits(rho) || !positive_bits(t) || !positive_bits(p)) st |= ST_NONPOSITIVE;
  if (!finite_bits(t) || !finite_bits(p) || !finite_bits(c) || !finite_bits(u[3])) st |= ST_NONFINITE;
  return st;
}

}  // namespace janc
