// First-order point-implicit chemistry (arXiv 2504.13750, Eq. 4.12-4.13) on
// every cell, after the flux RK3 of the step (advance_source_term, Sec. 4.3).
//
// Per cell: molar concentrations X_j (the ns-th species takes what is left of
// rho), forward rates k_f = A T^b exp(-Ea/(Ru T)) (Eq. 4.8), reverse rates
// through the equilibrium constant of Eq. 4.9, rates of progress with the
// third-body factor (Eq. 4.7), and the analytic Jacobian of the carried
// sources with respect to rho Y_1..rho Y_{ns-1} at fixed T and rho (text after
// Eq. 4.13). The linear system is solved in molar unknowns
// dx_l = d(rho Y_l) / M_l, where it reads
//   (I - dt J'') dx = dt wdot,  J''_kl = dWk/dX_l - (M_l / M_ns) dWk/dX_ns,
// (row k of the mass-based system divided by M_k), with an unrolled LU
// factorisation and partial pivoting whose search and row swaps are integer
// compares and selects. Then Newton T for the new state, aux planes and the
// alpha max for the next step.
//
// The reaction loop is written once over a structure policy: DynRx reads each
// reaction's species, coefficients and third-body data from the run-time
// table, FixRx<I> returns them as compile-time constants of the shipped H2-air
// mechanism (janc_mech_fixed.cuh). From the rate constants on both run the same
// operations in the same order (they agree to rounding, each within the oracle's
// bars); with FixRx the rate constants come from fixed-point logarithms
// (rate_constants), and every index of the per-cell arrays (concentrations,
// production rates, Jacobian) is a constant, so that the arrays live in registers
// instead of local memory.
//
// This file is compiled without contraction (-fmad=false), and the multiply-adds are
// written as fma: a cell gets the same bits from every kernel below, and which of
// them a grid takes depends on its size, on its being a slab or a request, and on
// the adjoint's store. As fast as with the compiler's own contraction (reactors
// 300 x 101: 72.5 us a step with both, 2048 x 256: 873 us).
//
// Bound: 840 FP64 of 12,000 instructions a cell at 8 or 12 warps an SM, the FP64
// pipe 60 to 70 % busy: that pipe and the length of a cell's chain together.
// 4096 x 512: 5.65 ms a launch when all of it was FP64, 3.46 ms now.
#include <utility>

#include "janc_device.cuh"
#include "janc_internal.h"
#include "janc_mech_fixed.cuh"
#include "janc_mech_policy.cuh"

namespace janc {

constexpr int CHEM_THREADS = 128;

// dt k_f and dt k_b of every reaction of the compiled structure, at
// out[2 i stride] and out[(2 i + 1) stride], from their base-2 logarithms in fixed
// point, units of 2^-54. log2 k_b is log2 k_f plus integer sums of the G_k, and
// dt and the power of P_ref/(Ru T) are summands, so that a reaction takes two
// exponentials, 2 x 55 integer instructions, and no FP64 one. (As FP64
// polynomials, nine exp(G_k), their reciprocals and products it was 196 of the
// cell's 1080 FP64 instructions: 30300 cells in 88 us then, 79 us with this.) Against 300 bits
// (H2-air, 257 to 8190 K) the G_k are good to 2^-46.6 and ln k_f to 2^-48.2, where the
// coefficients' rounding to double, before their conversion, is the limit; as FP64
// polynomials they were good to 2^-45.9 and 2^-46.1. The sums may wrap on
// the way, the results are within +-512 (MechDev::rate_ok). Cells outside
// 256 K <= T < 8192 K, time steps outside 2^-70 .. 2^20 and tables that do not fit
// take the FP64 form.
template <int NS>
__device__ __forceinline__ void rate_constants(const MechDev& m, double T, double dt, double* __restrict__ out,
                                               int stride) {
  using namespace soft;
  constexpr int NR = fixed_h2air::NR;
  const Parts d(dt);
  FixedT t;
  if (fixed_T(m, T, t) && !d.neg && d.e > 953 && d.e < 1043) {
    const long long ldt = ((long long)(d.e - 1023) << 54) + (long long)(log2_frac(d.m) >> 10);
    long long G[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) G[k] = fixed_gibbs(m, k, t);
    for_reactions<true>(m, [&](auto R) {
      const int i = R.idx();
      const long long f = fixed_arrhenius(m.kq[i][0] + ldt, m.kq[i][1], m.kq[i][2], t);
      long long b = f + R.dnu() * t.lref;
#pragma unroll
      for (int r = 0; r < R.nre(); ++r) b += R.rnu(r) * G[R.rsp(r)];
#pragma unroll
      for (int r = 0; r < R.npr(); ++r) b -= R.pnu(r) * G[R.psp(r)];
      out[(2 * i) * stride] = __longlong_as_double(f);
      out[(2 * i + 1) * stride] = __longlong_as_double(b);
    });
    // in a loop: 38 copies of the code in line wait for their instructions
#pragma unroll 1
    for (int i = 0; i < NR; ++i) {
#pragma unroll
      for (int q = 2 * i; q < 2 * i + 2; ++q) out[q * stride] = exp2_fixed(__double_as_longlong(out[q * stride]));
    }
  } else {
    const double lnT = log_t(T), rT = rcp(T), lcr = log_t((RU / P_REF) * T);
#pragma unroll 1
    for (int i = 0; i < NR; ++i) {
      double f, b;
      log_rates(m, i, T, lnT, rT, lcr, f, b);
      out[(2 * i) * stride] = dt * exp_t(f);
      out[(2 * i + 1) * stride] = dt * exp_t(b);
    }
  }
}

// y + nu ab for ab = a b; with the compiled structure, where nu is mostly +-1, one
// fma and no product (with the rounded product and an addition 300 x 101 takes 76.3 us).
template <bool FIXED>
__device__ __forceinline__ double add_times(double nu, double a, double b, double ab, double y) {
  if (FIXED && nu == 1.0) return fma(a, b, y);
  if (FIXED && nu == -1.0) return fma(-a, b, y);
  return fma(nu, ab, y);
}

// One CHEM_THREADS block `blk` of cells; shared by the single-grid and the
// batched kernels. STORE (the discrete adjoint's segment recompute): also
// keep, per cell, what the chemistry VJP reuses (chem_lin_entries doubles,
// entry e of cell q at clin[e * n + q]): dt k_f and dt k_b of every reaction
// (2i, 2i+1), then at 2 nr the LU factors of A = I - dt J'' in elimination
// order (row r, column k at 2 nr + r (ns-1) + k: the multiplier of row r at
// elimination step k for r > k, U for r < k, 1/U_kk on the diagonal), the
// pivot row of every step (4 bits each, one 64-bit word) and the solution x.
template <int NS, bool FIXED, bool STORE = false>
__device__ __forceinline__ void chem_block(const StateView& S, const GridDev& g, const MechDev* __restrict__ mech,
                                           const StepCtl& ctl, const unsigned long long* __restrict__ alpha_step,
                                           unsigned long long* alpha_out, int* status, long long blk,
                                           double* __restrict__ clin = nullptr) {
  // FIXED: the thread's column of rate constants
  const int exs = blockDim.x;
  extern __shared__ double ex_cols[];
  double* const ex = ex_cols + threadIdx.x;
  constexpr int NSP = NS - 1;
  constexpr int NV = NS + 3;
  const MechDev& m = *mech;
  const long long n = g.n;
  const long long idx = blk * blockDim.x + threadIdx.x;
  const double dt = step_dt(ctl, alpha_step) * ctl.chem_frac;
  unsigned long long sx = 0, sy = 0;
  int st = 0;
  if (idx < n) {
    double u[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) u[k] = S.plane(k, n)[idx];
    const double T = S.plane(NV, n)[idx];

    // concentrations (Eq. 4.7 uses molar concentrations X_j)
    double X[NS];
    double rest = u[0];
#pragma unroll
    for (int k = 0; k < NSP; ++k) {
      X[k] = u[4 + k] * m.invM[k];
      rest -= u[4 + k];
    }
    X[NSP] = rest * m.invM[NSP];
    double Ctot = X[0];
#pragma unroll
    for (int k = 1; k < NS; ++k)  // (a sum of X: 1024 x 128 reactors 247 to 256 us; fma with a table: 937 to 963 us, 1024 x 256)
      Ctot = FIXED ? fma(k < NSP ? u[4 + k] : rest, m.invM[k], Ctot) : Ctot + X[k];

    const double lnT = FIXED ? 0.0 : log_t(T);
    const double rT = FIXED ? 0.0 : rcp(T);
    // dt k_f and dt k_b (ex, 2 i and 2 i + 1) with the compiled structure; for a
    // run-time table exp(G_k) and exp(-G_k), G_k = s_k/R - h_k/(RT) (Eq. 4.9 bracket)
    double eG[NS], reG[NS];
    if constexpr (FIXED) {
      rate_constants<NS>(m, T, dt, ex, exs);
    } else {
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        eG[k] = exp_t(gibbs(m, k, T, lnT, rT));
        reG[k] = rcp(eG[k]);
      }
    }
    const double cref = (P_REF / RU) * rT;   // P_ref / (Ru T)
    const double rcref = (RU / P_REF) * T;

    // everything from k_f on carries the factor dt
    double wd[NSP];        // dt x molar production rates of the carried species
    double J[NSP][NSP];    // dt J'' of the header comment, less the third bodies' common part
    double S3[NSP];        // that part: row k is S3[k] (1 - M_l / M_ns)
#pragma unroll
    for (int k = 0; k < NSP; ++k) {
      wd[k] = S3[k] = 0.0;
#pragma unroll
      for (int l = 0; l < NSP; ++l) J[k][l] = 0.0;
    }

    for_reactions<FIXED>(m, [&](auto R) {
      const int i = R.idx();
      const int nre = R.nre(), npr = R.npr();
      double kf, kb;
      if constexpr (FIXED) {
        kf = ex[(2 * i) * exs];
        kb = ex[(2 * i + 1) * exs];
      } else {
        kf = kb = dt * exp_t(fma(m.b[i], lnT, fma(-m.EaR[i], rT, m.lnA[i])));
        // k_b = k_f / K_eq,  K_eq = prod_j exp(G_j)^{nu_j} (P_ref/(Ru T))^{dnu}
        for (int r = 0; r < nre; ++r)
          for (int q = 0; q < R.rnu(r); ++q) kb *= eG[R.rsp(r)];
        for (int r = 0; r < npr; ++r)
          for (int q = 0; q < R.pnu(r); ++q) kb *= reG[R.psp(r)];
        const int dn = R.dnu();
        for (int q = 0; q < dn; ++q) kb *= rcref;
        for (int q = 0; q < -dn; ++q) kb *= cref;
      }
      if (STORE) {
        clin[(2LL * i) * n + idx] = kf;
        clin[(2LL * i + 1) * n + idx] = kb;
      }
      // law of mass action and its derivatives with respect to each
      // participant; a rate is its first derivative times that concentration
      double xr[MAX_SIDE], xp[MAX_SIDE], dq[2 * MAX_SIDE];
      double lead[2 * MAX_SIDE], tail[2 * MAX_SIDE];  // dq = lead tail
      int dsp[2 * MAX_SIDE];
#pragma unroll
      for (int r = 0; r < nre; ++r) xr[r] = X[R.rsp(r)];
#pragma unroll
      for (int r = 0; r < npr; ++r) xp[r] = X[R.psp(r)];
#pragma unroll
      for (int r = 0; r < nre; ++r) {
        double d = R.rnu(r) == 1 ? kf : kf * R.rnud(r);
        lead[r] = d;
        tail[r] = 1.0;
#pragma unroll
        for (int s = 0; s < nre; ++s) {
          const int pw = R.rnu(s) - (s == r ? 1 : 0);
#pragma unroll
          for (int t = 0; t < pw; ++t) {
            lead[r] = d;
            tail[r] = xr[s];
            d *= xr[s];
          }
        }
        dq[r] = d;
        dsp[r] = R.rsp(r);
      }
#pragma unroll
      for (int r = 0; r < npr; ++r) {
        double d = R.pnu(r) == 1 ? kb : kb * R.pnud(r);
        lead[nre + r] = -d;
        tail[nre + r] = 1.0;
#pragma unroll
        for (int s = 0; s < npr; ++s) {
          const int pw = R.pnu(s) - (s == r ? 1 : 0);
#pragma unroll
          for (int t = 0; t < pw; ++t) {
            lead[nre + r] = -d;
            tail[nre + r] = xp[s];
            d *= xp[s];
          }
        }
        dq[nre + r] = -d;
        dsp[nre + r] = R.psp(r);
      }
      double net, bwd = kb;
      if (R.pnu(0) == 1) {
        bwd = -dq[nre] * xp[0];
      } else {
#pragma unroll
        for (int r = 0; r < npr; ++r)
#pragma unroll
          for (int q = 0; q < R.pnu(r); ++q) bwd *= xp[r];
      }
      if (R.rnu(0) == 1) {
        net = fma(dq[0], xr[0], -bwd);
      } else {
        double fwd = kf;
#pragma unroll
        for (int r = 0; r < nre; ++r)
#pragma unroll
          for (int q = 0; q < R.rnu(r); ++q) fwd *= xr[r];
        net = __dadd_rn(fwd, -bwd);
      }
      double q = net, Mi = 1.0;
      if (R.tb()) {
        Mi = Ctot;
#pragma unroll
        for (int e = 0; e < R.neff(); ++e) Mi = fma(m.effv[i][e], X[R.effsp(e)], Mi);
        q = Mi * net;
#pragma unroll
        for (int d = 0; d < nre + npr; ++d) {
          lead[d] = dq[d];
          tail[d] = Mi;
          dq[d] *= Mi;
        }
      }
      // sources: wdot_k += nu_ki q
#pragma unroll
      for (int r = 0; r < nre; ++r) {
        const int k = R.rsp(r);
        if (k < NSP) wd[k] = add_times<FIXED>(-R.rnud(r), net, Mi, q, wd[k]);
      }
#pragma unroll
      for (int r = 0; r < npr; ++r) {
        const int k = R.psp(r);
        if (k < NSP) wd[k] = add_times<FIXED>(R.pnud(r), net, Mi, q, wd[k]);
      }
      // rows: every carried species with nonzero net coefficient. A third-body
      // coefficient of one in every column goes to S3; one of the last species
      // that differs from one changes all columns.
      bool last = false;
      if (R.tb()) {
#pragma unroll
        for (int e = 0; e < R.neff(); ++e) last = last || R.effsp(e) == NSP;
      }
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int cnt = side ? npr : nre;
#pragma unroll
        for (int r = 0; r < cnt; ++r) {
          const int k = side ? R.psp(r) : R.rsp(r);
          if (k >= NSP) continue;
          const double nu = side ? R.pnud(r) : -R.rnud(r);
#pragma unroll
          for (int d = 0; d < nre + npr; ++d) {
            const int j = dsp[d];
            if (j < NSP) {
              J[k][j] = add_times<FIXED>(nu, lead[d], tail[d], dq[d], J[k][j]);
            } else {
              const double v = nu * dq[d];
#pragma unroll
              for (int l = 0; l < NSP; ++l) J[k][l] = fma(-m.mratio[l], v, J[k][l]);
            }
          }
          if (R.tb()) {
            const double v = nu * net;
            if (last) {
#pragma unroll
              for (int l = 0; l < NSP; ++l) J[k][l] = fma(v, m.ceff[i][l], J[k][l]);
            } else {
              S3[k] = fma(nu, net, S3[k]);
#pragma unroll
              for (int e = 0; e < R.neff(); ++e) J[k][R.effsp(e)] = fma(v, m.effv[i][e], J[k][R.effsp(e)]);
            }
          }
        }
      }
    });

    // (I - dt J'') dx = dt wd
    double A[NSP][NSP], b[NSP], ip[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) {
      b[k] = wd[k];
#pragma unroll
      for (int l = 0; l < NSP; ++l) {
        A[k][l] = fma(-S3[k], m.third[l], -J[k][l]);
        if (k == l) A[k][l] += 1.0;
      }
    }
    bool singular = false;
    const long long lu0 = 2LL * m.nr;  // STORE: first LU entry
    unsigned long long pivs = 0;
#pragma unroll
    for (int c = 0; c < NSP; ++c) {
      int piv = c;
      unsigned long long best = dbits(A[c][c]) & 0x7fffffffffffffffull;
#pragma unroll
      for (int r = c + 1; r < NSP; ++r) {
        const unsigned long long v = dbits(A[r][c]) & 0x7fffffffffffffffull;
        if (v > best) { best = v; piv = r; }
      }
      // row swap c <-> piv as selects: row c takes the pivot row's values and
      // the pivot row row c's old ones (nothing moves when piv == c). Written
      // as one gather and one scatter per column so that every index stays a
      // constant and the matrix stays in registers.
      if (piv != c) {
#pragma unroll
      for (int k = c; k < NSP; ++k) {
        const double ac = A[c][k];
        double v = ac;
#pragma unroll
        for (int r = c + 1; r < NSP; ++r) v = (piv == r) ? A[r][k] : v;
#pragma unroll
        for (int r = c + 1; r < NSP; ++r) A[r][k] = (piv == r) ? ac : A[r][k];
        A[c][k] = v;
      }
      {
        const double bc = b[c];
        double v = bc;
#pragma unroll
        for (int r = c + 1; r < NSP; ++r) v = (piv == r) ? b[r] : v;
#pragma unroll
        for (int r = c + 1; r < NSP; ++r) b[r] = (piv == r) ? bc : b[r];
        b[c] = v;
      }
      }
      if (best == 0ull) singular = true;
      ip[c] = rcp(A[c][c]);
      if (STORE) pivs |= (unsigned long long)piv << (4 * c);
#pragma unroll
      for (int r = c + 1; r < NSP; ++r) {
        const double f = A[r][c] * ip[c];
        if (STORE) clin[(lu0 + r * NSP + c) * n + idx] = f;
#pragma unroll
        for (int k = c + 1; k < NSP; ++k) A[r][k] = fma(-f, A[c][k], A[r][k]);
        b[r] = fma(-f, b[c], b[r]);
      }
    }
    if (STORE) {
#pragma unroll
      for (int r = 0; r < NSP; ++r) {
        clin[(lu0 + r * NSP + r) * n + idx] = ip[r];
#pragma unroll
        for (int k = r + 1; k < NSP; ++k) clin[(lu0 + r * NSP + k) * n + idx] = A[r][k];
      }
      reinterpret_cast<unsigned long long*>(clin)[(lu0 + NSP * NSP) * n + idx] = pivs;
    }
#pragma unroll
    for (int r = NSP - 1; r >= 0; --r) {
      double s = b[r];
#pragma unroll
      for (int k = r + 1; k < NSP; ++k) s = fma(-A[r][k], b[k], s);
      b[r] = s * ip[r];
    }
    if (STORE) {
#pragma unroll
      for (int k = 0; k < NSP; ++k) clin[(lu0 + NSP * NSP + 1 + k) * n + idx] = b[k];
    }
    if (singular) {
      st |= ST_SINGULAR;
    } else {
#pragma unroll
      for (int k = 0; k < NSP; ++k) u[4 + k] = fma(m.M[k], b[k], u[4 + k]);
    }
#pragma unroll
    for (int k = 4; k < NV; ++k) S.plane(k, n)[idx] = u[k];
    double Tn, p, c, rrho;
    st |= newton_cell<NS>(u, T, m, g.newton_tol, g.newton_maxit, Tn, p, c, rrho);
    const double vx = u[1] * rrho, vy = u[2] * rrho;
    S.plane(NV, n)[idx] = Tn;
    S.plane(NV + 1, n)[idx] = vx;
    S.plane(NV + 2, n)[idx] = vy;
    S.plane(NV + 3, n)[idx] = p;
    sx = dbits(dabs(vx) + c);
    sy = dbits(dabs(vy) + c);
  }
  block_reduce_alpha_status(sx, sy, st, alpha_out, status);
}

// BLOCKS of the compiled-structure kernels: 3 blocks of 128 threads an SM (12
// warps) at 168 registers, of which 516 B spill, or no bound (226 registers, 8
// warps). A third warp on each scheduler hides more than the spills cost (two steps
// of 4096 x 512: 20.6 ms with 8, 19.4 with 12), but a full round of 12 takes 86 us
// where one of 8 takes 74, so the sum of the rounds decides. A step of reactors, us
// with 8 and with 12: 300 x 101 (6.2 warps an SM) 70.3 and 71.3, 512 x 96 (10.1) 150
// and 109, 512 x 128 (13.5) 153 and 151, 640 x 128 (16.8) 225 and 176, 2048 x 256 1030
// and 874. With the factors kept (k_chem_lin: 255 registers, 872 B spilled) the same
// rule; four steps' adjoint forward, ms with 8 and with 12: 512 x 96 2.78 and 2.54,
// 512 x 128 3.12 and 3.21, 640 x 128 3.86 and 3.81, 700 x 128 4.07 and 4.01, 1024 x 128
// 5.52 and 5.61 (the one size seen where the rule takes the slower form), 1024 x 256
// 10.39 and 10.40.
static int chem_blocks_per_sm(long long n) {
  const long long per = 32LL * sm_count(), w = (n + per - 1) / per;  // warps an SM gets
  return 86 * ((w + 11) / 12) < 74 * ((w + 7) / 8) ? 3 : 0;
}

template <int NS, bool FIXED, int BLOCKS = 0>
__global__ void __launch_bounds__(CHEM_THREADS, BLOCKS) k_chem(StateView S, GridDev g, const MechDev* __restrict__ mech,
                                                       StepCtl ctl, const unsigned long long* __restrict__ alpha_step,
                                                       unsigned long long* alpha_out, int* status) {
  chem_block<NS, FIXED>(S, g, mech, ctl, alpha_step, alpha_out, status, blockIdx.x);
}

// k_chem that also keeps the chemistry VJP's factors (chem_block, STORE).
template <int NS, bool FIXED, int BLOCKS = 0>
__global__ void __launch_bounds__(CHEM_THREADS, BLOCKS) k_chem_lin(StateView S, GridDev g, const MechDev* __restrict__ mech,
                                                           StepCtl ctl,
                                                           const unsigned long long* __restrict__ alpha_step,
                                                           unsigned long long* alpha_out, int* status,
                                                           double* __restrict__ clin) {
  chem_block<NS, FIXED, true>(S, g, mech, ctl, alpha_step, alpha_out, status, blockIdx.x, clin);
}

// Batched chemistry over the flattened (request, block) list: in place on
// each request's S[0], output alpha in slot 4. 12 warps an SM: mixes of many cells gain
// (24 steps of 369,000 cells 49.9 ms with 8, 48.9 with 12; 167,000: 23.6 and 22.8), of
// few lose a little (31,000: 5.01 and 5.04; 9,500: 6.50 and 6.58).
template <int NS, bool FIXED>
__global__ void __launch_bounds__(CHEM_THREADS, FIXED ? 3 : 0) k_chem_batch(const BatchReq* __restrict__ reqs,
                                                             const int* __restrict__ first, int nreq) {
  const int total = first[nreq];
  for (int e = blockIdx.x; e < total; e += gridDim.x) {
    const int r = batch_owner(first, nreq, e);
    const BatchReq& q = reqs[r];
    chem_block<NS, FIXED>(q.S[0], q.g, q.mech, q.ctl, q.alpha, q.alpha + 8, q.status, e - first[r]);
    __syncthreads();
  }
}

bool fixed_structure(const janc_mechanism* m) {
  using namespace fixed_h2air;
  if (!m || m->ns != NS || m->nr != NR || !m->nuf || !m->nub || !m->tb || !m->eff) return false;
  for (int i = 0; i < NR; ++i) {
    if ((m->tb[i] ? 1 : 0) != kTb[i]) return false;
    for (int j = 0; j < NS; ++j) {
      if (m->nuf[i * NS + j] != kNuf[i * NS + j] || m->nub[i * NS + j] != kNub[i * NS + j]) return false;
      if (kTb[i] && (m->eff[i * NS + j] != 1.0 ? 1 : 0) != kEffNe1[i * NS + j]) return false;
    }
  }
  return true;
}

// Shared memory of the compiled-structure kernels: k_f and k_b of every reaction.
static size_t chem_smem(int threads) { return sizeof(double) * 2 * fixed_h2air::NR * threads; }

cudaError_t launch_chem_batch(int ns, const BatchReq* reqs, const int* first, int nreq, int total, bool fixed,
                              cudaStream_t st) {
  const int sms = sm_count();
  const int grid = total < sms * 16 ? total : sms * 16;
  if (grid <= 0) return cudaSuccess;
  switch (ns) {
    case 3: k_chem_batch<3, false><<<grid, CHEM_THREADS, 0, st>>>(reqs, first, nreq); break;
    case 9:
      if (fixed) k_chem_batch<9, true><<<grid, CHEM_THREADS, chem_smem(CHEM_THREADS), st>>>(reqs, first, nreq);
      else k_chem_batch<9, false><<<grid, CHEM_THREADS, 0, st>>>(reqs, first, nreq);
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

int chem_blocks(const GridDev& g) { return (int)((g.n + CHEM_THREADS - 1) / CHEM_THREADS); }

// Threads per block: CHEM_THREADS while that gives at least 4 blocks per SM,
// else 64 or 32, so that a small grid's cells spread over all SMs (each
// cell is one long dependent FP64 chain; a launch of a few blocks per SM is
// latency-bound).
static int chem_threads(long long n) {
  const int sms = sm_count();
  for (int t = CHEM_THREADS; t > 32; t /= 2)
    if ((n + t - 1) / t >= 4LL * sms) return t;
  return 32;
}

cudaError_t launch_chem(int ns, const StateView& S, const GridDev& g, const MechDev* mech, const StepCtl& ctl,
                        const unsigned long long* alpha_step, unsigned long long* alpha_out, int* status,
                        cudaStream_t st) {
  const int thr = chem_threads(g.n);
  const unsigned blocks = (unsigned)((g.n + thr - 1) / thr);
  switch (ns) {
    case 3: k_chem<3, false><<<blocks, thr, 0, st>>>(S, g, mech, ctl, alpha_step, alpha_out, status); break;
    case 9:
      if (g.chem_fixed && chem_blocks_per_sm(g.n) == 3)
        k_chem<9, true, 3><<<blocks, thr, chem_smem(thr), st>>>(S, g, mech, ctl, alpha_step, alpha_out, status);
      else if (g.chem_fixed)
        k_chem<9, true><<<blocks, thr, chem_smem(thr), st>>>(S, g, mech, ctl, alpha_step, alpha_out, status);
      else k_chem<9, false><<<blocks, thr, 0, st>>>(S, g, mech, ctl, alpha_step, alpha_out, status);
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

size_t chem_lin_entries(int ns, int nr) { return 2 * (size_t)nr + (size_t)(ns - 1) * (ns - 1) + 1 + (ns - 1); }

cudaError_t launch_chem_lin(int ns, const StateView& S, const GridDev& g, const MechDev* mech, const StepCtl& ctl,
                            const unsigned long long* alpha_step, unsigned long long* alpha_out, int* status,
                            double* clin, cudaStream_t st) {
  const int thr = chem_threads(g.n);
  const unsigned blocks = (unsigned)((g.n + thr - 1) / thr);
  switch (ns) {
    case 3: k_chem_lin<3, false><<<blocks, thr, 0, st>>>(S, g, mech, ctl, alpha_step, alpha_out, status, clin); break;
    case 9:
      if (g.chem_fixed && chem_blocks_per_sm(g.n) == 3)
        k_chem_lin<9, true, 3><<<blocks, thr, chem_smem(thr), st>>>(S, g, mech, ctl, alpha_step, alpha_out, status, clin);
      else if (g.chem_fixed)
        k_chem_lin<9, true><<<blocks, thr, chem_smem(thr), st>>>(S, g, mech, ctl, alpha_step, alpha_out, status, clin);
      else
        k_chem_lin<9, false><<<blocks, thr, 0, st>>>(S, g, mech, ctl, alpha_step, alpha_out, status, clin);
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace janc
