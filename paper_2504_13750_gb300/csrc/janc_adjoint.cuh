// Reverse-mode pieces of the discrete adjoint (transposes of the operators
// of janc_flux.cu / janc_update.cu / janc_chem.cu), shared by the adjoint
// kernels.
#pragma once

#include "janc_device.cuh"

namespace janc {

// Mixture quantities of one cell at a given T (the converged Newton T):
// W = sum z_k, hR_k(T) = h_k/(Ru/M_k), Cv = sum z_k cv_k / Ru and dCv/dT.
template <int NS>
struct CellThermo {
  double z[NS], hR[NS], cvR[NS];
  double W, Cv, dCv;
};

template <int NS>
__device__ __forceinline__ void cell_thermo(const double* u, double T, const MechDev& m, CellThermo<NS>& c) {
  double rest = u[0];
#pragma unroll
  for (int k = 0; k < NS - 1; ++k) {
    c.z[k] = u[4 + k] * m.invM[k];
    rest -= u[4 + k];
  }
  c.z[NS - 1] = rest * m.invM[NS - 1];
  c.W = 0.0;
  c.Cv = 0.0;
  c.dCv = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* h = m.hc[k];
    c.hR[k] = fma(T, fma(T, fma(T, fma(T, fma(T, h[4], h[3]), h[2]), h[1]), h[0]), h[5]);
    // cp/R = a0 + a1 T + ... with a_m = (m+1) hc_m
    const double cp = fma(T, fma(T, fma(T, fma(T, 5.0 * h[4], 4.0 * h[3]), 3.0 * h[2]), 2.0 * h[1]), h[0]);
    c.cvR[k] = cp - 1.0;
    const double dcp = fma(T, fma(T, fma(T, 20.0 * h[4], 12.0 * h[3]), 6.0 * h[2]), 2.0 * h[1]);
    c.W += c.z[k];
    c.Cv = fma(c.z[k], c.cvR[k], c.Cv);
    c.dCv = fma(c.z[k], dcp, c.dCv);
  }
}

// dT/dU (implicit derivative of the Newton T recovery) and dp/dU for one
// cell, NV = NS + 3 entries each. With F(T; U) = H(T; z) - W T - rho e / Ru:
// dT/dU = -(dF/dU) / Cv and p = Ru W T.
template <int NS>
__device__ __forceinline__ void dT_dp_dU(const double* u, double T, const MechDev& m, const CellThermo<NS>& c,
                                         double* dT, double* dp) {
  constexpr int NV = NS + 3;
  const double rrho = rcp(u[0]);
  const double vx = u[1] * rrho, vy = u[2] * rrho;
  double dF[NV], dW[NV];
  const double fN = (c.hR[NS - 1] - T) * m.invM[NS - 1];
  dF[0] = fN - 0.5 * (vx * vx + vy * vy) * (1.0 / RU);
  dF[1] = vx * (1.0 / RU);
  dF[2] = vy * (1.0 / RU);
  dF[3] = -1.0 / RU;
  dW[0] = m.invM[NS - 1];
  dW[1] = dW[2] = dW[3] = 0.0;
#pragma unroll
  for (int k = 0; k < NS - 1; ++k) {
    dF[4 + k] = (c.hR[k] - T) * m.invM[k] - fN;
    dW[4 + k] = m.invM[k] - m.invM[NS - 1];
  }
  const double rCv = rcp(c.Cv);
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    dT[q] = -dF[q] * rCv;
    dp[q] = RU * (T * dW[q] + c.W * dT[q]);
  }
}

// W, Cv = sum z_k cv_k / Ru and dCv/dT of one cell at T, on the mixture sums
// of the forward (janc_device.cuh), and the frozen sound speed as sound_speed
// forms it.
struct CellHeat {
  double W, Cv, dCv, c;
};
template <int NS>
__device__ __forceinline__ CellHeat cell_heat(const double* u, double T, double rrho, const MechDev& m) {
  CellHeat r;
  double h[5];
  mixture_sums<NS, 5>(u, m, r.W, h);
  const double c1 = 2.0 * h[1], c2 = 3.0 * h[2], c3 = 4.0 * h[3], c4 = 5.0 * h[4];
  r.Cv = fma(T, fma(T, fma(T, fma(T, c4, c3), c2), c1), h[0] - r.W);
  r.dCv = fma(T, fma(T, fma(T, 4.0 * c4, 3.0 * c3), 2.0 * c2), c1);
  r.c = speed(r.Cv + r.W, RU * r.W * T, rrho, r.Cv);
  return r;
}

__device__ __forceinline__ double enthalpy_R(const MechDev& m, int k, double T) {
  const double* h = m.hc[k];
  return fma(T, fma(T, fma(T, fma(T, fma(T, h[4], h[3]), h[2]), h[1]), h[0]), h[5]);
}

// a += sW dW/dU - sF dF/dU: the chain through T(U) and p = Ru W T (dT_dp_dU)
// with the two scalars formed first, sF = (Ru W a_p + a_T) / Cv and sW = Ru T a_p
// for cotangents a_T and a_p. 9 FP64 instructions a species; with the species'
// own cv, dT/dU and dp/dU it took 24.
template <int NS>
__device__ __forceinline__ void add_thermo_grad(double T, double vx, double vy, const MechDev& m, double sF, double sW,
                                                double* a) {
  const double q = sF * (1.0 / RU);
  const double fN = (enthalpy_R(m, NS - 1, T) - T) * m.invM[NS - 1];
  a[0] = fma(-sF, fN, fma(0.5 * q, fma(vx, vx, vy * vy), fma(sW, m.invM[NS - 1], a[0])));
  a[1] = fma(-q, vx, a[1]);
  a[2] = fma(-q, vy, a[2]);
  a[3] += q;
#pragma unroll
  for (int k = 0; k < NS - 1; ++k)
    a[4 + k] = fma(-sF, fma(enthalpy_R(m, k, T) - T, m.invM[k], -fN), fma(sW, m.Wd[k], a[4 + k]));
}

}  // namespace janc
