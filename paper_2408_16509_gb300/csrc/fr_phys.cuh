// Pointwise compressible Euler / Navier-Stokes physics on the device.
//
// Conserved variables u = (rho, rho u, rho v, rho w, E): the field index
// alpha of Eq. (gov) of the paper (Section 2).  The paper names the
// compressible Euler and Navier-Stokes solvers without printing their
// formulas; these are the standard nondimensional forms:
//   p = (gamma-1)(E - rho|v|^2/2)
//   inviscid flux F_j = (rho v_j, rho v v_j + p e_j, (E+p) v_j)
//   viscous flux (subtracted) (0, tau_.j, v.tau_.j + kappa de/dx_j),
//   tau = mu(grad v + grad v^T - 2/3 div v I), e = E/rho - |v|^2/2,
//   kappa = mu gamma / Pr
//   Rusanov common flux (Eq. comm_flux):
//   (F(u-)+F(u+)).n/2 - lambda (u+ - u-)/2,
//   lambda = max(|v-.n| + c-, |v+.n| + c+).
#pragma once
#include <cuda_runtime.h>

namespace frgb {

// beta, tau: LDG bias and penalty of the viscous coupling (0, 0: BR1)
template <typename T>
struct Phys {
  T gamma, gm1, mu, kappa;
  T beta = T(0), tau = T(0);
};

template <typename T>
__device__ __forceinline__ T fr_sqrt(T x);
template <>
__device__ __forceinline__ double fr_sqrt<double>(double x) { return sqrt(x); }
template <>
__device__ __forceinline__ float fr_sqrt<float>(float x) { return sqrtf(x); }

// Rusanov flux along n.  Both sides' inviscid fluxes are added before the
// halving (one flux per side: 7 FP64 instructions a pair more).  Products are
// of a momentum and a velocity: the momenta's squares leave the type's range at
// states of 1e19 or 1e-19 in FP32, and were slower (interface kernel, FP64-pipe
// bound, 24^3 p = 4: 447 us against 430).
template <typename T>
__device__ __forceinline__ void rusanov(const T ul[5], const T ur[5],
                                        const T n[3], const Phys<T>& ph,
                                        T F[5]) {
  const T il = T(1) / ul[0], ir = T(1) / ur[0];
  const T wl[3] = {ul[1] * il, ul[2] * il, ul[3] * il};
  const T wr[3] = {ur[1] * ir, ur[2] * ir, ur[3] * ir};
  const T vl = wl[0] * n[0] + wl[1] * n[1] + wl[2] * n[2];
  const T vr = wr[0] * n[0] + wr[1] * n[1] + wr[2] * n[2];
  const T pl = ph.gm1 * (ul[4] - T(0.5) * (ul[1] * wl[0] + ul[2] * wl[1] + ul[3] * wl[2]));
  const T pr = ph.gm1 * (ur[4] - T(0.5) * (ur[1] * wr[0] + ur[2] * wr[1] + ur[3] * wr[2]));
  const T a = fabs(vl) + fr_sqrt<T>(ph.gamma * pl * il);
  const T b = fabs(vr) + fr_sqrt<T>(ph.gamma * pr * ir);
  const T hl = T(0.5) * (a > b ? a : b), ps = pl + pr;
  F[0] = T(0.5) * (ul[0] * vl + ur[0] * vr) + hl * (ul[0] - ur[0]);
#pragma unroll
  for (int k = 0; k < 3; ++k)
    F[1 + k] = T(0.5) * (ul[1 + k] * vl + ur[1 + k] * vr + ps * n[k]) + hl * (ul[1 + k] - ur[1 + k]);
  F[4] = T(0.5) * ((ul[4] + pl) * vl + (ur[4] + pr) * vr) + hl * (ul[4] - ur[4]);
}

// inviscid flux F[j][k] in direction j of variable k
template <typename T>
__device__ __forceinline__ void euler_flux(const T u[5], const Phys<T>& ph,
                                           T F[3][5]) {
  T ri = T(1) / u[0];
  T v[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
  T p = ph.gm1 * (u[4] - T(0.5) * (u[1] * v[0] + u[2] * v[1] + u[3] * v[2]));
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    F[j][0] = u[1 + j];
    F[j][1] = u[1] * v[j];
    F[j][2] = u[2] * v[j];
    F[j][3] = u[3] * v[j];
    F[j][1 + j] += p;
    F[j][4] = (u[4] + p) * v[j];
  }
}

// viscous flux from u and its physical gradient g[j][k] = du_k/dx_j;
// accumulates  F[j][k] += sgn * Fv[j][k]
template <typename T>
__device__ __forceinline__ void viscous_flux_acc(const T u[5], const T g[3][5],
                                                 const Phys<T>& ph, T sgn,
                                                 T F[3][5]) {
  T ri = T(1) / u[0];
  T v[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
  T er = u[4] * ri;
  T gv[3][3], ge[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
#pragma unroll
    for (int i = 0; i < 3; ++i) gv[j][i] = (g[j][1 + i] - v[i] * g[j][0]) * ri;
    ge[j] = (g[j][4] - er * g[j][0]) * ri -
            (v[0] * gv[j][0] + v[1] * gv[j][1] + v[2] * gv[j][2]);
  }
  T div = gv[0][0] + gv[1][1] + gv[2][2];
  T mu = ph.mu;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    T tau[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) tau[i] = mu * (gv[j][i] + gv[i][j]);
    tau[j] -= T(2.0 / 3.0) * mu * div;
    F[j][1] += sgn * tau[0];
    F[j][2] += sgn * tau[1];
    F[j][3] += sgn * tau[2];
    F[j][4] += sgn * (v[0] * tau[0] + v[1] * tau[1] + v[2] * tau[2] +
                      ph.kappa * ge[j]);
  }
}

// Viscous flux at a point: stress (xx, yy, zz, xy, xz, yz) in tq[0..5] and
// energy flux v.tau + kappa grad e in tq[6..8].  The velocity gradient is
// left undivided by rho (d[j][i] = g_j(m_i) - v_i g_j(rho)): one factor
// mu / rho on the six stresses.
template <typename T>
__device__ __forceinline__ void viscous_point(const T u[5], const T (&g)[3][5],
                                              const Phys<T>& ph, T tq[9]) {
  const T ri = T(1) / u[0];
  const T v[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
  const T er = u[4] * ri, mr = ph.mu * ri, kr = ph.kappa * ri;
  T d[3][3];
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int i = 0; i < 3; ++i) d[j][i] = g[j][1 + i] - v[i] * g[j][0];
  const T m2 = T(2) * mr;
  const T dv = (T(2.0 / 3.0) * mr) * (d[0][0] + d[1][1] + d[2][2]);
#pragma unroll
  for (int j = 0; j < 3; ++j) tq[j] = m2 * d[j][j] - dv;
  tq[3] = mr * (d[0][1] + d[1][0]);
  tq[4] = mr * (d[0][2] + d[2][0]);
  tq[5] = mr * (d[1][2] + d[2][1]);
  const T t[3][3] = {{tq[0], tq[3], tq[4]}, {tq[3], tq[1], tq[5]}, {tq[4], tq[5], tq[2]}};
#pragma unroll
  for (int j = 0; j < 3; ++j)
    tq[6 + j] = kr * ((g[j][4] - er * g[j][0]) -
                      (v[0] * d[j][0] + v[1] * d[j][1] + v[2] * d[j][2])) +
                (v[0] * t[j][0] + v[1] * t[j][1] + v[2] * t[j][2]);
}

// Total flux at a point, the 12 distinct values of F[j][k]: mass (the
// momentum) f[0..2], momentum f[3..8] (xx, yy, zz, xy, xz, yz), energy
// f[9..11]; tq: viscous_point's values (NS).
template <typename T, bool NS>
__device__ __forceinline__ void flux_point(const T u[5], const T tq[9], const Phys<T>& ph,
                                           T f[12]) {
  const T ri = T(1) / u[0];
  const T v[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
  const T p = ph.gm1 * (u[4] - T(0.5) * (u[1] * v[0] + u[2] * v[1] + u[3] * v[2]));
  const T h = u[4] + p;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    f[j] = u[1 + j];
    f[3 + j] = u[1 + j] * v[j] + (NS ? p - tq[j] : p);
    f[9 + j] = NS ? h * v[j] - tq[6 + j] : h * v[j];
  }
  f[6] = NS ? u[1] * v[1] - tq[3] : u[1] * v[1];
  f[7] = NS ? u[1] * v[2] - tq[4] : u[1] * v[2];
  f[8] = NS ? u[2] * v[2] - tq[5] : u[2] * v[2];
}

// Normal viscous flux n.Fv accumulated into f[k] with weight wt.
// FP64: formed from the gradients along n (gn_k = n.grad u_k) and their
// transpose: with x_i = gn_i - v_i gn_0 + sum_j n_j (g_i(m_j) - v_j g_i(rho))
// - 2/3 n_i (div m - v.grad rho), (tau n)_i = (mu / rho) x_i, energy
// (mu / rho) v.x + (kappa / rho) rho n.grad e.  The velocity gradient is
// never built: 59 instructions a side against 75 (interface kernel, FP64-pipe
// bound, 24^3 p = 4: 485 -> 430 us with the Rusanov form above).
// FP32: (tau n)_i = mu (sum_j (dv_i/dx_j + dv_j/dx_i) n_j - 2/3 div v n_i) from
// the velocity gradient; the form above made the prism and tetrahedron
// gradient kernels 1 % slower.
template <typename T>
__device__ __forceinline__ void viscous_normal_acc(const T u[5],
                                                   const T g[3][5],
                                                   const T n[3],
                                                   const Phys<T>& ph, T wt,
                                                   T f[5]) {
  if constexpr (sizeof(T) == 8) {
    const T ri = T(1) / u[0];
    const T v[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
    const T er = u[4] * ri, mr = wt * (ph.mu * ri), kr = wt * (ph.kappa * ri);
    T gn[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) gn[k] = n[0] * g[0][k] + n[1] * g[1][k] + n[2] * g[2][k];
    const T vn = v[0] * n[0] + v[1] * n[1] + v[2] * n[2];
    const T div = (g[0][1] + g[1][2] + g[2][3]) -
                  (v[0] * g[0][0] + v[1] * g[1][0] + v[2] * g[2][0]);
    const T d23 = T(2.0 / 3.0) * div;
    T vx = T(0), vt = T(0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const T t = gn[1 + i] - v[i] * gn[0];
      const T s = n[0] * g[i][1] + n[1] * g[i][2] + n[2] * g[i][3] - vn * g[i][0];
      const T x = t + (s - d23 * n[i]);
      f[1 + i] += mr * x;
      vx += v[i] * x;
      vt += v[i] * t;
    }
    f[4] += mr * vx + kr * ((gn[4] - er * gn[0]) - vt);
  } else {
    const T ri = T(1) / u[0];
    const T v[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
    const T er = u[4] * ri;
    T gv[3][3];  // gv[j][i] = d v_i / d x_j
    T gen = T(0);  // n . grad e
#pragma unroll
    for (int j = 0; j < 3; ++j) {
#pragma unroll
      for (int i = 0; i < 3; ++i) gv[j][i] = (g[j][1 + i] - v[i] * g[j][0]) * ri;
      const T ge = (g[j][4] - er * g[j][0]) * ri -
                   (v[0] * gv[j][0] + v[1] * gv[j][1] + v[2] * gv[j][2]);
      gen += n[j] * ge;
    }
    const T div23 = T(2.0 / 3.0) * (gv[0][0] + gv[1][1] + gv[2][2]);
    T tn[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T s = -div23 * n[i];
#pragma unroll
      for (int j = 0; j < 3; ++j) s += (gv[j][i] + gv[i][j]) * n[j];
      tn[i] = ph.mu * s;
    }
    f[1] += wt * tn[0];
    f[2] += wt * tn[1];
    f[3] += wt * tn[2];
    f[4] += wt * (v[0] * tn[0] + v[1] * tn[1] + v[2] * tn[2] + ph.kappa * gen);
  }
}

}  // namespace frgb
