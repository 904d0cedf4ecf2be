// Pointwise fluxes of the ALE compressible Navier-Stokes discretization
// (Sec. 6: Eqs. ns1-ns5 and the ALE transformation of Eqs. ns-cons-ref,
// transform2-nogcl specialised to the rigid-body map of Eq. defmap, where
// G = Q, g = 1 and the transformed flux is the physical flux minus U (x) v_G
// evaluated with physical gradients and normals).
//
// Numerical fluxes (the paper defers them to its references; readings):
//  - inviscid: Roe's approximate Riemann solver applied to the ALE normal flux
//    F(U).n - (v_G.n) U, Harten entropy fix with delta = 0.1 c;
//  - viscous: the compact discontinuous Galerkin (CDG) scheme of Sec. 6: liftings of
//    the face jumps U_hat - U- into the element (the lifted gradients are formed by the
//    kernels from the reference lifting tables); on an interior face the element with
//    the smaller index supplies the viscous flux F_vis(U_S, grad U_S + r_f) . n with the
//    lifting of that face only; boundary faces add the penalty c11 (U_hat - U-);
//  - wall: no-slip, adiabatic; wall state with the mesh velocity; exact
//    no-penetration inviscid flux;  far field: free-stream state.
//
// Every function is templated on the scalar type so that the same code gives
// values (double) and exact directional derivatives (Dual).
#pragma once

#include "pp_internal.h"

namespace pp {

// An FP64 division costs about ten instructions of a pipe that issues one per 19 clocks and SM, so
// every function takes one reciprocal per state (ir = 1 / rho) and multiplies.
template <class T>
__device__ __forceinline__ T pressure(const T U[4], const T& ir, double gam) {
  return (gam - 1.0) * (U[3] - 0.5 * (U[1] * U[1] + U[2] * U[2]) * ir);
}

// F[a][d]: inviscid flux of variable a in direction d
template <class T>
__device__ __forceinline__ void inviscid_flux(const T U[4], const T& ir, double gam, T F[4][2]) {
  T u = U[1] * ir, v = U[2] * ir;
  T p = pressure(U, ir, gam);
  F[0][0] = U[1];
  F[1][0] = U[1] * u + p;
  F[2][0] = U[2] * u;
  F[3][0] = (U[3] + p) * u;
  F[0][1] = U[2];
  F[1][1] = U[1] * v;
  F[2][1] = U[2] * v + p;
  F[3][1] = (U[3] + p) * v;
}

// viscous flux from the state and its physical gradient dU[a][d];
// q = -(mu/Pr) grad(E + p/rho - |u|^2/2) = -(mu gamma/Pr) grad(e)
template <class T>
__device__ __forceinline__ void viscous_flux(const T U[4], const T& ir, const T dU[4][2], const Phys& ph,
                                             bool adiabatic, T F[4][2]) {
  T u = U[1] * ir, v = U[2] * ir, E = U[3] * ir;
  T du[2], dv[2], dE[2];
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    du[d] = (dU[1][d] - u * dU[0][d]) * ir;
    dv[d] = (dU[2][d] - v * dU[0][d]) * ir;
    dE[d] = (dU[3][d] - E * dU[0][d]) * ir;
  }
  T div = du[0] + dv[1];
  T txx = ph.mu * (2.0 * du[0] - (2.0 / 3.0) * div);
  T tyy = ph.mu * (2.0 * dv[1] - (2.0 / 3.0) * div);
  T txy = ph.mu * (du[1] + dv[0]);
  double kq = adiabatic ? 0.0 : ph.mu * ph.gam / ph.Pr;
  T qx = -kq * (dE[0] - u * du[0] - v * dv[0]);
  T qy = -kq * (dE[1] - u * du[1] - v * dv[1]);
  F[0][0] = T(0.0);
  F[1][0] = txx;
  F[2][0] = txy;
  F[3][0] = u * txx + v * txy - qx;
  F[0][1] = T(0.0);
  F[1][1] = txy;
  F[2][1] = tyy;
  F[3][1] = u * txy + v * tyy - qy;
}

// total ALE volume flux F_inv - U (x) v_G - F_vis
template <class T>
__device__ __forceinline__ void volume_flux(const T U[4], const T dU[4][2], const T vG[2], const Phys& ph,
                                            T F[4][2]) {
  T Fi[4][2], Fv[4][2];
  const T ir = 1.0 / U[0];
  inviscid_flux(U, ir, ph.gam, Fi);
  viscous_flux(U, ir, dU, ph, false, Fv);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int d = 0; d < 2; ++d) F[a][d] = Fi[a][d] - U[a] * vG[d] - Fv[a][d];
}

template <class T>
__device__ __forceinline__ void normal_flux(const T U[4], const T& ir, const T& p, const T n[2], const T& vn, T out[4]) {
  const T un = (U[1] * n[0] + U[2] * n[1]) * ir;
  const T w = un - vn;
  out[0] = U[0] * w;
  out[1] = U[1] * w + p * n[0];
  out[2] = U[2] * w + p * n[1];
  out[3] = U[3] * w + p * un;
}

// Harten's fix with delta = 0.1 c; h = 1 / (2 delta)
template <class T>
__device__ __forceinline__ T entropy_fix(const T& l, const T& delta, const T& h) {
  T al = absT(l);
  if (val(al) < val(delta)) return (l * l + delta * delta) * h;
  return al;
}

// Roe flux of the ALE normal flux; |A - vn I| (UR - UL) written with the two
// wave-strength scalars of the acoustic pair.  iL, iR: 1 / rho of the two states.
template <class T>
__device__ __forceinline__ void roe_flux(const T UL[4], const T& iL, const T UR[4], const T& iR, const T n[2],
                                         const T& vn, double gam, T out[4]) {
  const T pL = pressure(UL, iL, gam), pR = pressure(UR, iR, gam);
  const T sL = sqrtT(UL[0]), sR = sqrtT(UR[0]);
  const T isum = 1.0 / (sL + sR);
  // sqrt(rho) / rho weights: s u = (s / rho) (rho u)
  const T wL = sL * iL * isum, wR = sR * iR * isum;
  const T ut = wL * UL[1] + wR * UR[1];
  const T vt = wL * UL[2] + wR * UR[2];
  const T Ht = wL * (UL[3] + pL) + wR * (UR[3] + pR);
  const T hq2 = 0.5 * (ut * ut + vt * vt);
  const T c2 = (gam - 1.0) * (Ht - hq2);
  const T c = sqrtT(c2);
  const T ic = 1.0 / c;
  const T un = ut * n[0] + vt * n[1];
  const T lu = un - vn;
  const T delta = 0.1 * c, h = 5.0 * ic;
  const T l1 = entropy_fix(lu + c, delta, h);
  const T l2 = entropy_fix(lu - c, delta, h);
  const T l3 = entropy_fix(lu, delta, h);
  T D[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) D[a] = UR[a] - UL[a];
  const T dp = (gam - 1.0) * (hq2 * D[0] - ut * D[1] - vt * D[2] + D[3]);
  const T dUn = D[1] * n[0] + D[2] * n[1] - un * D[0];
  const T s1 = 0.5 * (l1 + l2) - l3;
  const T s2 = 0.5 * (l1 - l2) * ic;
  const T G1 = s1 * dp * (ic * ic) + s2 * dUn;
  const T G2 = s2 * dp + s1 * dUn;
  T FL[4], FR[4];
  normal_flux(UL, iL, pL, n, vn, FL);
  normal_flux(UR, iR, pR, n, vn, FR);
  out[0] = 0.5 * (FL[0] + FR[0] - (l3 * D[0] + G1));
  out[1] = 0.5 * (FL[1] + FR[1] - (l3 * D[1] + G1 * ut + G2 * n[0]));
  out[2] = 0.5 * (FL[2] + FR[2] - (l3 * D[2] + G1 * vt + G2 * n[1]));
  out[3] = 0.5 * (FL[3] + FR[3] - (l3 * D[3] + G1 * Ht + G2 * un));
}

// No-slip wall state: the interior density and internal energy, moving with the wall.
template <class T>
__device__ __forceinline__ void wall_state(const T Um[4], const T vG[2], T Ub[4]) {
  const T r = Um[0];
  Ub[0] = r;
  Ub[1] = r * vG[0];
  Ub[2] = r * vG[1];
  // rho (E - |u|^2 / 2) + rho |v_G|^2 / 2
  Ub[3] = Um[3] - 0.5 * (Um[1] * Um[1] + Um[2] * Um[2]) / r + 0.5 * (r * (vG[0] * vG[0] + vG[1] * vG[1]));
}

// Face value U_hat of U at one face point: the neighbour trace (tag 0), the wall state
// (tag 1) or the free stream (tag 2).
template <class T>
__device__ __forceinline__ void face_value(int tag, const T Um[4], const T Up[4], const T vG[2], const Phys& ph,
                                           T Uh[4]) {
  if (tag == 1) {
    wall_state(Um, vG, Uh);
  } else if (tag == 0) {
#pragma unroll
    for (int a = 0; a < 4; ++a) Uh[a] = Up[a];
  } else {
#pragma unroll
    for (int a = 0; a < 4; ++a) Uh[a] = T(ph.Uinf[a]);
  }
}

// CDG numerical flux H (outward from the "-" element, per unit length) at one face point:
//   H = H_inv(U-, U+) - F_vis(U_S, Q_S) . n - c11 (U_hat - U-)
// with H_inv Roe's flux (interior, far field) or the exact wall flux, and Q_S the lifted
// gradient of the side S that supplies the viscous flux (side = 1: this element, whose
// viscous state is U- or, on the wall, the wall state; side = 0: the neighbour, U+).
// The wall flux is adiabatic (zero heat flux); c11 is zero on interior faces.
template <class T>
__device__ __forceinline__ void face_flux(int tag, int side, const T Um[4], const T Up[4], const T QS[4][2],
                                          const T n[2], const T vG[2], double c11, const Phys& ph, T H[4]) {
  T vn = vG[0] * n[0] + vG[1] * n[1];
  T Hi[4], Uh[4], Fv[4][2];
  face_value(tag, Um, Up, vG, ph, Uh);
  const T iL = 1.0 / Um[0];
  if (tag == 1) {
    // the wall state shares the density
    normal_flux(Uh, iL, pressure(Uh, iL, ph.gam), n, vn, Hi);
    viscous_flux(Uh, iL, QS, ph, true, Fv);
  } else {
    const T iR = 1.0 / Uh[0];
    roe_flux(Um, iL, Uh, iR, n, vn, ph.gam, Hi);
    T Us[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) Us[a] = pick(side, Um[a], Up[a]);
    viscous_flux(Us, pick(side, iL, iR), QS, ph, false, Fv);
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) H[a] = Hi[a] - (Fv[a][0] * n[0] + Fv[a][1] * n[1] + c11 * (Uh[a] - Um[a]));
}

}  // namespace pp
