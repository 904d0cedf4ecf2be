// Element-local quadrature kernels of the ALE DG discretization (Sec. 6):
//  - k_residual     r(u, mu, t) of M du/dt = r (Eq. semidisc) with the CDG viscous
//                   terms (liftings of the face jumps); with a frame that carries
//                   derivatives it gives kappa . dr/ds for the motion seeds s (theta,
//                   theta', h') of dr/dmu in Eq. funcl-grad-nosens-dirk;
//  - k_jacobian     element block Jacobian dr/du (diagonal + 3 face-neighbour
//                   blocks): exact flux derivatives at every quadrature point by
//                   forward-mode dual numbers, contracted with the basis;
//  - k_qoi*         instantaneous power and x-force on the wall (Eq. qoi) and
//                   their exact derivatives with respect to u and the frame.
//
// Layouts: u[e][a][i] (nb = 4 Np doubles per element, contiguous); Jacobian
// blocks [e][slot][col][row] (column-major nb x nb).
#include "fixed.cuh"
#include "flux.cuh"
#include "prof.h"
#include "../../include/pp_prof.h"

namespace pp {

namespace {

constexpr int RES_WARPS = 4;
constexpr int NSV = 12;  // seeds of a point: U (4) + grad U (8)

template <class T>
__device__ __forceinline__ void frame_P(const FrameT<T>& fr, const double* BinvT, T P[4]) {
  // grad_x phi = Q grad_X phi = Q B^{-T} grad_xi phi  =>  P = Q B^{-T}
  P[0] = fr.Q[0] * BinvT[0] + fr.Q[1] * BinvT[2];
  P[1] = fr.Q[0] * BinvT[1] + fr.Q[1] * BinvT[3];
  P[2] = fr.Q[2] * BinvT[0] + fr.Q[3] * BinvT[2];
  P[3] = fr.Q[2] * BinvT[1] + fr.Q[3] * BinvT[3];
}

template <class T>
__device__ __forceinline__ void mesh_velocity(const FrameT<T>& fr, const Phys& ph, double X, double Y, T vG[2]) {
  double dx = X - ph.x0[0], dy = Y - ph.x0[1];
  vG[0] = fr.Qd[0] * dx + fr.Qd[1] * dy;
  vG[1] = fr.Qd[2] * dx + fr.Qd[3] * dy + fr.hd;
}

__device__ __forceinline__ void ref_to_X(const DevMesh& m, int e, double xi, double eta, double& X, double& Y) {
  const double* B = m.B + 4 * e;
  X = m.X0[2 * e] + B[0] * xi + B[1] * eta;
  Y = m.X0[2 * e + 1] + B[2] * xi + B[3] * eta;
}

// state and physical gradient at a point from nodal values ue[a*Np + i]
template <class T>
__device__ __forceinline__ void interp(const double* ue, int Np, const double* phi, const double* dphi,
                                       const T P[4], T U[4], T dU[4][2]) {
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    double s = 0.0, s0 = 0.0, s1 = 0.0;
    for (int i = 0; i < Np; ++i) {
      double c = ue[a * Np + i];
      s += phi[i] * c;
      s0 += dphi[2 * i] * c;
      s1 += dphi[2 * i + 1] * c;
    }
    U[a] = T(s);
    dU[a][0] = P[0] * s0 + P[1] * s1;
    dU[a][1] = P[2] * s0 + P[3] * s1;
  }
}

template <class T>
__device__ __forceinline__ void rotate_normal(const FrameT<T>& fr, const double* N, T n[2]) {
  n[0] = fr.Q[0] * N[0] + fr.Q[1] * N[1];
  n[1] = fr.Q[2] * N[0] + fr.Q[3] * N[1];
}

// value of U at a point from nodal values ue[a*Np + i]
__device__ __forceinline__ void interp_val(const double* ue, int Np, const double* phi, double U[4]) {
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    double s = 0.0;
    for (int i = 0; i < Np; ++i) s += phi[i] * ue[a * Np + i];
    U[a] = s;
  }
}

// CDG lifting of face jumps into a gradient at one point: dU[a][d] += s n[d] sum_p A[p*step] J[p][a]
// (A: one row of a reference lifting table, read forwards (step 1) or in reverse (step -1)
// for a neighbour's face whose points are matched in reverse order).
template <class T, class TJ>
__device__ __forceinline__ void lift_add(T dU[4][2], const T n[2], double s, const double* A, int step,
                                         const TJ* J, int nqf) {
  TJ l[4] = {TJ(0.0), TJ(0.0), TJ(0.0), TJ(0.0)};
  for (int p = 0; p < nqf; ++p) {
    const double c = A[p * step];
#pragma unroll
    for (int a = 0; a < 4; ++a) l[a] += c * J[p * 4 + a];
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    dU[a][0] += s * (l[a] * n[0]);
    dU[a][1] += s * (l[a] * n[1]);
  }
}

// lifting-table row of face f at point q of this element, for the side that lifts it
// (side 1: the element's own face f; side 0: the neighbour's face g, points reversed)
__device__ __forceinline__ const double* lift_row(const DevTables& tb, int side, int f, int g, int q, int& step) {
  const int nqf = tb.nqf;
  if (side) {
    step = 1;
    return tb.lift_f + (f * nqf + q) * nqf;
  }
  step = -1;
  return tb.lift_f + (g * nqf + nqf - 1 - q) * nqf + nqf - 1;
}

// s + sum_t a_t b_t over N fixed-point terms, `stride` words apart in a (at most 60 per exact sum)
template <int N>
__device__ __forceinline__ double fix_dot(const Fix* a, const Fix* b, int ea, int eb, double s, int stride = 1) {
  constexpr int parts = (N + 59) / 60, M = (N + parts - 1) / parts;
  static_assert((parts == 1 || parts * M == N) && M <= kFixTerms, "equal parts, one exact sum each");
#pragma unroll
  for (int p = 0; p < parts; ++p) {
    FixDot acc;
    acc.clear();
#pragma unroll(M <= 30 ? M : M % 10 == 0 ? 10 : 12)
    for (int t = 0; t < M; ++t) acc.add(a[(p * M + t) * stride], b[p * M + t]);
    s = acc.result(ea + eb, ea == 0x7ff || eb == 0x7ff, s);
  }
  return s;
}

// s - sum_t a_t b_t
template <int N>
__device__ __forceinline__ double fix_dot_minus(const Fix* a, const Fix* b, int ea, int eb, double s) {
  return -fix_dot<N>(a, b, ea, eb, -s);
}

// A group's entry as a double, its exponent collected in ge; turned into fixed point after a barrier.
__device__ __forceinline__ void fix_put(double* w, int* ge, double v) {
  *w = v;
  atomicMax(ge, fix_exponent(v));
}
__device__ __forceinline__ void fix_enc(double* w, int ge) { *reinterpret_cast<Fix*>(w) = fix_encode(*w, ge); }

// ------------------------------------------------------------------------ residual
// T = double: the residual r, or (NEWTON) the residual of a stage's Newton iteration,
//   u = base + a_ii k (written, with its neighbours' values formed on the way in),
//   R = M k - dt r(u), and per element |R|^2 and |M u|^2,
// in place of seven launches (two vector combinations, the residual, two mass products, two norms).
// T = DualV<3>: kappa . dr/ds for three motion seeds s carried by the
// frame, summed per element (dr itself is not written).
//
// A CTA takes groups of elements and deals (element, point) and (element, row) tasks to its threads, so
// that the warps are full (a warp per element leaves 44% of the lanes of the 36 + 18 points at p = 4
// idle, and a warp instruction costs the FP64 pipe the same whatever its active lanes).  Bound:
// FP64 issue.  The interpolations and the projection on the test functions run on the integer pipe
// (fixed.cuh); what remains in FP64 are the fluxes.
// Phases: A jumps U_hat - U- at the face points; B volume points with the element's own liftings;
// C face points with the lifted gradient of the side that supplies the viscous flux; D projection.
template <int PD, class T, bool NEWTON>
struct Res {
  static constexpr int NP = (PD + 1) * (PD + 2) / 2, NB = 4 * NP, NF = PD + 2, NV = NF * NF, F3 = 3 * NF;
  static constexpr bool VAL = sizeof(T) == sizeof(double);
  static constexpr int NC = VAL ? 1 : 3;                      // components projected
  static constexpr int W = sizeof(T) / sizeof(double);
  static constexpr int THREADS = VAL ? 256 : 128;
  static constexpr int EB = THREADS / NV;                     // most elements of a group
  static constexpr int LP = NP | 1;                           // odd table rows: no bank conflicts
  // shared memory in 8-byte words: tables, then per element
  static constexpr int pv = 0, dv = pv + NV * LP, pf = dv + 2 * NV * LP, df = pf + F3 * LP,
                       ms = df + 2 * F3 * LP, elems = ms + (NEWTON ? NP * LP : 0);
  static constexpr int su = 0, Uf = su + 4 * NB, Js = Uf + F3 * 8, G = Js + F3 * 4 * W, H = G + NC * 4 * 2 * NV,
                       ks = H + NC * 4 * F3, per = (ks + (NEWTON ? NB : 0)) | 1;
  static constexpr int words = elems + EB * per;
};
template <int PD, class T, bool NEWTON>
struct ResExp {
  using L = Res<PD, T, NEWTON>;
  int tab[5];
  int u[L::EB][4][4], k[L::EB][4], G[L::EB][L::NC][4], H[L::EB][L::NC][4];
};

__device__ __forceinline__ double part(double a, int) { return a; }
__device__ __forceinline__ double part(const DualV<3>& a, int k) { return a.d[k]; }

template <int PD, class T, bool NEWTON>
__global__ void __launch_bounds__(Res<PD, T, NEWTON>::THREADS, 2)
    k_residual(DevMesh m, DevTables tb, Phys ph, FrameT<T> fr, const double* __restrict__ u,
               const double* __restrict__ kappa, double* __restrict__ out, StageNewton nw, int eb) {
  using L = Res<PD, T, NEWTON>;
  constexpr int NP = L::NP, NB = L::NB, NF = L::NF, NV = L::NV, F3 = L::F3, NT = L::THREADS, NC = L::NC, LP = L::LP;
  extern __shared__ double smem[];
  __shared__ ResExp<PD, T, NEWTON> ex;
  const int tid = threadIdx.x;
  // tables, one exponent each
  if (tid < 5) ex.tab[tid] = 0;
  __syncthreads();
  auto each_table = [&](auto&& f) {
    for (int i = tid; i < NV * NP; i += NT) {
      const int q = i / NP, j = i - q * NP;
      f(smem + L::pv + q * LP + j, &ex.tab[0], tb.phi_v + i);
      f(smem + L::dv + q * LP + j, &ex.tab[1], tb.dphi_v + 2 * i);
      f(smem + L::dv + (NV + q) * LP + j, &ex.tab[1], tb.dphi_v + 2 * i + 1);
    }
    for (int i = tid; i < F3 * NP; i += NT) {
      const int q = i / NP, j = i - q * NP;
      f(smem + L::pf + q * LP + j, &ex.tab[2], tb.phi_f + i);
      f(smem + L::df + q * LP + j, &ex.tab[3], tb.dphi_f + 2 * i);
      f(smem + L::df + (F3 + q) * LP + j, &ex.tab[3], tb.dphi_f + 2 * i + 1);
    }
    if constexpr (NEWTON)
      for (int i = tid; i < NP * NP; i += NT) f(smem + L::ms + i / NP * LP + i % NP, &ex.tab[4], tb.Mref + i);
  };
  each_table([](double* w, int* ge, const double* v) { fix_put(w, ge, *v); });
  __syncthreads();
  each_table([](double* w, int* ge, const double*) { fix_enc(w, *ge); });
  auto fix = [&](int off) { return reinterpret_cast<const Fix*>(smem + off); };

  for (int e0 = blockIdx.x * eb; e0 < m.ne; e0 += gridDim.x * eb) {
    const int n = min(eb, m.ne - e0);
    __syncthreads();
    for (int k = tid; k < (int)((sizeof(ex.u) + sizeof(ex.k) + sizeof(ex.G) + sizeof(ex.H)) / 4); k += NT)
      (&ex.u[0][0][0])[k] = 0;
    __syncthreads();
    for (int idx = tid; idx < n * 4 * NB; idx += NT) {
      const int el = idx / (4 * NB), r = idx - el * 4 * NB, slot = r / NB, k = r - slot * NB;
      int src = e0 + el;
      if (slot > 0) {
        const int nn = m.nbr[3 * src + slot - 1];
        src = nn >= 0 ? nn : src;
      }
      const size_t at = (size_t)src * NB + k;
      double v;
      if constexpr (NEWTON) {
        const double kv = nw.k[at];
        v = nw.base[at] + nw.aii * kv;
        if (slot == 0) {
          nw.us[at] = v;
          fix_put(smem + L::elems + el * L::per + L::ks + k, &ex.k[el][k / NP], kv);
        }
      } else {
        v = u[at];
      }
      fix_put(smem + L::elems + el * L::per + L::su + r, &ex.u[el][slot][k / NP], v);
    }
    __syncthreads();
    for (int idx = tid; idx < n * 4 * NB; idx += NT) {
      const int el = idx / (4 * NB), r = idx - el * 4 * NB, slot = r / NB, k = r - slot * NB;
      fix_enc(smem + L::elems + el * L::per + L::su + r, ex.u[el][slot][k / NP]);
      if (NEWTON && slot == 0) fix_enc(smem + L::elems + el * L::per + L::ks + k, ex.k[el][k / NP]);
    }
    __syncthreads();
    // phase A: both traces and the jumps
    for (int task = tid; task < n * F3; task += NT) {
      const int el = task / F3, fq = task - el * F3, f = fq / NF, q = fq - f * NF, e = e0 + el;
      double* const S = smem + L::elems + el * L::per;
      const Fix* su = reinterpret_cast<const Fix*>(S + L::su);
      const int tag = m.tag[3 * e + f];
      const int fn = tag == 0 ? m.nbrface[3 * e + f] * NF + NF - 1 - q : fq;
      const int sn = tag == 0 ? 1 + f : 0;
      T Um[4], Up[4], vG[2], Uh[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const double um = fix_dot<NP>(fix(L::pf) + fq * LP, su + a * NP, ex.tab[2], ex.u[el][0][a], 0.0);
        const double up = tag == 0 ? fix_dot<NP>(fix(L::pf) + fn * LP, su + sn * NB + a * NP, ex.tab[2], ex.u[el][sn][a], 0.0) : um;
        S[L::Uf + fq * 8 + a] = um;
        S[L::Uf + fq * 8 + 4 + a] = up;
        Um[a] = T(um);
        Up[a] = T(up);
      }
      double X, Y;
      ref_to_X(m, e, tb.xi_f[2 * fq], tb.xi_f[2 * fq + 1], X, Y);
      mesh_velocity(fr, ph, X, Y, vG);
      face_value(tag, Um, Up, vG, ph, Uh);
      T* Js = reinterpret_cast<T*>(S + L::Js);
#pragma unroll
      for (int a = 0; a < 4; ++a) Js[fq * 4 + a] = Uh[a] - Um[a];
    }
    __syncthreads();
    // phases B and C: volume points, then face points from the next full warp on
    const int nvol = (n * NV + 31) / 32 * 32;
    for (int task = tid; task < nvol + n * F3; task += NT) {
      if (task < nvol) {
        if (task >= n * NV) continue;
        const int el = task / NV, q = task - el * NV, e = e0 + el;
        double* const S = smem + L::elems + el * L::per;
        const Fix* su = reinterpret_cast<const Fix*>(S + L::su);
        const T* Js = reinterpret_cast<const T*>(S + L::Js);
        T P[4], U[4], dU[4][2], vG[2], F[4][2];
        frame_P(fr, m.BinvT + 4 * e, P);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const int eu = ex.u[el][0][a];
          U[a] = T(fix_dot<NP>(fix(L::pv) + q * LP, su + a * NP, ex.tab[0], eu, 0.0));
          const double s0 = fix_dot<NP>(fix(L::dv) + q * LP, su + a * NP, ex.tab[1], eu, 0.0);
          const double s1 = fix_dot<NP>(fix(L::dv) + (NV + q) * LP, su + a * NP, ex.tab[1], eu, 0.0);
          dU[a][0] = P[0] * s0 + P[1] * s1;
          dU[a][1] = P[2] * s0 + P[3] * s1;
        }
        for (int f = 0; f < 3; ++f)
          if (m.side[3 * e + f]) {
            T nf[2];
            rotate_normal(fr, m.N + 6 * e + 2 * f, nf);
            lift_add(dU, nf, m.s_own[3 * e + f], tb.lift_v + (f * NV + q) * NF, 1, Js + f * NF * 4, NF);
          }
        double X, Y;
        ref_to_X(m, e, tb.xi_v[2 * q], tb.xi_v[2 * q + 1], X, Y);
        mesh_velocity(fr, ph, X, Y, vG);
        volume_flux(U, dU, vG, ph, F);
        const double wq = tb.w_v[q] * m.detB[e];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const T g0 = wq * (P[0] * F[a][0] + P[2] * F[a][1]), g1 = wq * (P[1] * F[a][0] + P[3] * F[a][1]);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            double* G = S + L::G + (c * 4 + a) * 2 * NV;
            fix_put(G + q, &ex.G[el][c][a], part(g0, c));
            fix_put(G + NV + q, &ex.G[el][c][a], part(g1, c));
          }
        }
      } else {
        const int t2 = task - nvol, el = t2 / F3, fq = t2 - el * F3, f = fq / NF, q = fq - f * NF, e = e0 + el;
        double* const S = smem + L::elems + el * L::per;
        const Fix* su = reinterpret_cast<const Fix*>(S + L::su);
        const T* Js = reinterpret_cast<const T*>(S + L::Js);
        const int tag = m.tag[3 * e + f], side = m.side[3 * e + f];
        // the gradient of the side that supplies the viscous flux
        const int g = tag == 0 ? m.nbrface[3 * e + f] : 0;
        const int slot = side ? 0 : 1 + f, fs = side ? fq : g * NF + NF - 1 - q, es = side ? e : m.nbr[3 * e + f];
        T P[4], Um[4], Up[4], QS[4][2], n2[2], vG[2], H[4];
        frame_P(fr, m.BinvT + 4 * es, P);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const Fix* ua = su + slot * NB + a * NP;
          const double s0 = fix_dot<NP>(fix(L::df) + fs * LP, ua, ex.tab[3], ex.u[el][slot][a], 0.0);
          const double s1 = fix_dot<NP>(fix(L::df) + (F3 + fs) * LP, ua, ex.tab[3], ex.u[el][slot][a], 0.0);
          QS[a][0] = P[0] * s0 + P[1] * s1;
          QS[a][1] = P[2] * s0 + P[3] * s1;
          Um[a] = T(S[L::Uf + fq * 8 + a]);
          Up[a] = T(S[L::Uf + fq * 8 + 4 + a]);
        }
        rotate_normal(fr, m.N + 6 * e + 2 * f, n2);
        int step;
        const double* A = lift_row(tb, side, f, g, q, step);
        lift_add(QS, n2, side ? m.s_own[3 * e + f] : m.s_nbr[3 * e + f], A, step, Js + f * NF * 4, NF);
        double X, Y;
        ref_to_X(m, e, tb.xi_f[2 * fq], tb.xi_f[2 * fq + 1], X, Y);
        mesh_velocity(fr, ph, X, Y, vG);
        face_flux(tag, side, Um, Up, QS, n2, vG, m.c11[3 * e + f], ph, H);
        const double wl = tb.w_f[q] * m.L[3 * e + f];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int c = 0; c < NC; ++c)
            fix_put(S + L::H + (c * 4 + a) * F3 + fq, &ex.H[el][c][a], wl * part(H[a], c));
      }
    }
    __syncthreads();
    for (int idx = tid; idx < n * NC * 4 * (2 * NV + F3); idx += NT) {
      const int el = idx / (NC * 4 * (2 * NV + F3)), r = idx - el * NC * 4 * (2 * NV + F3), ca = r / (2 * NV + F3),
                t = r - ca * (2 * NV + F3);
      double* const S = smem + L::elems + el * L::per;
      if (t < 2 * NV) fix_enc(S + L::G + ca * 2 * NV + t, (&ex.G[el][0][0])[ca]);
      else fix_enc(S + L::H + ca * F3 + t - 2 * NV, (&ex.H[el][0][0])[ca]);
    }
    __syncthreads();
    // phase D
    for (int idx = tid; idx < n * NB; idx += NT) {
      const int el = idx / NB, o = idx - el * NB, a = o / NP, i = o - a * NP;
      double* const S = smem + L::elems + el * L::per;
      double acc[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const Fix* G = reinterpret_cast<const Fix*>(S + L::G) + (c * 4 + a) * 2 * NV;
        const Fix* H = reinterpret_cast<const Fix*>(S + L::H) + (c * 4 + a) * F3;
        acc[c] = -fix_dot<F3>(fix(L::pf) + i, H, ex.tab[2], ex.H[el][c][a], 0.0, LP);
        acc[c] = fix_dot<2 * NV>(fix(L::dv) + i, G, ex.tab[1], ex.G[el][c][a], acc[c], LP);
      }
      if constexpr (NEWTON) {
        const double detB = m.detB[e0 + el];
        const Fix* mi = fix(L::ms) + i * LP;
        const double mk = detB * fix_dot<NP>(mi, reinterpret_cast<const Fix*>(S + L::ks) + a * NP, ex.tab[4], ex.k[el][a], 0.0);
        const double mu = detB * fix_dot<NP>(mi, reinterpret_cast<const Fix*>(S + L::su) + a * NP, ex.tab[4], ex.u[el][0][a], 0.0);
        const double R = mk - nw.dt * acc[0];
        out[(size_t)(e0 + el) * NB + o] = R;
        // in place of the neighbours' states
        S[L::su + NB + o] = R;
        S[L::su + 2 * NB + o] = mu;
      } else if constexpr (L::VAL) {
        out[(size_t)(e0 + el) * NB + o] = acc[0];
      } else {
        // kappa times the rows, in place of the states
        const double kp = kappa[(size_t)(e0 + el) * NB + o];
#pragma unroll
        for (int c = 0; c < NC; ++c) S[L::su + c * NB + o] = kp * acc[c];
      }
    }
    if constexpr (!L::VAL || NEWTON) {
      __syncthreads();
      // per-element sums: eight lanes per (element, seed or norm), then a butterfly over them
      constexpr int NS = NEWTON ? 2 : 3;
      double* const sums = NEWTON ? nw.sums : out;
      const int l = tid & 7;
      for (int g8 = tid >> 3; g8 < (n * NS + 3) / 4 * 4; g8 += NT / 8) {
        const int el = g8 / NS, c = g8 - el * NS;
        double s = 0.0;
        if (el < n) {
          const double* v = smem + L::elems + el * L::per + L::su + (NEWTON ? c + 1 : c) * NB;
          for (int o = l; o < NB; o += 8) s += NEWTON ? v[o] * v[o] : v[o];
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (l == 0 && el < n) sums[(size_t)(e0 + el) * NS + c] = s;
      }
    }
  }
}

// ------------------------------------------------------------------------ Jacobian
// Element block Jacobian dr/du, one CTA per element, templated on the degree.
//
// Phase 0: U and grad U at every point (both traces on faces), the face jumps U_hat - U- and, at
// wall points, d U_wall / d U-; then the CDG liftings: the volume gradients and the flux side's
// face gradients become the lifted ones.
// Phase 1: exact derivatives of the quadrature-point fluxes with respect to (U, lifted grad U),
// weighted and projected on the reference gradients of test and trial functions: state seeds by
// forward-mode derivatives (one thread carries 4 seeds of a volume point, 2 of a face point, so
// that the value part with its divisions and roots is shared), gradient seeds in closed form (the
// viscous flux is linear in the gradient at fixed U).
// Phase 2, per row variable a and column variables b: W = C T over the trial functions,
// J_ab = D W, plus the liftings' chain: Lam = d r_a / d jump_b at the face points (through the
// volume and the face gradients), contracted with d jump / d u (-phi of this element, +phi of the
// neighbour; at wall points d U_wall / d U- couples b to every variable, added per row a).  The
// mass equation has no viscous flux and the momentum equations none from grad(rho E): those pairs
// have no gradient part and no liftings.
//
// Bound: FP64 issue (one warp instruction per 19 clocks and SM).  The contractions (D W, Lam, the
// lifting chain: 260,000 multiply-adds per element at p = 3) run on the integer pipe (fixed.cuh):
// factors are written as doubles with the largest exponent of their group, encoded in place, and a
// sum costs two FP64 instructions instead of one per term.
template <int PD>
struct Jac {
  static constexpr int NP = (PD + 1) * (PD + 2) / 2, NB = 4 * NP, NF = PD + 2, NV = NF * NF, F3 = 3 * NF;
  static constexpr int T = 256;              // threads
  static constexpr int NBV = PD <= 3 ? 2 : 1;  // column variables at a time
  // term strides, odd: lanes over rows read different banks
  static constexpr int LV = 2 * NV + 1, LF = F3 | 1, LY = NV | 1;
  // shared memory in 8-byte words
  static constexpr int su = 0;
  static constexpr int SV = su + 4 * NB;               // [q][12]: U, lifted grad U at the volume points
  static constexpr int SF = SV + NV * 12;              // [side][f][q][12]: both traces (flux side: lifted gradient)
  static constexpr int Cv = SF + 2 * F3 * 12;          // [q][a][k][12]
  static constexpr int Cf = Cv + NV * 8 * 12;          // [f][q][a][16]: U- | U+ | gradient of the flux side
  static constexpr int Js = Cf + F3 * 4 * 16;          // [f][q][4] jumps
  static constexpr int Gb = Js + F3 * 4;               // [f][q][4][4] d U_wall / d U- at wall points
  static constexpr int dV = Gb + F3 * 16;              // [i][LV] test gradients (k, q)
  static constexpr int pF = dV + NP * LV;              // [i][LF] own face basis values
  static constexpr int pN = pF + NP * LF;              // [j][LF] the neighbours' at the matched points
  static constexpr int lv = pN + NP * LF;              // [f][p][LY] lifting at the volume points
  static constexpr int Wv = lv + F3 * LY;              // [b][j][LV]
  static constexpr int Wf = Wv + NBV * NP * LV;        // [b][j][LF]
  static constexpr int Wn = Wf + NBV * NP * LF;        // [b][j][LF]
  static constexpr int cv = Wn + NBV * NP * LF;        // [b][f][q][2] gradient coefficients along n_f
  static constexpr int cf = cv + NBV * 3 * NV * 2;     // [b][f][q]
  static constexpr int Y = cf + NBV * F3;              // [b][f][i][LY] cv contracted with the test gradients
  static constexpr int Lam = Y + NBV * 3 * NP * LY;    // [b][i][LF] d r_(a,i) / d jump_(f,b)(p)
  static constexpr int LamW = Lam + NBV * NP * LF;     // [f][b][i][NF] of the wall faces, doubles
  static constexpr int words = LamW + 3 * 4 * NP * NF;
};
// exponents of the groups
template <int PD>
struct JacExp {
  using L = Jac<PD>;
  int dV[L::NP], pF[L::NP], pN[L::NP], lv[L::F3];
  int Wv[L::NBV][L::NP], Wf[L::NBV][L::NP], Wn[L::NBV][3][L::NP], Y[L::NBV][3][L::NP], Lam[L::NBV][L::NP];
};

// per-face data of one element
struct JacFaces {
  double P[4], nf[3][2], Pn[3][4], s_lift[3];
  double nuo[3][2], nus[3][2];  // P^-1 n of this element and of the flux side
  int side[3], tag[3], g[3];
};

// viscous flux derivative for the unit gradient of variable b along d: F[a - 1][dir], a = 1 .. 3
__device__ __forceinline__ void viscous_seed(int b, int d, double u, double v, double E, double ir, double mu, double kq,
                                             double F[3][2]) {
  const double du = b == 0 ? -u * ir : b == 1 ? ir : 0.0;
  const double dv = b == 0 ? -v * ir : b == 2 ? ir : 0.0;
  const double dE = b == 0 ? -E * ir : b == 3 ? ir : 0.0;
  const double q = kq * (dE - u * du - v * dv);
  // along x: div = du, shear = dv; along y: div = dv, shear = du
  const double nrm = mu * (d == 0 ? du : dv), sh = mu * (d == 0 ? dv : du);
  const double txx = d == 0 ? (4.0 / 3.0) * nrm : (-2.0 / 3.0) * nrm;
  const double tyy = d == 0 ? (-2.0 / 3.0) * nrm : (4.0 / 3.0) * nrm;
  F[0][0] = txx;
  F[0][1] = sh;
  F[1][0] = sh;
  F[1][1] = tyy;
  F[2][0] = u * txx + v * sh + (d == 0 ? q : 0.0);
  F[2][1] = u * sh + v * tyy + (d == 1 ? q : 0.0);
}

template <int PD>
__global__ void __launch_bounds__(Jac<PD>::T, 2)
    k_jacobian(DevMesh m, DevTables tb, Phys ph, FrameT<double> fr, const double* __restrict__ u,
               double* __restrict__ J) {
  using L = Jac<PD>;
  constexpr int NP = L::NP, NB = L::NB, NF = L::NF, NV = L::NV, F3 = L::F3, T = L::T, NBV = L::NBV;
  constexpr int LV = L::LV, LF = L::LF, LY = L::LY;
  extern __shared__ double smem[];
  __shared__ JacExp<PD> ex;
  const int e = blockIdx.x, tid = threadIdx.x;
  double* const su = smem + L::su;
  double* const SV = smem + L::SV;
  double* const SF = smem + L::SF;
  double* const Cv = smem + L::Cv;
  double* const Cf = smem + L::Cf;
  double* const Js = smem + L::Js;
  double* const Gb = smem + L::Gb;
  double* const cvv = smem + L::cv;
  double* const cff = smem + L::cf;
  double* const LamW = smem + L::LamW;
  auto put = [](double* w, int* ge, double v) { fix_put(w, ge, v); };
  auto enc = [](double* w, int ge) { fix_enc(w, ge); };
  auto fix = [&](int off) { return reinterpret_cast<const Fix*>(smem + off); };

  for (int k = tid; k < (int)(sizeof(ex) / sizeof(int)); k += T) reinterpret_cast<int*>(&ex)[k] = 0;
  for (int idx = tid; idx < 4 * NB; idx += T) {
    int slot = idx / NB, k = idx - slot * NB;
    int src = e;
    if (slot > 0) {
      int nn = m.nbr[3 * e + slot - 1];
      src = nn >= 0 ? nn : e;
    }
    su[idx] = u[(size_t)src * NB + k];
  }
  __shared__ JacFaces fc;
  double(&P)[4] = fc.P;
  double(&nf)[3][2] = fc.nf;
  double(&Pn)[3][4] = fc.Pn;
  double(&nuo)[3][2] = fc.nuo;
  double(&nus)[3][2] = fc.nus;
  double(&s_lift)[3] = fc.s_lift;
  int(&sidef)[3] = fc.side;
  int(&tagf)[3] = fc.tag;
  int(&gf)[3] = fc.g;
  if (tid < 3) {
    const int f = tid;
    double Po[4], Pf[4], n[2];
    frame_P(fr, m.BinvT + 4 * e, Po);
    rotate_normal(fr, m.N + 6 * e + 2 * f, n);
    const int side = m.side[3 * e + f], tag = m.tag[3 * e + f];
    frame_P(fr, m.BinvT + 4 * (tag == 0 ? m.nbr[3 * e + f] : e), Pf);
    sidef[f] = side;
    tagf[f] = tag;
    gf[f] = tag == 0 ? m.nbrface[3 * e + f] : 0;
    s_lift[f] = side ? m.s_own[3 * e + f] : m.s_nbr[3 * e + f];
    const double io = 1.0 / (Po[0] * Po[3] - Po[1] * Po[2]), in = 1.0 / (Pf[0] * Pf[3] - Pf[1] * Pf[2]);
    nuo[f][0] = (Po[3] * n[0] - Po[1] * n[1]) * io;
    nuo[f][1] = (Po[0] * n[1] - Po[2] * n[0]) * io;
    nus[f][0] = side ? nuo[f][0] : (Pf[3] * n[0] - Pf[1] * n[1]) * in;
    nus[f][1] = side ? nuo[f][1] : (Pf[0] * n[1] - Pf[2] * n[0]) * in;
    for (int k = 0; k < 2; ++k) nf[f][k] = n[k];
    for (int k = 0; k < 4; ++k) {
      Pn[f][k] = Pf[k];
      if (f == 0) P[k] = Po[k];
    }
  }
  const double detB = m.detB[e];
  __syncthreads();
  const bool has_wall = tagf[0] == 1 || tagf[1] == 1 || tagf[2] == 1;

  // reference tables, as doubles
  for (int idx = tid; idx < NP * 2 * NV; idx += T) {
    const int i = idx / (2 * NV), r = idx - i * 2 * NV, k = r / NV, q = r - k * NV;
    put(smem + L::dV + i * LV + r, &ex.dV[i], tb.dphi_v[2 * (q * NP + i) + k]);
  }
  for (int idx = tid; idx < NP * F3; idx += T) {
    const int i = idx / F3, fq = idx - i * F3, f = fq / NF, q = fq - f * NF;
    put(smem + L::pF + i * LF + fq, &ex.pF[i], tb.phi_f[fq * NP + i]);
    put(smem + L::pN + i * LF + fq, &ex.pN[i], tagf[f] == 0 ? tb.phi_f[(gf[f] * NF + NF - 1 - q) * NP + i] : 0.0);
  }
  for (int idx = tid; idx < F3 * NV; idx += T) {
    const int fp = idx / NV, q = idx - fp * NV, f = fp / NF, p = fp - f * NF;
    put(smem + L::lv + fp * LY + q, &ex.lv[fp], tb.lift_v[(f * NV + q) * NF + p]);
  }
  // phase 0a: U and grad U at every quadrature point, once (both traces on faces)
  for (int task = tid; task < NV + 2 * F3; task += T) {
    double U0[4], dU0[4][2];
    double* dst;
    if (task < NV) {
      interp(su, NP, tb.phi_v + task * NP, tb.dphi_v + 2 * task * NP, P, U0, dU0);
      dst = SV + task * 12;
    } else {
      const int t2 = task - NV, side = t2 / F3, fq = t2 - side * F3, f = fq / NF, q = fq - f * NF;
      dst = SF + (side * F3 + fq) * 12;
      if (side == 0 || tagf[f] != 0) {
        interp(su, NP, tb.phi_f + fq * NP, tb.dphi_f + 2 * fq * NP, P, U0, dU0);
      } else {
        const int g = gf[f], qq = NF - 1 - q;
        interp(su + (1 + f) * NB, NP, tb.phi_f + (g * NF + qq) * NP, tb.dphi_f + 2 * (g * NF + qq) * NP, Pn[f], U0,
               dU0);
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      dst[a] = U0[a];
      dst[4 + 2 * a] = dU0[a][0];
      dst[5 + 2 * a] = dU0[a][1];
    }
  }
  __syncthreads();
  for (int idx = tid; idx < NP * 2 * NV; idx += T) enc(smem + L::dV + idx / (2 * NV) * LV + idx % (2 * NV), ex.dV[idx / (2 * NV)]);
  for (int idx = tid; idx < NP * F3; idx += T) {
    enc(smem + L::pF + idx / F3 * LF + idx % F3, ex.pF[idx / F3]);
    enc(smem + L::pN + idx / F3 * LF + idx % F3, ex.pN[idx / F3]);
  }
  for (int idx = tid; idx < F3 * NV; idx += T) enc(smem + L::lv + idx / NV * LY + idx % NV, ex.lv[idx / NV]);
  // phase 0b: jumps, and d U_wall / d U- at wall points
  for (int fq = tid; fq < F3; fq += T) {
    const int f = fq / NF;
    const double* Sm = SF + fq * 12;
    const double* Sp = SF + (F3 + fq) * 12;
    double X, Yc, vG[2], Uh[4];
    ref_to_X(m, e, tb.xi_f[2 * fq], tb.xi_f[2 * fq + 1], X, Yc);
    mesh_velocity(fr, ph, X, Yc, vG);
    face_value(tagf[f], Sm, Sp, vG, ph, Uh);
#pragma unroll
    for (int a = 0; a < 4; ++a) Js[fq * 4 + a] = Uh[a] - Sm[a];
    if (tagf[f] == 1) {
      DualV<4> Ud[4], vd[2] = {DualV<4>(vG[0]), DualV<4>(vG[1])}, Ub[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        Ud[a] = DualV<4>(Sm[a]);
        Ud[a].d[a] = 1.0;
      }
      wall_state(Ud, vd, Ub);
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int c = 0; c < 4; ++c) Gb[(fq * 4 + b) * 4 + c] = Ub[b].d[c];
    }
  }
  __syncthreads();
  // phase 0c: lifted gradients (volume points; the flux side's trace on each face)
  for (int task = tid; task < NV + F3; task += T) {
    double dU[4][2];
    double* dst;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      dU[a][0] = 0.0;
      dU[a][1] = 0.0;
    }
    if (task < NV) {
      dst = SV + task * 12;
      for (int f = 0; f < 3; ++f)
        if (sidef[f]) lift_add(dU, nf[f], s_lift[f], tb.lift_v + (f * NV + task) * NF, 1, Js + f * NF * 4, NF);
    } else {
      const int fq = task - NV, f = fq / NF, q = fq - f * NF;
      dst = SF + ((sidef[f] ? 0 : F3) + fq) * 12;
      int step;
      const double* A = lift_row(tb, sidef[f], f, gf[f], q, step);
      lift_add(dU, nf[f], s_lift[f], A, step, Js + f * NF * 4, NF);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      dst[4 + 2 * a] += dU[a][0];
      dst[5 + 2 * a] += dU[a][1];
    }
  }
  __syncthreads();

  // phase 1.  The heavy tasks go to warps of their own: the volume points to warp 0, the face points'
  // state seeds (two per thread) to warps 1 .. 3 and the gradient seeds to the others; which warps
  // these are turns with the block, so that co-resident CTAs load the SM's four partitions evenly.
  const double kq0 = ph.mu * ph.gam / ph.Pr;
  const int warp = ((tid >> 5) + blockIdx.x) & 7, lane = tid & 31;
  if (warp == 0) {
    for (int q = lane; q < NV; q += 32) {
      const double* Sq = SV + q * 12;
      DualV<4> U[4], dU[4][2], vG[2], F[4][2];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        U[a] = DualV<4>(Sq[a]);
        U[a].d[a] = 1.0;
        dU[a][0] = DualV<4>(Sq[4 + 2 * a]);
        dU[a][1] = DualV<4>(Sq[5 + 2 * a]);
      }
      double X, Yc, vg[2];
      ref_to_X(m, e, tb.xi_v[2 * q], tb.xi_v[2 * q + 1], X, Yc);
      mesh_velocity(fr, ph, X, Yc, vg);
      vG[0] = DualV<4>(vg[0]);
      vG[1] = DualV<4>(vg[1]);
      volume_flux(U, dU, vG, ph, F);
      const double wq = tb.w_v[q] * detB;
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          Cv[((q * 4 + a) * 2 + 0) * 12 + s] = wq * (P[0] * F[a][0].d[s] + P[2] * F[a][1].d[s]);
          Cv[((q * 4 + a) * 2 + 1) * 12 + s] = wq * (P[1] * F[a][0].d[s] + P[3] * F[a][1].d[s]);
        }
    }
  } else if (warp <= 3) {
    // state seeds of the face points: U- (s0 = 0, 2) and U+ (s0 = 4, 6)
    for (int task = (warp - 1) * 32 + lane; task < F3 * 4; task += 96) {
      const int fq = task >> 2, s0 = (task & 3) * 2, f = fq / NF;
      const int tag = tagf[f], side = sidef[f];
      const bool plus = s0 >= 4;
      double* out = Cf + fq * 64 + s0;
      if (tag != 0 && plus) {
#pragma unroll
        for (int a = 0; a < 4; ++a) out[a * 16] = out[a * 16 + 1] = 0.0;
        continue;
      }
      const double* Sm = SF + fq * 12;
      const double* Sp = SF + (F3 + fq) * 12;
      const double* SS = side ? Sm : Sp;
      DualV<2> Um[4], Up[4], QS[4][2], n[2], vG[2], H[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        Um[a] = DualV<2>(Sm[a]);
        Up[a] = DualV<2>(Sp[a]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          Um[a].d[k] = s0 + k == a ? 1.0 : 0.0;
          Up[a].d[k] = s0 + k == 4 + a ? 1.0 : 0.0;
        }
        QS[a][0] = DualV<2>(SS[4 + 2 * a]);
        QS[a][1] = DualV<2>(SS[5 + 2 * a]);
      }
      double X, Yc, vg[2];
      ref_to_X(m, e, tb.xi_f[2 * fq], tb.xi_f[2 * fq + 1], X, Yc);
      mesh_velocity(fr, ph, X, Yc, vg);
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        n[d] = DualV<2>(nf[f][d]);
        vG[d] = DualV<2>(vg[d]);
      }
      face_flux(tag, side, Um, Up, QS, n, vG, m.c11[3 * e + f], ph, H);
      const double wl = tb.w_f[fq - f * NF] * m.L[3 * e + f];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        out[a * 16] = wl * H[a].d[0];
        out[a * 16 + 1] = wl * H[a].d[1];
      }
    }
  } else {
    // gradient seeds, as coefficients of the reference gradient of the trial function
    for (int task = (warp - 4) * 32 + lane; task < 4 * (NV + F3); task += 128) {
      const bool vol = task < 4 * NV;
      const int q = vol ? task >> 2 : (task - 4 * NV) >> 2, b = task & 3;
      if (vol) {
        const double* Sq = SV + q * 12;
        const double ir = 1.0 / Sq[0], wq = tb.w_v[q] * detB;
        double F[2][3][2];
#pragma unroll
        for (int d = 0; d < 2; ++d) viscous_seed(b, d, Sq[1] * ir, Sq[2] * ir, Sq[3] * ir, ir, ph.mu, kq0, F[d]);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int l = 0; l < 2; ++l) {
              double s = 0.0;
              if (a > 0)
                s = P[k] * (F[0][a - 1][0] * P[l] + F[1][a - 1][0] * P[2 + l]) +
                    P[2 + k] * (F[0][a - 1][1] * P[l] + F[1][a - 1][1] * P[2 + l]);
              Cv[((q * 4 + a) * 2 + k) * 12 + 4 + 2 * b + l] = -wq * s;
            }
      } else {
        const int f = q / NF, tag = tagf[f];
        const double* SS = SF + ((sidef[f] ? 0 : F3) + q) * 12;
        const double* PS = sidef[f] ? P : Pn[f];
        double U[4] = {SS[0], SS[1], SS[2], SS[3]};
        if (tag == 1) {
          // wall: the viscous flux is evaluated at the wall state, adiabatic
          double X, Yc, vG[2], Ub[4];
          ref_to_X(m, e, tb.xi_f[2 * q], tb.xi_f[2 * q + 1], X, Yc);
          mesh_velocity(fr, ph, X, Yc, vG);
          wall_state(U, vG, Ub);
#pragma unroll
          for (int a = 0; a < 4; ++a) U[a] = Ub[a];
        }
        const double ir = 1.0 / U[0], wl = tb.w_f[q - f * NF] * m.L[3 * e + f];
        double F[2][3][2];
#pragma unroll
        for (int d = 0; d < 2; ++d)
          viscous_seed(b, d, U[1] * ir, U[2] * ir, U[3] * ir, ir, ph.mu, tag == 1 ? 0.0 : kq0, F[d]);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int l = 0; l < 2; ++l) {
            double s = 0.0;
            if (a > 0)
              s = (F[0][a - 1][0] * nf[f][0] + F[0][a - 1][1] * nf[f][1]) * PS[l] +
                  (F[1][a - 1][0] * nf[f][0] + F[1][a - 1][1] * nf[f][1]) * PS[2 + l];
            Cf[q * 64 + a * 16 + 8 + 2 * b + l] = -wl * s;
          }
      }
    }
  }

  // phase 2: per row variable a and NBV column variables
  const size_t nb2 = (size_t)NB * NB;
  double* Jd = J + (size_t)e * 4 * nb2;
  auto has_grad = [](int a, int b) { return a > 0 && (a == 3 || b < 3); };
  for (int ab = 0; ab < 16; ab += NBV) {
    const int a = ab >> 2, b0 = ab & 3;
    __syncthreads();
    for (int k = tid; k < (int)(sizeof(ex.Wv) + sizeof(ex.Wf) + sizeof(ex.Wn) + sizeof(ex.Y) + sizeof(ex.Lam)) / 4; k += T)
      (&ex.Wv[0][0])[k] = 0;
    __syncthreads();
    // W = C T, and the gradient coefficients along each face normal for the liftings
    for (int idx = tid; idx < NBV * NP * 2 * NV; idx += T) {
      const int jj = idx % NP, r = idx / NP, kq = r % (2 * NV), bb = r / (2 * NV), k = kq / NV, q = kq - k * NV, b = b0 + bb;
      const double* C = Cv + ((q * 4 + a) * 2 + k) * 12;
      double w = C[b] * tb.phi_v[q * NP + jj];
      if (has_grad(a, b)) {
        const double* dj = tb.dphi_v + 2 * (q * NP + jj);
        w += C[4 + 2 * b] * dj[0] + C[5 + 2 * b] * dj[1];
      }
      put(smem + L::Wv + (bb * NP + jj) * LV + kq, &ex.Wv[bb][jj], w);
    }
    for (int idx = tid; idx < NBV * NP * F3; idx += T) {
      const int jj = idx % NP, r = idx / NP, fq = r % F3, bb = r / F3, f = fq / NF, q = fq - f * NF, b = b0 + bb;
      const double* C = Cf + fq * 64 + a * 16;
      const int fn = gf[f] * NF + NF - 1 - q;
      double wo = C[b] * tb.phi_f[fq * NP + jj];
      double wn = tagf[f] == 0 ? C[4 + b] * tb.phi_f[fn * NP + jj] : 0.0;
      if (has_grad(a, b)) {
        const double* dj = tb.dphi_f + 2 * ((sidef[f] ? fq : fn) * NP + jj);
        const double g = C[8 + 2 * b] * dj[0] + C[9 + 2 * b] * dj[1];
        if (sidef[f]) wo += g;
        else wn += g;
      }
      put(smem + L::Wf + (bb * NP + jj) * LF + fq, &ex.Wf[bb][jj], wo);
      put(smem + L::Wn + (bb * NP + jj) * LF + fq, &ex.Wn[bb][f][jj], wn);
    }
    if (a > 0) {
      // cv[f][q][k] = s_f sum_d C_v(q, a, k; grad_d U_b) n_f[d] (faces this element lifts)
      for (int idx = tid; idx < NBV * 3 * NV * 2; idx += T) {
        const int k = idx & 1, r = idx >> 1, q = r % NV, fb = r / NV, f = fb % 3, b = b0 + fb / 3;
        const double* C = Cv + ((q * 4 + a) * 2 + k) * 12;
        cvv[idx] = sidef[f] ? s_lift[f] * (C[4 + 2 * b] * nuo[f][0] + C[5 + 2 * b] * nuo[f][1]) : 0.0;
      }
      // cf[f][q] = s_S sum_d C_f(f, q, a; grad_d U_b of the flux side) n_f[d]
      for (int idx = tid; idx < NBV * F3; idx += T) {
        const int fq = idx % F3, f = fq / NF, b = b0 + idx / F3;
        const double* C = Cf + fq * 64 + a * 16 + 8 + 2 * b;
        cff[idx] = s_lift[f] * (C[0] * nus[f][0] + C[1] * nus[f][1]);
      }
    }
    __syncthreads();
    for (int idx = tid; idx < NBV * NP * 2 * NV; idx += T) {
      const int jj = idx % NP, r = idx / NP, kq = r % (2 * NV), bb = r / (2 * NV);
      enc(smem + L::Wv + (bb * NP + jj) * LV + kq, ex.Wv[bb][jj]);
    }
    for (int idx = tid; idx < NBV * NP * F3; idx += T) {
      const int jj = idx % NP, r = idx / NP, fq = r % F3, bb = r / F3;
      enc(smem + L::Wf + (bb * NP + jj) * LF + fq, ex.Wf[bb][jj]);
      enc(smem + L::Wn + (bb * NP + jj) * LF + fq, ex.Wn[bb][fq / NF][jj]);
    }
    if (a > 0) {
      // Y[f][i][q] = sum_k dphi_k,i(q) cv[f][q][k]
      for (int idx = tid; idx < NBV * 3 * NP * NV; idx += T) {
        const int i = idx % NP, r = idx / NP, q = r % NV, fb = r / NV, f = fb % 3, bb = fb / 3;
        if (!sidef[f]) continue;
        const double* di = tb.dphi_v + 2 * (q * NP + i);
        const double* c = cvv + ((size_t)fb * NV + q) * 2;
        put(smem + L::Y + (fb * NP + i) * LY + q, &ex.Y[bb][f][i], di[0] * c[0] + di[1] * c[1]);
      }
      __syncthreads();
      for (int idx = tid; idx < NBV * 3 * NP * NV; idx += T) {
        const int i = idx % NP, r = idx / NP, q = r % NV, fb = r / NV, f = fb % 3, bb = fb / 3;
        if (sidef[f]) enc(smem + L::Y + (fb * NP + i) * LY + q, ex.Y[bb][f][i]);
      }
      __syncthreads();
      // Lam[f][i][p] = d r_(a,i) / d jump_(f,b)(p): volume part (faces this element lifts)
      // minus the face part (test function phi_i on face f, the flux side's lifting row)
      for (int idx = tid; idx < NBV * NP * F3; idx += T) {
        const int i = idx % NP, r = idx / NP, fp = r % F3, bb = r / F3, f = fp / NF, p = fp - f * NF;
        double acc = 0.0;
        if (has_grad(a, b0 + bb)) {
          for (int q = 0; q < NF; ++q) {
            int step;
            const double* A = lift_row(tb, sidef[f], f, gf[f], q, step);
            acc -= tb.phi_f[(f * NF + q) * NP + i] * (cff[bb * F3 + f * NF + q] * A[p * step]);
          }
          if (sidef[f])
            acc = fix_dot<NV>(fix(L::Y) + ((bb * 3 + f) * NP + i) * LY, fix(L::lv) + fp * LY, ex.Y[bb][f][i], ex.lv[fp], acc);
        }
        put(smem + L::Lam + (bb * NP + i) * LF + fp, &ex.Lam[bb][i], acc);
        if (tagf[f] == 1) LamW[((f * 4 + b0 + bb) * NP + i) * NF + p] = acc;
      }
      __syncthreads();
      for (int idx = tid; idx < NBV * NP * F3; idx += T) {
        const int i = idx % NP, r = idx / NP, fp = r % F3, bb = r / F3;
        enc(smem + L::Lam + (bb * NP + i) * LF + fp, ex.Lam[bb][i]);
      }
    }
    __syncthreads();
    for (int idx = tid; idx < NBV * 4 * NP * NP; idx += T) {
      const int i = idx % NP, r = idx / NP, jj = r % NP, sb = r / NP, slot = sb & 3, bb = sb >> 2, b = b0 + bb;
      const bool grad = has_grad(a, b);
      const Fix* lam = fix(L::Lam) + (bb * NP + i) * LF;
      double acc = 0.0;
      if (slot == 0) {
        acc = fix_dot<2 * NV>(fix(L::dV) + i * LV, fix(L::Wv) + (bb * NP + jj) * LV, ex.dV[i], ex.Wv[bb][jj], acc);
        acc = fix_dot_minus<F3>(fix(L::pF) + i * LF, fix(L::Wf) + (bb * NP + jj) * LF, ex.pF[i], ex.Wf[bb][jj], acc);
        // d jump / d u_e = -phi_j (the wall state's own dependence is added below)
        if (grad) acc = fix_dot_minus<F3>(lam, fix(L::pF) + jj * LF, ex.Lam[bb][i], ex.pF[jj], acc);
      } else {
        const int f = slot - 1, o = f * NF;
        if (tagf[f] == 0) {
          acc = fix_dot_minus<NF>(fix(L::pF) + i * LF + o, fix(L::Wn) + (bb * NP + jj) * LF + o, ex.pF[i],
                                  ex.Wn[bb][f][jj], acc);
          // d jump / d u_nbr = +phi_j of the neighbour at the matched point
          if (grad) acc = fix_dot<NF>(lam + o, fix(L::pN) + jj * LF + o, ex.Lam[bb][i], ex.pN[jj], acc);
        }
      }
      Jd[(size_t)slot * nb2 + (size_t)(b * NP + jj) * NB + a * NP + i] = acc;
    }
    if (has_wall && a > 0 && b0 + NBV == 4) {
      __syncthreads();
      // wall points: the jump U_wall(U-) - U- also depends on U- through the wall state:
      // J_(a,c) += sum_b sum_p Lam_(a,b)[i][p] dU_wall,b/dU-_c phi_j(p)
      for (int idx = tid; idx < 4 * NP * NP; idx += T) {
        const int c = idx / (NP * NP), rem = idx - c * NP * NP, jj = rem / NP, i = rem - jj * NP;
        double acc = 0.0;
        for (int f = 0; f < 3; ++f) {
          if (tagf[f] != 1) continue;
          for (int p = 0; p < NF; ++p) {
            const double phij = tb.phi_f[(f * NF + p) * NP + jj];
            const double* G = Gb + (f * NF + p) * 16;
            double s = 0.0;
#pragma unroll
            for (int bb = 0; bb < 4; ++bb) s += LamW[((f * 4 + bb) * NP + i) * NF + p] * G[bb * 4 + c];
            acc += s * phij;
          }
        }
        Jd[(size_t)(c * NP + jj) * NB + a * NP + i] += acc;
      }
    }
  }
}

// ------------------------------------------------------------------------ QoI
// Per element: sum over its wall faces of w L (f . v_G, f_x), f = momentum part of the wall
// flux (with the CDG lifting of the wall jump; the wall faces are always lifted by the element);
// T = DualV<3>: their derivatives for the three motion seeds of the frame, (power, force) by seed.
template <class T>
__global__ void __launch_bounds__(RES_WARPS * 32)
    k_qoi(DevMesh m, DevTables tb, Phys ph, FrameT<T> fr, const double* __restrict__ u, double* __restrict__ out) {
  constexpr int W = sizeof(T) / sizeof(double);
  __shared__ double s_J[RES_WARPS][3 * kMaxQf * 4 * W];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e = blockIdx.x * RES_WARPS + warp;
  if (e >= m.ne) return;
  const int Np = tb.Np, nb = tb.nb, nqf = tb.nqf;
  const double* ue = u + (size_t)e * nb;
  T* Js = reinterpret_cast<T*>(s_J[warp]);
  T P[4];
  frame_P(fr, m.BinvT + 4 * e, P);
  for (int idx = lane; idx < 3 * nqf; idx += 32) {
    int f = idx / nqf, q = idx - f * nqf;
    if (m.tag[3 * e + f] != 1) continue;
    double um[4];
    interp_val(ue, Np, tb.phi_f + (f * nqf + q) * Np, um);
    T Um[4], vG[2], Ub[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) Um[a] = T(um[a]);
    double X, Y;
    ref_to_X(m, e, tb.xi_f[2 * (f * nqf + q)], tb.xi_f[2 * (f * nqf + q) + 1], X, Y);
    mesh_velocity(fr, ph, X, Y, vG);
    wall_state(Um, vG, Ub);
#pragma unroll
    for (int a = 0; a < 4; ++a) Js[(f * kMaxQf + q) * 4 + a] = Ub[a] - Um[a];
  }
  __syncwarp();
  T pw(0.0), fx(0.0);
  for (int idx = lane; idx < 3 * nqf; idx += 32) {
    int f = idx / nqf, q = idx - f * nqf;
    if (m.tag[3 * e + f] != 1) continue;
    T Um[4], dUm[4][2], n[2], vG[2], H[4];
    interp(ue, Np, tb.phi_f + (f * nqf + q) * Np, tb.dphi_f + 2 * (f * nqf + q) * Np, P, Um, dUm);
    rotate_normal(fr, m.N + 6 * e + 2 * f, n);
    lift_add(dUm, n, m.s_own[3 * e + f], tb.lift_f + (f * nqf + q) * nqf, 1, Js + f * kMaxQf * 4, nqf);
    double X, Y;
    ref_to_X(m, e, tb.xi_f[2 * (f * nqf + q)], tb.xi_f[2 * (f * nqf + q) + 1], X, Y);
    mesh_velocity(fr, ph, X, Y, vG);
    face_flux(1, 1, Um, Um, dUm, n, vG, m.c11[3 * e + f], ph, H);
    double wl = tb.w_f[q] * m.L[3 * e + f];
    pw += wl * (H[1] * vG[0] + H[2] * vG[1]);
    fx += wl * H[1];
  }
  constexpr int NC = sizeof(T) == sizeof(double) ? 1 : 3;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    double a0 = part(pw, c), a1 = part(fx, c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    }
    if (lane == 0) {
      out[(size_t)2 * NC * e + 2 * c] = a0;
      out[(size_t)2 * NC * e + 2 * c + 1] = a1;
    }
  }
}

// g_e = d(w0 P^h + w1 F_x^h)/du_e on wall elements (zero elsewhere).  Seeds at each wall
// point: U- (4) and the lifted gradient Q (8); the lifting adds the chain through the
// jumps U_wall(U-) - U- at every point p of the face: Lam_b(p) = sum_q sum_d C_Q(q)_(b,d)
// n_d s lift_f[q][p], folded into the state seeds as Lam(p) (dU_wall/dU- - I).
__global__ void __launch_bounds__(RES_WARPS * 32)
    k_qoi_du(DevMesh m, DevTables tb, Phys ph, FrameT<double> fr, const double* __restrict__ u, double w0, double w1,
             double* __restrict__ g) {
  __shared__ double s_C[RES_WARPS][3 * kMaxQf * NSV];
  __shared__ double s_J[RES_WARPS][3 * kMaxQf * 4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e = blockIdx.x * RES_WARPS + warp;
  if (e >= m.ne) return;
  const int Np = tb.Np, nb = tb.nb, nqf = tb.nqf;
  const bool wall = m.tag[3 * e] == 1 || m.tag[3 * e + 1] == 1 || m.tag[3 * e + 2] == 1;
  if (!wall) {
    for (int o = lane; o < nb; o += 32) g[(size_t)e * nb + o] = 0.0;
    return;
  }
  double* C = s_C[warp];
  double* Js = s_J[warp];
  const double* ue = u + (size_t)e * nb;
  double P[4];
  frame_P(fr, m.BinvT + 4 * e, P);
  FrameT<Dual> frd;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    frd.Q[k] = Dual(fr.Q[k]);
    frd.Qd[k] = Dual(fr.Qd[k]);
  }
  frd.hd = Dual(fr.hd);
  for (int idx = lane; idx < 3 * nqf; idx += 32) {
    int f = idx / nqf, q = idx - f * nqf;
    if (m.tag[3 * e + f] != 1) continue;
    double Um[4], vG[2], Ub[4], X, Y;
    interp_val(ue, Np, tb.phi_f + (f * nqf + q) * Np, Um);
    ref_to_X(m, e, tb.xi_f[2 * (f * nqf + q)], tb.xi_f[2 * (f * nqf + q) + 1], X, Y);
    mesh_velocity(fr, ph, X, Y, vG);
    wall_state(Um, vG, Ub);
#pragma unroll
    for (int a = 0; a < 4; ++a) Js[(f * kMaxQf + q) * 4 + a] = Ub[a] - Um[a];
  }
  __syncwarp();
  for (int task = lane; task < 3 * nqf * NSV; task += 32) {
    int f = task / (nqf * NSV);
    int rem = task - f * nqf * NSV;
    int q = rem / NSV, s = rem - q * NSV;
    if (m.tag[3 * e + f] != 1) {
      C[(f * kMaxQf + q) * NSV + s] = 0.0;
      continue;
    }
    double U0[4], dU0[4][2], n0[2];
    interp(ue, Np, tb.phi_f + (f * nqf + q) * Np, tb.dphi_f + 2 * (f * nqf + q) * Np, P, U0, dU0);
    rotate_normal(fr, m.N + 6 * e + 2 * f, n0);
    lift_add(dU0, n0, m.s_own[3 * e + f], tb.lift_f + (f * nqf + q) * nqf, 1, Js + f * kMaxQf * 4, nqf);
    Dual Um[4], dUm[4][2], n[2], vG[2], H[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      Um[a] = Dual(U0[a], s == a ? 1.0 : 0.0);
      dUm[a][0] = Dual(dU0[a][0], s == 4 + 2 * a ? 1.0 : 0.0);
      dUm[a][1] = Dual(dU0[a][1], s == 5 + 2 * a ? 1.0 : 0.0);
    }
    rotate_normal(frd, m.N + 6 * e + 2 * f, n);
    double X, Y;
    ref_to_X(m, e, tb.xi_f[2 * (f * nqf + q)], tb.xi_f[2 * (f * nqf + q) + 1], X, Y);
    mesh_velocity(frd, ph, X, Y, vG);
    face_flux(1, 1, Um, Um, dUm, n, vG, m.c11[3 * e + f], ph, H);
    double wl = tb.w_f[q] * m.L[3 * e + f];
    Dual val = w0 * (H[1] * vG[0] + H[2] * vG[1]) + w1 * H[1];
    C[(f * kMaxQf + q) * NSV + s] = wl * val.d;
  }
  __syncwarp();
  // fold the lifting chain into the state seeds (reads gradient seeds, writes state seeds)
  double add[4] = {0.0, 0.0, 0.0, 0.0};
  int fp = -1;
  if (lane < 3 * nqf) {
    const int f = lane / nqf, p = lane - f * nqf;
    if (m.tag[3 * e + f] == 1) {
      fp = lane;
      double n0[2];
      rotate_normal(fr, m.N + 6 * e + 2 * f, n0);
      const double s = m.s_own[3 * e + f];
      double lam[4] = {0.0, 0.0, 0.0, 0.0};
      for (int q = 0; q < nqf; ++q) {
        const double A = tb.lift_f[(f * nqf + q) * nqf + p] * s;
        const double* Cq = C + (f * kMaxQf + q) * NSV;
#pragma unroll
        for (int bb = 0; bb < 4; ++bb) lam[bb] += A * (Cq[4 + 2 * bb] * n0[0] + Cq[5 + 2 * bb] * n0[1]);
      }
      double Um[4], vG[2], X, Y;
      interp_val(ue, Np, tb.phi_f + (f * nqf + p) * Np, Um);
      ref_to_X(m, e, tb.xi_f[2 * (f * nqf + p)], tb.xi_f[2 * (f * nqf + p) + 1], X, Y);
      mesh_velocity(fr, ph, X, Y, vG);
      Dual vd[2] = {Dual(vG[0]), Dual(vG[1])};
      for (int c = 0; c < 4; ++c) {
        Dual Ud[4], Ub[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) Ud[a] = Dual(Um[a], a == c ? 1.0 : 0.0);
        wall_state(Ud, vd, Ub);
#pragma unroll
        for (int bb = 0; bb < 4; ++bb) add[c] += lam[bb] * (Ub[bb].d - (bb == c ? 1.0 : 0.0));
      }
    }
  }
  __syncwarp();
  if (fp >= 0) {
    const int f = fp / nqf, p = fp - f * nqf;
#pragma unroll
    for (int c = 0; c < 4; ++c) C[(f * kMaxQf + p) * NSV + c] += add[c];
  }
  __syncwarp();
  for (int o = lane; o < nb; o += 32) {
    int b = o / Np, j = o - b * Np;
    double acc = 0.0;
    for (int f = 0; f < 3; ++f) {
      if (m.tag[3 * e + f] != 1) continue;
      for (int q = 0; q < nqf; ++q) {
        const double* dj = tb.dphi_f + 2 * ((f * nqf + q) * Np + j);
        double phij = tb.phi_f[(f * nqf + q) * Np + j];
        double g0 = P[0] * dj[0] + P[1] * dj[1];
        double g1 = P[2] * dj[0] + P[3] * dj[1];
        const double* Cq = C + (f * kMaxQf + q) * NSV;
        acc += Cq[b] * phij + Cq[4 + 2 * b] * g0 + Cq[5 + 2 * b] * g1;
      }
    }
    g[(size_t)e * nb + o] = acc;
  }
}

}  // namespace

static int res_blocks(int ne) { return (ne + RES_WARPS - 1) / RES_WARPS; }

template <int PD, class T, bool NEWTON = false>
static cudaError_t run_residual(const DevMesh& m, const DevTables& tb, const Phys& ph, const FrameT<T>& fr,
                                const double* u, const double* kappa, double* out, cudaStream_t st,
                                const StageNewton& nw = {}) {
  using L = Res<PD, T, NEWTON>;
  struct Setup {
    cudaError_t err;
    int resident;
  };
  // one device per process (see pp_create)
  static const Setup setup = [] {
    Setup r{cudaSuccess, 0};
    r.err = cudaFuncSetAttribute(k_residual<PD, T, NEWTON>, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * L::words);
    if (r.err != cudaSuccess) return r;
    int per_sm = 0, dev = 0, sms = 0;
    r.err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_residual<PD, T, NEWTON>, L::THREADS, 8 * L::words);
    if (r.err == cudaSuccess) r.err = cudaGetDevice(&dev);
    if (r.err == cudaSuccess) r.err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (r.err == cudaSuccess && per_sm < 1) r.err = cudaErrorInvalidConfiguration;
    r.resident = per_sm * sms;
    return r;
  }();
  if (setup.err != cudaSuccess) return setup.err;
  // groups as large as fill the warps, smaller on meshes that would leave SMs without one
  int eb = (m.ne + setup.resident - 1) / setup.resident;
  eb = eb < 1 ? 1 : eb > L::EB ? L::EB : eb;
  const int groups = (m.ne + eb - 1) / eb, grid = groups < setup.resident ? groups : setup.resident;
  k_residual<PD, T, NEWTON><<<grid, L::THREADS, 8 * L::words, st>>>(m, tb, ph, fr, u, kappa, out, nw, eb);
  return cudaGetLastError();
}

cudaError_t launch_residual(const DevMesh& m, const DevTables& tb, const Phys& ph, const FrameT<double>& fr,
                            const double* u, double* r, cudaStream_t st) {
  ProfScope ps(PP_K_RESIDUAL, st);
  switch (tb.p) {
    case 1: return run_residual<1, double>(m, tb, ph, fr, u, nullptr, r, st);
    case 2: return run_residual<2, double>(m, tb, ph, fr, u, nullptr, r, st);
    case 3: return run_residual<3, double>(m, tb, ph, fr, u, nullptr, r, st);
    case 4: return run_residual<4, double>(m, tb, ph, fr, u, nullptr, r, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_stage_residual(const DevMesh& m, const DevTables& tb, const Phys& ph, const FrameT<double>& fr,
                                  const StageNewton& nw, double* R, cudaStream_t st) {
  ProfScope ps(PP_K_RESIDUAL, st);
  switch (tb.p) {
    case 1: return run_residual<1, double, true>(m, tb, ph, fr, nullptr, nullptr, R, st, nw);
    case 2: return run_residual<2, double, true>(m, tb, ph, fr, nullptr, nullptr, R, st, nw);
    case 3: return run_residual<3, double, true>(m, tb, ph, fr, nullptr, nullptr, R, st, nw);
    case 4: return run_residual<4, double, true>(m, tb, ph, fr, nullptr, nullptr, R, st, nw);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_residual_dframe(const DevMesh& m, const DevTables& tb, const Phys& ph, const FrameT<DualV<3>>& fr,
                                   const double* u, const double* kappa, double* per_elem, cudaStream_t st) {
  ProfScope ps(PP_K_OTHER, st);
  switch (tb.p) {
    case 1: return run_residual<1, DualV<3>>(m, tb, ph, fr, u, kappa, per_elem, st);
    case 2: return run_residual<2, DualV<3>>(m, tb, ph, fr, u, kappa, per_elem, st);
    case 3: return run_residual<3, DualV<3>>(m, tb, ph, fr, u, kappa, per_elem, st);
    case 4: return run_residual<4, DualV<3>>(m, tb, ph, fr, u, kappa, per_elem, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_jacobian(const DevMesh& m, const DevTables& tb, const Phys& ph, const FrameT<double>& fr,
                            const double* u, double* J, cudaStream_t st) {
  ProfScope ps(PP_K_JACOBIAN, st);
  switch (tb.p) {
#define PP_JAC(PD)                                                                                       \
  case PD: {                                                                                             \
    constexpr int bytes = 8 * Jac<PD>::words;                                                            \
    static const cudaError_t attr =                                                                      \
        cudaFuncSetAttribute(k_jacobian<PD>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);        \
    if (attr != cudaSuccess) return attr;                                                                \
    k_jacobian<PD><<<m.ne, Jac<PD>::T, bytes, st>>>(m, tb, ph, fr, u, J);                                \
    break;                                                                                               \
  }
    PP_JAC(1)
    PP_JAC(2)
    PP_JAC(3)
    PP_JAC(4)
#undef PP_JAC
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_qoi(const DevMesh& m, const DevTables& tb, const Phys& ph, const FrameT<double>& fr,
                       const double* u, double* per_elem, cudaStream_t st) {
  ProfScope ps(PP_K_OTHER, st);
  k_qoi<double><<<res_blocks(m.ne), RES_WARPS * 32, 0, st>>>(m, tb, ph, fr, u, per_elem);
  return cudaGetLastError();
}

cudaError_t launch_qoi_dframe(const DevMesh& m, const DevTables& tb, const Phys& ph, const FrameT<DualV<3>>& fr,
                              const double* u, double* per_elem, cudaStream_t st) {
  ProfScope ps(PP_K_OTHER, st);
  k_qoi<DualV<3>><<<res_blocks(m.ne), RES_WARPS * 32, 0, st>>>(m, tb, ph, fr, u, per_elem);
  return cudaGetLastError();
}

cudaError_t launch_qoi_du(const DevMesh& m, const DevTables& tb, const Phys& ph, const FrameT<double>& fr,
                          const double* u, double w0, double w1, double* g, cudaStream_t st) {
  ProfScope ps(PP_K_OTHER, st);
  k_qoi_du<<<res_blocks(m.ne), RES_WARPS * 32, 0, st>>>(m, tb, ph, fr, u, w0, w1, g);
  return cudaGetLastError();
}

}  // namespace pp
