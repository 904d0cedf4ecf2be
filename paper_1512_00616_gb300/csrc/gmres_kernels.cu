// A whole stage solve in one launch: restarted GMRES on the folded stage operator
// (M - cJ) D^{-1} = I + B (B = O D^{-1}, three nb x nb blocks per element), with half of the
// elements eliminated exactly.
//
// Red-black reduction.  The mesh gives every element a class (see pp_mesh_create): the
// eliminated elements I are pairwise not face neighbours, so the rows of I read
//   y_I = b_I - B_IR y_R,
// and the kept elements R satisfy (I + K) y_R = b_R - B_RI b_I with
//   K v = B_RR v - B_RI (B_IR v).
// One application of K reads every block of B once, like one application of B, but the Krylov
// vectors have half the length and the Krylov space of K advances by two applications of B per
// step (the O-grids are two-colourable, so B_RR = 0 there and K = -B_RI B_IR), so a solve takes
// about half the steps.  The residual of the reduced system is the residual of the full one
// (the eliminated rows hold exactly), so the stopping rule is the same:
// |b - (I + B) y| <= max(rtol |b|, atol).
//
// The recurrence runs on K with the unit shift added back to the Hessenberg diagonal, classical
// Gram-Schmidt with a second pass only when the first cancels more than half of |w|^2 (as the
// separate kernels of linalg_kernels.cu do it for the other GMRES levels).
//
// Why one launch: a step of the separate kernels was two launches (operator, Arnoldi) with an
// event and a host wait, plus about ten small launches per solve; at 32 triangles a step took
// 32 us of which under 1 us is arithmetic, at 2048 triangles (p = 3) 65 us for 26 us of FP64
// issue.  Here every CTA keeps its elements for the whole solve:
//  - one CTA per SM (cooperative launch), kept elements split evenly, eliminated likewise; up to
//    kClusterRows kept rows a single cluster of 8 CTAs with the hardware cluster barrier
//    (0.24 us against 1.2 us for the barrier of the whole grid);
//  - one thread per matrix row: 3 nb column-major entries read straight from L2 / HBM (a warp
//    reads 256 contiguous bytes per column) against operand slices staged in shared memory.
//    The FP64 pipe issues one warp instruction per 19 clocks and SM, so this path needs no
//    shared-memory staging of the blocks; the first columns of a phase are loaded before
//    the barrier that its operand waits for;
//  - the own slices of the basis live in shared memory when they fit;
//  - three barriers per step (v -> B_IR v -> K v and its projections -> next v); every CTA sums
//    the CTA partials itself in one fixed order, so all CTAs hold bitwise the same coefficients,
//    take the same decisions, and results are reproducible bit for bit;
//  - the Givens update runs on one thread of each CTA while the others wait at the barrier.
// Barrier waits of the whole grid are bounded (about a second); an expired wait sets the error
// word and ends the CTA, and every other CTA's wait then expires too.
#include <algorithm>

#include "pp_internal.h"
#include "prof.h"
#include "reduce.cuh"
#include "../../include/pp_prof.h"

namespace pp {

namespace {

constexpr int GT = 320;                // threads per CTA
constexpr int GW = GT / 32;
constexpr int GM = kGmresMaxRestart;   // most basis vectors per cycle
constexpr int GCTAS = 152;             // partial columns
constexpr int GLD = GM + 2;            // partial rows
constexpr int kCluster = 8;
constexpr unsigned long long kBarrierNs = 1000000000ull;
// barrier words, on their own 128-byte lines
constexpr int BAR_COUNT = 0, BAR_EXIT = 32, BAR_ERROR = 64, BAR_WORDS = 96;
constexpr int kDynSmemMax = 180 * 1024;

// What a stage solve leaves for the host (device memory, sticky over a sweep).
// rec[0]: failure code (0 none, 1 cap reached, 4 non-finite, 8 barrier), rec[1]: steps taken.

template <class S>
struct GArgs {
  int ne, nR;
  const int* list;     // [ne] element at each position, kept elements first
  const int* src;      // [ne][3] position of the face neighbours, -1 on the boundary
  const S* B;          // [ne][3][nb nb]
  const S* D;          // [ne][nb nb] block inverses: x = D y
  int d_row, d_col;    // strides of a row / column of D
  const S* b;          // [ne][nb] right-hand side
  S* x;                // [ne][nb] solution
  S* ywarm;            // [nR nb] y of the kept elements: initial guess (warm), written at the end; or null
  int warm;
  double rtol, atol;
  int maxit, m, need_conv;
  S* V;                // [m + 1][nR nb]
  S* z;                // [(ne - nR) nb]
  S* y;                // [nR nb]
  double* partial;     // [2][GLD][GCTAS]
  unsigned* bar;
  double* rec;
  int v_smem;          // own basis slices in dynamic shared memory
  int own_max;         // most kept rows of a CTA
};

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier over all CTAs of the launch, split into arrive and wait so that loads that do not
// depend on it go between.  Whole grid: a monotonic count (arrivals add with release, waiters
// poll it with acquire), reset by the CTA that leaves the kernel last.  Cluster: the hardware
// barrier, which orders global memory at cluster scope.
template <bool CL>
struct Barrier {
  unsigned* bar;
  unsigned target;
  int* s_ok;
  __device__ void arrive() {
    if constexpr (CL) {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    } else {
      __syncthreads();
      target += gridDim.x;
      if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar + BAR_COUNT) : "memory");
    }
  }
  __device__ bool wait() {
    if constexpr (CL) {
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      return true;
    } else {
      if (threadIdx.x == 0) {
        unsigned v = 0, it = 0;
        unsigned long long t0 = 0;
        int ok = 1;
        for (;;) {
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar + BAR_COUNT) : "memory");
          if (v >= target) break;
          if ((++it & 255u) == 0u) {
            if (t0 == 0) t0 = now_ns();
            else if (now_ns() - t0 > kBarrierNs) {
              atomicExch(bar + BAR_ERROR, 1u);
              ok = 0;
              break;
            }
          }
        }
        *s_ok = ok;
      }
      __syncthreads();
      return *s_ok != 0;
    }
  }
  // after the last barrier of the launch
  __device__ void leave() {
    if constexpr (!CL) {
      if (threadIdx.x == 0 && atomicAdd(bar + BAR_EXIT, 1u) == gridDim.x - 1u) {
        bar[BAR_COUNT] = 0u;
        bar[BAR_EXIT] = 0u;
      }
    }
  }
};

template <int NB>
struct Rows {
  static constexpr int E = GT / NB;       // elements per pass, one thread per row
  static constexpr int C = 3 * NB;        // columns of a row of B
  static constexpr int U = NB == 12 ? 12 : NB == 24 ? 18 : 20;  // columns in flight per thread
  static constexpr int XS = E * C;        // operand slices of a pass
  static constexpr int XP = (XS + GT - 1) / GT;
};

template <int NB, class S>
struct GShared {
  double H[GM * (GM + 1) / 2];  // triangular factor, packed columns
  double g[GM + 1], cs[GM], sn[GM], red[GLD], coef[GM];
  S xs[2][Rows<NB>::XS];
  double nrm2, inv, beta, tol;
  int need, ok, stop;
};

// First U columns of this thread's row of pass 0 (they do not depend on the operand).
template <int NB, class S>
__device__ __forceinline__ void load_cols(const S* row, int c0, S* out) {
#pragma unroll
  for (int u = 0; u < Rows<NB>::U; ++u) out[u] = __ldg(row + (size_t)(c0 + u) * NB);
}

template <int NB, class S>
struct RowRef {
  bool on;
  const S* row;
  __device__ RowRef(const GArgs<S>& a, int pos, int end) {
    const int el = threadIdx.x / NB;
    on = el < Rows<NB>::E && pos + el < end;
    row = on ? a.B + (size_t)a.list[pos + el] * (3 * NB * NB) + (threadIdx.x - el * NB) : a.B;
  }
};

// operand entry idx of the pass at `pos`: the neighbours' slices of v (kept) or z (eliminated)
template <int NB, class S>
__device__ __forceinline__ S operand(const GArgs<S>& a, int pos, int end, int idx, const S* v, const S* z) {
  const int el = idx / (3 * NB), rem = idx - el * 3 * NB, f = rem / NB, c = rem - f * NB;
  if (idx >= Rows<NB>::XS || pos + el >= end) return S(0);
  const int s = a.src[3 * (pos + el) + f];
  if (s < 0) return S(0);
  return s < a.nR ? __ldcg(v + (size_t)s * NB + c) : __ldcg(z + (size_t)(s - a.nR) * NB + c);
}

// Rows [p0, p1) of B times the operand: epi(position, row of the element, sum).  `ready` is
// called between the first block loads and the first operand loads (the barrier wait); when it
// returns false nothing further is done.
template <int NB, class S, class Ready, class Epi>
__device__ __forceinline__ bool rows_product(const GArgs<S>& a, GShared<NB, S>& sh, int p0, int p1, const S* v,
                                             const S* z, Ready ready, Epi epi) {
  using R = Rows<NB>;
  S cur[R::U], nxt[R::U];
  RowRef<NB, S> ref(a, p0, p1);
  if (ref.on) load_cols<NB, S>(ref.row, 0, cur);
  if (!ready()) return false;
#pragma unroll
  for (int q = 0; q < R::XP; ++q) {
    const int idx = threadIdx.x + q * GT;
    if (idx < R::XS) sh.xs[0][idx] = operand<NB, S>(a, p0, p1, idx, v, z);
  }
  __syncthreads();
  int buf = 0;
  for (int pos = p0; pos < p1; pos += R::E) {
    const bool more = pos + R::E < p1;
    S xr[R::XP];
    if (more) {
#pragma unroll
      for (int q = 0; q < R::XP; ++q) xr[q] = operand<NB, S>(a, pos + R::E, p1, threadIdx.x + q * GT, v, z);
    }
    const int el = threadIdx.x / NB, row = threadIdx.x - el * NB;
    const RowRef<NB, S> next(a, pos + R::E, p1);
    S acc[4] = {S(0), S(0), S(0), S(0)};
    if (ref.on) {
      const S* xe = sh.xs[buf] + el * R::C;
#pragma unroll
      for (int c0 = 0; c0 < R::C; c0 += R::U) {
        if (c0 + R::U < R::C) load_cols<NB, S>(ref.row, c0 + R::U, nxt);
        else if (next.on) load_cols<NB, S>(next.row, 0, nxt);
#pragma unroll
        for (int u = 0; u < R::U; ++u) acc[u & 3] += cur[u] * xe[c0 + u];
#pragma unroll
        for (int u = 0; u < R::U; ++u) cur[u] = nxt[u];
      }
      epi(pos + el, row, (acc[0] + acc[1]) + (acc[2] + acc[3]));
    }
    ref = next;
    if (more) {
      buf ^= 1;
#pragma unroll
      for (int q = 0; q < R::XP; ++q)
        if (threadIdx.x + q * GT < R::XS) sh.xs[buf][threadIdx.x + q * GT] = xr[q];
      __syncthreads();
    }
  }
  return true;
}

// CTA partials of (V_0 .. V_{k-1}, w) . w over the own rows -> region[t][cta].  A warp takes Q
// vectors at a time over all own rows, so no second reduction over the warps is needed.
template <int Q, class S>
__device__ __forceinline__ void own_dots(const S* V, size_t ldv, int k, const S* w, int n, double* region) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t0 = warp * Q; t0 <= k; t0 += GW * Q) {
    const S* p[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) p[q] = t0 + q < k ? V + (size_t)(t0 + q) * ldv : w;
    S a[Q], c[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) a[q] = c[q] = S(0);
    int i = lane;
    for (; i + 32 < n; i += 64) {
      const S w0 = w[i], w1 = w[i + 32];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        a[q] += p[q][i] * w0;
        c[q] += p[q][i + 32] * w1;
      }
    }
    if (i < n) {
      const S w0 = w[i];
#pragma unroll
      for (int q = 0; q < Q; ++q) a[q] += p[q][i] * w0;
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) a[q] += c[q];
    warp_reduce_scatter<Q, S>(a, lane);
    constexpr int sh = 5 - ILog2<Q>::value;
    if ((lane & ((1 << sh) - 1)) == 0) {
      const int t = t0 + (lane >> sh);
      if (t <= k) region[(size_t)t * GCTAS + blockIdx.x] = (double)a[0];
    }
  }
}

template <class S>
__device__ __forceinline__ void cta_dots(const S* V, size_t ldv, int k, const S* w, int n, double* region) {
  if (k < GW) own_dots<1, S>(V, ldv, k, w, n, region);
  else if (k < 2 * GW) own_dots<2, S>(V, ldv, k, w, n, region);
  else own_dots<4, S>(V, ldv, k, w, n, region);
}

// out[t] = sum over the CTAs of region[t][.], t < nk, the same order in every CTA
template <int Q>
__device__ __forceinline__ void sum_region(int nk, const double* region, double* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = gridDim.x;
  for (int t0 = warp * Q; t0 < nk; t0 += GW * Q) {
    double a[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      a[q] = 0.0;
      if (t0 + q < nk)
#pragma unroll
        for (int r = 0; r < (GCTAS + 31) / 32; ++r) {
          const int c = lane + 32 * r;
          if (c < G) a[q] += __ldcg(region + (size_t)(t0 + q) * GCTAS + c);
        }
    }
    warp_reduce_scatter<Q, double>(a, lane);
    constexpr int sh = 5 - ILog2<Q>::value;
    if ((lane & ((1 << sh) - 1)) == 0 && t0 + (lane >> sh) < nk) out[t0 + (lane >> sh)] = a[0];
  }
}

__device__ __forceinline__ void sum_partials(int nk, const double* region, double* out) {
  if (nk <= GW) sum_region<1>(nk, region, out);
  else if (nk <= 2 * GW) sum_region<2>(nk, region, out);
  else sum_region<4>(nk, region, out);
  __syncthreads();
}

template <int NB, class S, bool CL>
__global__ void __launch_bounds__(GT, 1) k_stage_gmres(const GArgs<S> a) {
  __shared__ GShared<NB, S> sh;
  extern __shared__ __align__(16) unsigned char dyn[];
  if (__ldcg(a.rec) != 0.0) return;  // an earlier solve of the sweep failed
  const int tid = threadIdx.x, G = gridDim.x, bi = blockIdx.x;
  const int nR = a.nR, nI = a.ne - a.nR;
  const int r0 = (int)((long long)nR * bi / G), r1 = (int)((long long)nR * (bi + 1) / G);
  const int i0 = nR + (int)((long long)nI * bi / G), i1 = nR + (int)((long long)nI * (bi + 1) / G);
  const int own = (r1 - r0) * NB;
  const size_t nv = (size_t)nR * NB;
  // own slices of the basis: shared memory, or the slices of V itself
  S* Vo = a.v_smem ? reinterpret_cast<S*>(dyn) : a.V + (size_t)r0 * NB;
  const size_t ldv = a.v_smem ? (size_t)a.own_max : nv;
  Barrier<CL> bar{a.bar, 0u, &sh.ok};
  double* const region0 = a.partial;
  double* const region1 = a.partial + (size_t)GLD * GCTAS;
  S* const yo = a.y + (size_t)r0 * NB;
  bool alive = true;
  bool guess = a.ywarm && a.warm;
  int total = 0, flag = 0;

  if (guess)
    for (int i = tid; i < own; i += GT) yo[i] = a.ywarm[(size_t)r0 * NB + i];
  bar.arrive();
  for (bool first = true; alive; first = false) {
    // ---- residual of the reduced system: z = b_I - B_IR y, r = b_R - y - B_RR y - B_RI z
    const S* yv = a.y;
    if (guess) {
      alive = rows_product<NB, S>(a, sh, i0, i1, yv, a.z, [&] { return bar.wait(); },
                                  [&](int pos, int row, S s) {
                                    a.z[(size_t)(pos - nR) * NB + row] = a.b[(size_t)a.list[pos] * NB + row] - s;
                                  });
    } else {
      alive = bar.wait();
      for (int i = tid; alive && i < (i1 - i0) * NB; i += GT) {
        const int pos = i0 + i / NB, row = i % NB;
        a.z[(size_t)(pos - nR) * NB + row] = a.b[(size_t)a.list[pos] * NB + row];
      }
      for (int i = tid; alive && i < own; i += GT) yo[i] = S(0);
    }
    if (!alive) break;
    double bb = 0.0;
    if (first) {
      // |b|^2 over all own rows
      S s = S(0);
      for (int i = tid; i < own + (i1 - i0) * NB; i += GT) {
        const int pos = i < own ? r0 + i / NB : i0 + (i - own) / NB;
        const S v = a.b[(size_t)a.list[pos] * NB + i % NB];
        s += v * v;
      }
      S t[1] = {s};
      warp_reduce_scatter<1, S>(t, tid & 31);
      bb = (double)t[0];
    }
    bar.arrive();
    alive = rows_product<NB, S>(a, sh, r0, r1, yv, a.z, [&] { return bar.wait(); }, [&](int pos, int row, S s) {
      const int i = (pos - r0) * NB + row;
      Vo[i] = a.b[(size_t)a.list[pos] * NB + row] - __ldcg(yo + i) - s;
    });
    if (!alive) break;
    if (first) {
      if ((tid & 31) == 0) sh.coef[tid >> 5] = bb;
    }
    __syncthreads();
    if (first && tid == 0) {
      double s = 0.0;
      for (int w = 0; w < GW; ++w) s += sh.coef[w];
      region0[GCTAS + bi] = s;
    }
    own_dots<1, S>(Vo, ldv, 0, Vo, own, region0);
    bar.arrive();
    if (!(alive = bar.wait())) break;
    sum_partials(first ? 2 : 1, region0, sh.red);
    if (tid == 0) {
      const double beta = sqrt(fmax(sh.red[0], 0.0));
      if (first) sh.tol = fmax(a.rtol * sqrt(fmax(sh.red[1], 0.0)), a.atol);
      sh.beta = beta;
      sh.inv = beta > 0.0 ? 1.0 / beta : 0.0;
      sh.g[0] = beta;
      sh.stop = !isfinite(sh.red[0]) || (first && !isfinite(sh.red[1])) ? 4 : (beta <= sh.tol ? 1 : 0);
    }
    __syncthreads();
    flag = sh.stop;
    int k = 0;  // columns of this cycle
    if (flag == 0) {
      const S inv = S(sh.inv);
      for (int i = tid; i < own; i += GT) {
        const S v = Vo[i] * inv;
        Vo[i] = v;
        if (a.v_smem) a.V[(size_t)r0 * NB + i] = v;
      }
      __syncthreads();
      if (tid == 0) sh.stop = 0;
      bar.arrive();
      for (int j = 0; j < a.m; ++j) {
        const S* vj = a.V + (size_t)j * nv;
        S* wo = Vo + (size_t)(j + 1) * ldv;
        k = j + 1;
        // ---- z = -B_IR v_j; the wait publishes the Givens update of the step before
        alive = rows_product<NB, S>(
            a, sh, i0, i1, vj, a.z,
            [&] {
              if (!bar.wait()) return false;
              if constexpr (CL) __syncthreads();
              return sh.stop == 0;
            },
            [&](int pos, int row, S s) { a.z[(size_t)(pos - nR) * NB + row] = -s; });
        if (!alive) {
          k = j;
          break;
        }
        bar.arrive();
        // ---- w = B_RR v_j + B_RI z
        alive = rows_product<NB, S>(a, sh, r0, r1, vj, a.z, [&] { return bar.wait(); },
                                    [&](int pos, int row, S s) { wo[(pos - r0) * NB + row] = s; });
        if (!alive) break;
        __syncthreads();
        // ---- projections and |w|^2
        cta_dots<S>(Vo, ldv, k, wo, own, region1);
        bar.arrive();
        if (!(alive = bar.wait())) break;
        sum_partials(k + 1, region1, sh.red);
        if (tid < 32) {
          double s = 0.0;
          for (int t = tid; t < k; t += 32) s += sh.red[t] * sh.red[t];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (tid == 0) {
            const double w2 = sh.red[k], n2 = w2 - s;
            sh.need = !(s <= 0.5 * w2);
            sh.nrm2 = n2;
            sh.inv = n2 > 0.0 ? 1.0 / sqrt(n2) : 0.0;
          }
          for (int t = tid; t < k; t += 32) sh.coef[t] = sh.red[t];
        }
        __syncthreads();
        const bool need = sh.need != 0;
        if (need) {
          // second pass: w -= V h1, h2 = V^T w, |w|^2; then w -= V h2 with its norm by a third exchange
          for (int pass = 0; pass < 2 && alive; ++pass) {
            for (int i = tid; i < own; i += GT) {
              S s = wo[i];
              for (int t = 0; t < k; ++t) s -= S(sh.red[t]) * Vo[(size_t)t * ldv + i];
              wo[i] = s;
            }
            __syncthreads();
            double* region = pass == 0 ? region0 : region1;
            if (pass == 0) cta_dots<S>(Vo, ldv, k, wo, own, region);
            else own_dots<1, S>(Vo, ldv, 0, wo, own, region);
            bar.arrive();
            if (!(alive = bar.wait())) break;
            sum_partials(pass == 0 ? k + 1 : 1, region, sh.red);
            if (pass == 0) {
              for (int t = tid; t < k; t += GT) sh.coef[t] += sh.red[t];
              __syncthreads();
            }
          }
          if (!alive) break;
          if (tid == 0) {
            sh.nrm2 = sh.red[0];
            sh.inv = sh.red[0] > 0.0 ? 1.0 / sqrt(sh.red[0]) : 0.0;
          }
          __syncthreads();
        }
        // ---- v_{j+1}
        const S inv = S(sh.inv);
        S* vn = a.V + (size_t)(j + 1) * nv + (size_t)r0 * NB;
        for (int i = tid; i < own; i += GT) {
          S s = wo[i];
          if (!need) {
            S s1 = S(0), s2 = S(0), s3 = S(0);
            int t = 0;
            for (; t + 3 < k; t += 4) {
              const S* p = Vo + (size_t)t * ldv + i;
              s -= S(sh.coef[t]) * p[0];
              s1 -= S(sh.coef[t + 1]) * p[ldv];
              s2 -= S(sh.coef[t + 2]) * p[2 * ldv];
              s3 -= S(sh.coef[t + 3]) * p[3 * ldv];
            }
            for (; t < k; ++t) s -= S(sh.coef[t]) * Vo[(size_t)t * ldv + i];
            s = (s + s1) + (s2 + s3);
          }
          s *= inv;
          wo[i] = s;
          if (a.v_smem) vn[i] = s;
        }
        bar.arrive();
        // ---- Givens update of column j on one thread, behind the barrier's latency
        if (tid == 32) {
          double* col = sh.H + j * (j + 1) / 2;
          const double hn = sqrt(fmax(sh.nrm2, 0.0));
          double carry = sh.coef[0] + (j == 0 ? 1.0 : 0.0);
          for (int i = 0; i < j; ++i) {
            const double nxt = sh.coef[i + 1] + (i + 1 == j ? 1.0 : 0.0);
            const double c = sh.cs[i], s = sh.sn[i];
            col[i] = c * carry + s * nxt;
            carry = c * nxt - s * carry;
          }
          const double rr = hypot(carry, hn);
          const double ir = rr > 0.0 ? 1.0 / rr : 0.0;
          const double c = rr > 0.0 ? carry * ir : 1.0, s = hn * ir;
          sh.cs[j] = c;
          sh.sn[j] = s;
          col[j] = rr;
          const double gj = sh.g[j], gn = -s * gj;
          sh.g[j + 1] = gn;
          sh.g[j] = c * gj;
          int stop = 0;
          if (fabs(gn) <= sh.tol) stop = 1;
          if (hn == 0.0) stop = 2;
          if (!isfinite(hn) || !isfinite(gn)) stop = 4;
          if (stop == 0 && total + k >= a.maxit) stop = 3;
          sh.stop = stop;
        }
        __syncwarp();
      }
      // a stop seen in the wait of the next step ends the cycle there; the last step's own wait follows here
      if (alive) {
        if (!(alive = bar.wait())) break;
        __syncthreads();
      } else if (sh.ok == 0 && !CL) {
        break;
      }
      alive = true;
      flag = sh.stop;
      total += k;
      __syncthreads();
    }
    if (flag == 4) break;
    // ---- y_R += V c, c = H^{-1} g (one warp, column oriented)
    if (tid < 32) {
      for (int t = tid; t < k; t += 32) sh.coef[t] = sh.g[t];
      __syncwarp();
      for (int i = k - 1; i >= 0; --i) {
        const double* col = sh.H + i * (i + 1) / 2;
        const double d = col[i], c = d != 0.0 ? sh.coef[i] / d : 0.0;
        __syncwarp();
        if (tid == 0) sh.coef[i] = c;
        for (int r = tid; r < i; r += 32) sh.coef[r] -= col[r] * c;
        __syncwarp();
      }
    }
    __syncthreads();
    for (int i = tid; i < own; i += GT) {
      S s = __ldcg(yo + i);
      for (int t = 0; t < k; ++t) s += S(sh.coef[t]) * Vo[(size_t)t * ldv + i];
      yo[i] = s;
      if (a.ywarm) a.ywarm[(size_t)r0 * NB + i] = s;
    }
    bar.arrive();
    guess = true;
    if (flag != 0 || total >= a.maxit) break;
  }
  if (alive && flag != 4) {
    // ---- y_I = b_I - B_IR y_R, then x = D y element by element
    alive = rows_product<NB, S>(a, sh, i0, i1, a.y, a.z, [&] { return bar.wait(); }, [&](int pos, int row, S s) {
      a.z[(size_t)(pos - nR) * NB + row] = a.b[(size_t)a.list[pos] * NB + row] - s;
    });
  }
  if (alive && flag != 4) {
    using R = Rows<NB>;
    __syncthreads();
    const int nown = (r1 - r0) + (i1 - i0);
    const int el = tid / NB, row = tid - el * NB;
    for (int q0 = 0; q0 < nown; q0 += R::E) {
      __syncthreads();
      for (int idx = tid; idx < R::E * NB && q0 + idx / NB < nown; idx += GT) {
        const int q = q0 + idx / NB, c = idx % NB;
        sh.xs[0][idx] = q < r1 - r0 ? __ldcg(yo + (size_t)q * NB + c)
                                    : __ldcg(a.z + (size_t)(i0 - nR + q - (r1 - r0)) * NB + c);
      }
      __syncthreads();
      if (el < R::E && q0 + el < nown) {
        const int q = q0 + el, pos = q < r1 - r0 ? r0 + q : i0 + q - (r1 - r0);
        const size_t e = a.list[pos];
        const S* d = a.D + e * (NB * NB) + (size_t)row * a.d_row;
        S acc[4] = {S(0), S(0), S(0), S(0)};
#pragma unroll(NB % 20 == 0 ? 20 : 12)
        for (int c = 0; c < NB; ++c) acc[c & 3] += __ldg(d + (size_t)c * a.d_col) * sh.xs[0][el * NB + c];
        a.x[e * NB + row] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
      }
    }
  }
  if (bi == 0 && tid == 0) {
    a.rec[1] += (double)total;
    if (!alive) a.rec[0] = 8.0;
    else if (flag == 4) a.rec[0] = 4.0;
    else if (a.need_conv && flag != 1 && flag != 2) a.rec[0] = 1.0;
  }
  if (alive) bar.leave();
}

struct GSetup {
  cudaError_t err = cudaSuccess;
  int sms = 0;
};

template <int NB, class S>
cudaError_t launch_gmres(GArgs<S>& a, cudaStream_t st) {
  // one device per process (see pp_create); thread-safe static initialization
  static const GSetup setup = [] {
    GSetup s;
    int dev = 0;
    s.err = cudaGetDevice(&dev);
    if (s.err == cudaSuccess) s.err = cudaDeviceGetAttribute(&s.sms, cudaDevAttrMultiProcessorCount, dev);
    if (s.err == cudaSuccess)
      s.err = cudaFuncSetAttribute(k_stage_gmres<NB, S, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemMax);
    if (s.err == cudaSuccess)
      s.err = cudaFuncSetAttribute(k_stage_gmres<NB, S, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemMax);
    return s;
  }();
  if (setup.err != cudaSuccess) return setup.err;
  const bool cluster = (int64_t)a.nR * NB <= kClusterRows;
  const int G = cluster ? kCluster : std::min(std::min(setup.sms, GCTAS), a.nR);
  a.own_max = (a.nR + G - 1) / G * NB;
  const size_t need = sizeof(S) * (size_t)(a.m + 1) * a.own_max;
  a.v_smem = need <= (size_t)kDynSmemMax;
  const size_t smem = a.v_smem ? need : 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(GT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  if (cluster) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
  } else {
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
  }
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cluster ? cudaLaunchKernelEx(&cfg, k_stage_gmres<NB, S, true>, (const GArgs<S>)a)
                 : cudaLaunchKernelEx(&cfg, k_stage_gmres<NB, S, false>, (const GArgs<S>)a);
}

}  // namespace

size_t stage_gmres_partial_words() { return (size_t)2 * GLD * GCTAS; }
int stage_gmres_barrier_words() { return BAR_WORDS; }

template <class S>
cudaError_t launch_stage_gmres(const DevMesh& m, int nb, const StageGmres<S>& q, cudaStream_t st) {
  if (q.m < 1 || q.m > GM || m.n_kept < 1) return cudaErrorInvalidValue;
  ProfScope ps(sizeof(S) == 8 ? PP_K_STAGE_GMRES : PP_K_STAGE_GMRES32, st);
  GArgs<S> a{};
  a.ne = m.ne;
  a.nR = m.n_kept;
  a.list = m.order;
  a.src = m.order_nbr;
  a.B = q.B;
  a.D = q.D;
  a.d_row = q.d_trans ? nb : 1;
  a.d_col = q.d_trans ? 1 : nb;
  a.b = q.b;
  a.x = q.x;
  a.ywarm = q.ywarm;
  a.warm = q.warm;
  a.rtol = q.rtol;
  a.atol = q.atol;
  a.maxit = q.maxit;
  a.m = q.m;
  a.need_conv = q.need_conv;
  a.V = q.V;
  a.z = q.z;
  a.y = q.y;
  a.partial = q.partial;
  a.bar = q.bar;
  a.rec = q.rec;
  switch (nb) {
    case 12: return launch_gmres<12, S>(a, st);
    case 24: return launch_gmres<24, S>(a, st);
    case 40: return launch_gmres<40, S>(a, st);
    case 60: return launch_gmres<60, S>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_stage_gmres<double>(const DevMesh&, int, const StageGmres<double>&, cudaStream_t);
template cudaError_t launch_stage_gmres<float>(const DevMesh&, int, const StageGmres<float>&, cudaStream_t);

}  // namespace pp
