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
// event and a host wait, plus about ten small launches per solve; at 32 triangles (p = 1) a step
// took 32 us of which under 1 us is arithmetic, at 2048 triangles (p = 3) 65 us.  Here every CTA
// keeps its elements for the whole solve:
//  - one CTA per SM (cooperative launch), kept elements split evenly, eliminated likewise; up to
//    kClusterRows kept rows a single cluster of 8 CTAs with the hardware cluster barrier
//    (0.24 us against 1.2 us for the barrier of the whole grid);
//  - FP64 products run on the integer pipe (fixed.cuh): the FP64 pipe issues one warp instruction
//    per 19 clocks and SM, so one application of K at 2048 triangles is 19 us of FP64 issue against
//    10 us for its 79 MB from L2 at the 25 bytes per clock and SM that were measured;
//  - one thread per matrix row: its 3 nb entries through a ring in shared memory that cp.async fills
//    ahead, over passes and barriers; with the columns in registers instead (two chunks of 20) the
//    compiler spilled and a product of 8192 triangles ran at 4.2 TB/s instead of 5.9;
//  - the own slices of the basis live in shared memory when they fit beside a short ring;
//  - three barriers per step (v -> B_IR v -> K v and its projections -> next v); every CTA sums
//    the CTA partials itself in one fixed order, so all CTAs hold bitwise the same coefficients,
//    take the same decisions, and results are reproducible bit for bit;
//  - the Givens update runs on a warp of its own during the next step's first product.
// Measured (GB300), time of a reduced step (which does the work of two steps of the separate
// kernels): 2048 triangles, p = 3: 25 us (two separate steps 130 us; the first one-launch version
// with FP64 FMAs 44 us; 10 us are the blocks from L2, 5 us the three barriers); 8192 triangles: 100 us
// (330; 155; 46 us at the HBM rate); 32 triangles, p = 1: 12 us (64; 19).
// Barrier waits of the whole grid are bounded (about a second); an expired wait ends the CTA, which
// reports it in the record itself (solve_record.h).  The host then clears the barrier words.
#pragma once

#include <algorithm>

#include "fixed.cuh"
#include "pp_internal.h"
#include "prof.h"
#include "reduce.cuh"
#include "solve_record.h"
#include "../../include/pp_prof.h"

namespace pp {

namespace {

constexpr int GT = 320;                // worker threads per CTA; one more warp does the scalar chain
constexpr int GW = GT / 32;
constexpr int GALL = GT + 32;
constexpr int GM = kGmresMaxRestart;   // most basis vectors per cycle
constexpr int GCTAS = 152;             // partial columns
constexpr int GLD = GM + 2;            // partial rows
constexpr int kCluster = 8;
// how the CTAs of a solve exchange data
enum Mode { kGrid, kClusters, kSingle };
constexpr unsigned long long kBarrierNs = 1000000000ull;
// barrier words, on their own 128-byte lines
constexpr int BAR_COUNT = 0, BAR_EXIT = 32, BAR_WORDS = 64;
constexpr int kSmemMax = 227 * 1024;   // shared memory of a CTA

// Blocks and exchanged vectors: FP64 ones travel as 58-bit fixed-point words with one exponent
// per block row / element slice (fixed.cuh), FP32 ones as they are.
template <class S>
struct Wire {
  using T = float;
};
template <>
struct Wire<double> {
  using T = Fix;
};

template <class S>
struct GArgs {
  using W = typename Wire<S>::T;
  int ne, nR;
  const int* list;     // [ne] element at each position, kept elements first
  const int* src;      // [ne][3] position of the face neighbours, -1 on the boundary
  const W* B;          // [ne][3][nb nb]
  const int* Bexp;     // [ne][3][nb] exponents of the rows (FP64)
  const S* D;          // [ne][nb nb] block inverses: x = D y
  int d_row, d_col;    // strides of a row / column of D
  const S* b;          // [ne][nb] right-hand side
  S* x;                // [ne][nb] solution
  S* ywarm;            // [nR nb] (scaled) y of the kept elements: initial guess (warm), written at the end; or null
  int warm;
  double rtol, atol;
  int maxit, m, need_conv;
  W* V;                // [m + 1][nR nb] own slices of the basis (unless in shared memory)
  int* Vexp;           // [m + 1][nR] their exponents (FP64)
  S* y;                // [ne nb] y by position, each slice read by its own CTA only
  W* wire;             // [ne nb] exchanged operand by position: v or y (kept), z (eliminated)
  int* wexp;           // [ne] exponents of its slices (FP64)
  double* partial;     // [2][GLD][GCTAS]
  unsigned* bar;
  double* rec;         // [0] failure: 1 cap, 4 non-finite, 8 barrier; [1] steps taken
  int own_max;         // most kept elements of a CTA
  VarScale scale;      // FP64: B and all vectors but b and x are scaled by these powers of two
};

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier over all CTAs of the launch, split into arrive and wait so that loads that do not
// depend on it go between.  One CTA: a block barrier.  Whole grid: a monotonic count (arrivals add with release, waiters
// poll it with acquire), reset by the CTA that leaves the kernel last.  Cluster: the hardware
// barrier, which orders global memory at cluster scope.
template <int MODE>
struct Barrier {
  unsigned* bar;
  unsigned target;
  int* s_ok;
  __device__ void arrive() {
    if constexpr (MODE == kClusters) {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    } else if constexpr (MODE == kGrid) {
      __syncthreads();
      target += gridDim.x;
      if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar + BAR_COUNT) : "memory");
    }
  }
  __device__ bool wait() {
    if constexpr (MODE == kClusters) {
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      return true;
    } else if constexpr (MODE == kSingle) {
      __syncthreads();
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
    if constexpr (MODE == kGrid) {
      if (threadIdx.x == 0 && atomicAdd(bar + BAR_EXIT, 1u) == gridDim.x - 1u) {
        bar[BAR_COUNT] = 0u;
        bar[BAR_EXIT] = 0u;
      }
    }
  }
};

template <int NB, class S>
struct Rows {
  static constexpr int E = GT / NB;  // most elements per pass, one thread per row
  static constexpr int CE = E >= 13 ? E : 24 / E * E;  // elements whose coefficients are held at a time
  static constexpr int C = 3 * NB;   // columns of a row of B
  static constexpr int U = (NB <= 24 ? 6 : 10) * (sizeof(S) == 8 ? 1 : 2);  // columns per ring chunk
  static constexpr int NCH = C / U;  // chunks per row
  // chunks of the deep ring: a ring runs on from row to row, so its length divides NCH (a slot would
  // hold another chunk than the one that is read from it otherwise, and a row shorter than the ring
  // would be read beyond its end)
  static constexpr int DEEP = NCH % 6 == 0 ? 6 : 3;
  static_assert(C % U == 0 && NCH % 3 == 0 && NCH % DEEP == 0, "a ring takes whole rows");
  static constexpr int XS = E * C;   // operand entries of a pass
  static constexpr int XP = (XS + GT - 1) / GT;
};

// Ring of a thread's next columns of B in shared memory, filled by cp.async: a thread copies and
// reads only its own words, so no barrier is involved, and the ring runs on over passes, products
// and grid barriers.  ST chunks of U columns: 3 (at most 77 KB) beside a basis in shared memory,
// Rows::DEEP without (6, and 3 for FP32 rows of 12 and 60 columns, which 6 chunks do not divide).
// The blocks interleave VW columns (fold_index), so a copy is 16 bytes per thread and 512
// contiguous bytes per warp: with one word per copy the SM's outstanding requests, not the bytes,
// were the limit (8192 triangles: a product at 5.1 TB/s instead of 5.9 in FP64 words, mixed-precision
// sweeps 231 ms instead of 205).
template <int NB, class S, int ST>
struct Ring {
  using R = Rows<NB, S>;
  using W = typename Wire<S>::T;
  static constexpr int VW = FoldOut<S>::VW, UV = R::U / VW;
  static constexpr int WORDS = ST * R::U * GT;
  int4* mine;  // this thread's vectors, GT apart
  __device__ explicit Ring(void* base) : mine(reinterpret_cast<int4*>(base) + threadIdx.x) {}
  // vector v of chunk `slot`
  __device__ __forceinline__ void get(int slot, int v, W (&w)[VW]) const {
    const int4 x = mine[(slot * UV + v) * GT];
    if constexpr (sizeof(S) == 8) {
      w[0] = Fix{x.x, x.y};
      w[1] = Fix{x.z, x.w};
    } else {
      w[0] = __int_as_float(x.x);
      w[1] = __int_as_float(x.y);
      w[2] = __int_as_float(x.z);
      w[3] = __int_as_float(x.w);
    }
  }
  // chunk c of the row into `slot`, as one group (an empty one without a row)
  __device__ __forceinline__ void put(int slot, const W* row, bool on, int c) const {
    if (on) {
#pragma unroll
      for (int v = 0; v < UV; ++v) {
        const unsigned dst = static_cast<unsigned>(__cvta_generic_to_shared(mine + (slot * UV + v) * GT));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(row + (size_t)(c * UV + v) * (NB * VW))
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ __forceinline__ void wait() const { asm volatile("cp.async.wait_group %0;" ::"n"(ST - 1) : "memory"); }
  __device__ __forceinline__ void drain() const { asm volatile("cp.async.wait_all;" ::: "memory"); }
  __device__ __forceinline__ void prime(const W* row, bool on) const {
#pragma unroll
    for (int c = 0; c < ST; ++c) put(c, row, on, c);
  }
};

template <int NB, class S>
struct GShared {
  double H[GM * (GM + 1) / 2];  // triangular factor, packed columns
  double g[GM + 1], cs[GM], sn[GM], red[GLD], coef[GM];
  typename Wire<S>::T xs[2][Rows<NB, S>::XS];
  int xe[2][3 * Rows<NB, S>::E];
  int emax[3][Rows<NB, S>::E];  // exponents of the slices being published
  typename Wire<S>::T cq[sizeof(S) == 8 ? Rows<NB, S>::CE * GM : 1];  // coefficients against the elements' slices
  int ce[sizeof(S) == 8 ? Rows<NB, S>::CE : 1];
  double dpart[3][GLD], single[2][GLD];
  double nrm2, inv, tol;
  int need, ok, stop;
};

// One pass over up to E elements at positions pos .. end - 1: thread = row of an element.
template <int NB>
struct Lane {
  int el, row;
  __device__ Lane() : el(threadIdx.x / NB), row(threadIdx.x - threadIdx.x / NB * NB) {}
};

// Word of a row in an own slice of the basis in global memory (FP64): the eight lanes that share a slice in
// cta_dots, two per variable, read consecutive words.  In shared memory the rows lie in their order: the
// lanes' words two apart then fall into different banks as they are.
template <int NB, bool VS>
__host__ __device__ constexpr int slice_at(int row) {
  constexpr int NP = NB / 4;
  if (VS) return row;
  const int var = row / NP, j = row - var * NP;
  return j / 2 * 8 + (NP % 2 == 1 && j == NP - 1 ? var : 2 * var + j % 2);
}

// Writes a pass's rows (one value per thread, `on` where there is one) to the exchanged operand
// (shared = true) and to the own slice `slot` of the basis (with exponents at slot_e, element
// index own_el) unless that is null.
template <int NB, class S, bool VS>
__device__ __forceinline__ void publish(const GArgs<S>& a, GShared<NB, S>& sh, int& turn, bool on, int el, int row,
                                        int pos, S val, bool shared, typename Wire<S>::T* slot = nullptr,
                                        int* slot_e = nullptr, int own_el = 0) {
  if constexpr (sizeof(S) == 8) {
    // three exponent buffers in turn: the one cleared here is used by the call after the next
    int* em = sh.emax[turn];
    turn = turn == 2 ? 0 : turn + 1;
    if (on) atomicMax(em + el, fix_exponent(val));
    __syncthreads();
    if (on) {
      const int e = em[el];
      const Fix q = fix_encode(val, e);
      if (shared) {
        reinterpret_cast<int2*>(a.wire)[(size_t)pos * NB + row] = make_int2(q.hi, q.lo);
        if (row == 0) a.wexp[pos] = e;
      }
      if (slot) {
        slot[own_el * NB + slice_at<NB, VS>(row)] = q;
        if (row == 0) slot_e[own_el] = e;
      }
    }
    const int clear = turn == 2 ? 0 : turn + 1;
    if (threadIdx.x < Rows<NB, S>::E) sh.emax[clear][threadIdx.x] = 0;
  } else if (on) {
    if (shared) a.wire[(size_t)pos * NB + row] = val;
    if (slot) slot[own_el * NB + slice_at<NB, VS>(row)] = val;
  }
}

// operand entry idx of the pass at `pos`
template <int NB, class S, int MODE>
__device__ __forceinline__ typename Wire<S>::T operand(const GArgs<S>& a, int pos, int end, int idx) {
  using W = typename Wire<S>::T;
  const int el = idx / (3 * NB), rem = idx - el * 3 * NB, f = rem / NB, c = rem - f * NB;
  if (idx >= Rows<NB, S>::XS || pos + el >= end) return W{};
  const int s = a.src[3 * (pos + el) + f];
  if (s < 0) return W{};
  if constexpr (sizeof(S) == 8) {
    const int2* p = reinterpret_cast<const int2*>(a.wire) + (size_t)s * NB + c;
    const int2 v = MODE == kSingle ? *p : __ldcg(p);
    return Fix{v.x, v.y};
  } else {
    const W* p = a.wire + (size_t)s * NB + c;
    return MODE == kSingle ? *p : __ldcg(p);
  }
}

template <class S, int MODE>
__device__ __forceinline__ int operand_exp(const GArgs<S>& a, int pos, int end, int idx) {
  if (sizeof(S) != 8 || pos + idx / 3 >= end) return 0;
  const int s = a.src[3 * pos + idx];
  return s < 0 ? 0 : MODE == kSingle ? a.wexp[s] : __ldcg(a.wexp + s);
}

// this thread's row of B in the first of the equal passes over [p0, p1), or null
template <int NB, class S>
__device__ __forceinline__ const typename Wire<S>::T* first_row_of(const GArgs<S>& a, int p0, int p1) {
  using R = Rows<NB, S>;
  const Lane<NB> ln;
  const int np = (p1 - p0 + R::E - 1) / R::E, per = np > 0 ? (p1 - p0 + np - 1) / np : 0;
  return ln.el < per && p0 + ln.el < p1 ? a.B + (size_t)a.list[p0 + ln.el] * (3 * NB * NB) + ln.row * FoldOut<S>::VW : nullptr;
}

// Rows at positions [p0, p1) of B times the exchanged operand: epi(on, element of the pass, row,
// position, sum) is called by every thread of the CTA.  On entry the ring holds the first chunks of
// `row` (first_row_of the range), on return those of `after`.  `ready` is called before the first
// operand loads (the barrier wait); when it returns false nothing is done.  The scalar warp calls
// `side` while the others do the first pass.
template <int NB, class S, int ST, int MODE, class Ready, class Side, class Epi>
__device__ __forceinline__ bool rows_product(const GArgs<S>& a, GShared<NB, S>& sh, const Ring<NB, S, ST>& ring,
                                             int p0, int p1, const typename Wire<S>::T* row,
                                             const typename Wire<S>::T* after, Ready ready, Side side, Epi epi) {
  using R = Rows<NB, S>;
  using W = typename Wire<S>::T;
  constexpr int NBB = 3 * NB * NB, VW = FoldOut<S>::VW;
  static_assert(R::NCH % ST == 0, "slot c % ST holds chunk c of every row");
  static_assert(NB <= kFixTerms, "a block row is one exact sum");
  const Lane<NB> ln;
  // passes of equal size
  const int np = (p1 - p0 + R::E - 1) / R::E, per = np > 0 ? (p1 - p0 + np - 1) / np : 0;
  if (!ready()) return false;
  if (p0 == p1) {
    ring.drain();
    ring.prime(after, after != nullptr);
  }
  if (threadIdx.x < GT) {
#pragma unroll
    for (int q = 0; q < R::XP; ++q) {
      const int idx = threadIdx.x + q * GT;
      if (idx < R::XS) sh.xs[0][idx] = operand<NB, S, MODE>(a, p0, p1, idx);
    }
    if (threadIdx.x < 3 * R::E) sh.xe[0][threadIdx.x] = operand_exp<S, MODE>(a, p0, p1, threadIdx.x);
  }
  __syncthreads();
  if (threadIdx.x >= GT) side();
  int buf = 0;
  for (int pos = p0; pos < p1; pos += per) {
    const int nx = pos + per;
    const bool more = nx < p1, on = row != nullptr;
    W xr[R::XP];
    int er = 0;
    if (more && threadIdx.x < GT) {
#pragma unroll
      for (int q = 0; q < R::XP; ++q) xr[q] = operand<NB, S, MODE>(a, nx, p1, threadIdx.x + q * GT);
      if (threadIdx.x < 3 * R::E) er = operand_exp<S, MODE>(a, nx, p1, threadIdx.x);
    }
    const W* const row2 = !more ? after
                          : ln.el < per && nx + ln.el < p1 ? a.B + (size_t)a.list[nx + ln.el] * NBB + ln.row * VW : nullptr;
    const W* xe = sh.xs[buf] + ln.el * R::C;
    S sum = S(0);
    if constexpr (sizeof(S) == 8) {
      int eb[3] = {0, 0, 0};
      if (on) {
        // the row's exponents lie as its block does
        const int* be = a.Bexp + ((size_t)(row - a.B) - ln.row * VW) / NB + ln.row;
#pragma unroll
        for (int f = 0; f < 3; ++f) eb[f] = __ldg(be + f * NB);
      }
      FixDot acc;
#pragma unroll
      for (int c = 0; c < R::NCH; ++c) {
        ring.wait();
        if (on) {
#pragma unroll
          for (int u = 0; u < R::U; u += VW) {
            const int col = c * R::U + u;
            W w[VW];
            ring.get(c % ST, u / VW, w);
            if (col % NB == 0) acc.clear();
            acc.add(w[0], xe[col]);
            acc.add(w[1], xe[col + 1]);
            if ((col + VW) % NB == 0) {
              const int f = col / NB, ex = sh.xe[buf][3 * ln.el + f];
              sum = acc.result(eb[f] + ex, eb[f] == 0x7ff || ex == 0x7ff, sum);
            }
          }
        }
        if (c + ST < R::NCH) ring.put(c % ST, row, on, c + ST);
        else ring.put(c % ST, row2, row2 != nullptr, c + ST - R::NCH);
      }
    } else {
      S acc[4] = {S(0), S(0), S(0), S(0)};
#pragma unroll
      for (int c = 0; c < R::NCH; ++c) {
        ring.wait();
        if (on) {
#pragma unroll
          for (int u = 0; u < R::U; u += VW) {
            W w[VW];
            ring.get(c % ST, u / VW, w);
#pragma unroll
            for (int v = 0; v < VW; ++v) acc[v] += w[v] * xe[c * R::U + u + v];
          }
        }
        if (c + ST < R::NCH) ring.put(c % ST, row, on, c + ST);
        else ring.put(c % ST, row2, row2 != nullptr, c + ST - R::NCH);
      }
      sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    }
    epi(on, ln.el, ln.row, pos + ln.el, sum);
    row = row2;
    if (more) {
      buf ^= 1;
      if (threadIdx.x < GT) {
#pragma unroll
        for (int q = 0; q < R::XP; ++q)
          if (threadIdx.x + q * GT < R::XS) sh.xs[buf][threadIdx.x + q * GT] = xr[q];
        if (threadIdx.x < 3 * R::E) sh.xe[buf][threadIdx.x] = er;
      }
      __syncthreads();
    }
  }
  return true;
}

// CTA partials of (V_0 .. V_{k-1}, w) . w over the own rows -> region[t][cta], w in slot k.
// FP32: a warp takes Q vectors at a time over all own rows.
template <int Q>
__device__ __forceinline__ void own_dots(const float* V, size_t ldv, int k, int from, int n, double* region,
                                         int rs) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp >= GW) return;
  const float* w = V + (size_t)k * ldv;
  for (int t0 = from + warp * Q; t0 <= k; t0 += GW * Q) {
    const float* p[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) p[q] = t0 + q < k ? V + (size_t)(t0 + q) * ldv : w;
    float a[Q], c[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) a[q] = c[q] = 0.f;
    int i = lane;
    for (; i + 32 < n; i += 64) {
      const float w0 = w[i], w1 = w[i + 32];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        a[q] += p[q][i] * w0;
        c[q] += p[q][i + 32] * w1;
      }
    }
    if (i < n) {
      const float w0 = w[i];
#pragma unroll
      for (int q = 0; q < Q; ++q) a[q] += p[q][i] * w0;
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) a[q] += c[q];
    warp_reduce_scatter<Q, float>(a, lane);
    constexpr int sh = 5 - ILog2<Q>::value;
    if ((lane & ((1 << sh) - 1)) == 0) {
      const int t = t0 + (lane >> sh);
      if (t <= k) region[(size_t)(t - from) * rs + blockIdx.x] = (double)a[0];
    }
  }
}

// `from`: first vector (0, or k for |w|^2 alone), written from region row 0 on.
template <int NB, bool VS, bool Small = false>
__device__ __forceinline__ void cta_dots(const float* V, const int*, const VarScale&, size_t ldv, size_t, int k,
                                         int from, int nel, double* region, int rs, double (*)[GLD]) {
  const int nk = k - from, n = nel * NB;
  if (nk < GW) own_dots<1>(V, ldv, k, from, n, region, rs);
  else if (nk < 2 * GW) own_dots<2>(V, ldv, k, from, n, region, rs);
  else own_dots<4>(V, ldv, k, from, n, region, rs);
}

// FP64: eight lanes per vector, two per variable, so that a lane's words have one scale; each lane turns
// its exact integer sum over every other entry of its variable into a double, so the FP64 pipe sees two
// instructions per slice.  A warp takes four vectors; with few vectors up to three warps share the elements
// of four.  Small: the vector may be small (residuals; the basis is normalized).
template <int NB, bool VS, bool Small = false>
__device__ __forceinline__ void cta_dots(const Fix* V, const int* Vexp, const VarScale& scale, size_t ldv, size_t lde,
                                         int k, int from, int nel, double* region, int rs, double (*dpart)[GLD]) {
  constexpr int NP = NB / 4, P = (NP + 1) / 2;
  const int lane = threadIdx.x & 31, l = lane & 7, warp = threadIdx.x >> 5, var = l >> 1, half = l & 1;
  const int unscale = -2 * scale[var];
  const int groups = (k - from) / 4 + 1, share = min(3, max(1, GW / groups));
  const Fix* w = V + (size_t)k * ldv;
  const int* we = Vexp + (size_t)k * lde;
  for (int g = warp; g < groups * share && warp < GW; g += GW) {
    const int sp = g / groups, t = from + (g - sp * groups) * 4 + (lane >> 3);
    double s = 0.0;
    if (t <= k) {
      const Fix* v = V + (size_t)t * ldv;
      const int* ve = Vexp + (size_t)t * lde;
#pragma unroll 3
      for (int el = sp; el < nel; el += share) {
        FixDot acc;
        acc.clear();
#pragma unroll
        for (int c = 0; c < P; ++c) {
          // slice_at of row var NP + 2 c + half
          const bool odd = NP % 2 == 1 && c == P - 1;
          const int i = el * NB + (VS ? var * NP + 2 * c + half : 8 * c + (odd ? var : l));
          if (!odd || half == 0) acc.add(v[i], w[i]);
        }
        const int e1 = ve[el], e2 = we[el];
        s = acc.result<Small>(e1 + e2 + unscale, e1 == 0x7ff || e2 == 0x7ff, s);
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (l == 0 && t <= k) dpart[sp][t - from] = s;
  }
  __syncthreads();
  for (int t = threadIdx.x; t <= k - from; t += GALL) {
    double s = dpart[0][t];
    for (int sp = 1; sp < share; ++sp) s += dpart[sp][t];
    region[(size_t)t * rs + blockIdx.x] = s;
  }
}

// out[t] = sum over the CTAs of region[t][.], t < nk, the same in every CTA: a warp per output, the
// partials as integers against their largest exponent (exact sums, no FP64 additions).
template <int MODE, bool Small = false>
__device__ __forceinline__ void sum_partials(int nk, const double* region, double* out) {
  if constexpr (MODE == kSingle) {
    for (int t = threadIdx.x; t < nk; t += GALL) out[t] = region[t];
    __syncthreads();
    return;
  }
  constexpr int R = (GCTAS + 31) / 32, Q = 3;  // Q outputs of a warp at a time: their loads overlap
  const int lane = threadIdx.x & 31, G = gridDim.x;
  for (int t0 = threadIdx.x >> 5; t0 < nk && threadIdx.x < GT; t0 += Q * GW) {
    double v[Q][R];
#pragma unroll
    for (int p = 0; p < Q; ++p)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int c = lane + 32 * r, t = t0 + p * GW;
        v[p][r] = c < G && t < nk ? __ldcg(region + (size_t)t * GCTAS + c) : 0.0;
      }
    long long q[Q];
    int e[Q];
#pragma unroll
    for (int p = 0; p < Q; ++p) {
      e[p] = 0;
#pragma unroll
      for (int r = 0; r < R; ++r) e[p] = max(e[p], fix_exponent(v[p][r]));
      e[p] = __reduce_max_sync(0xffffffffu, e[p]);
      // |q| < 2^54 each, at most 160 of them
      q[p] = 0;
#pragma unroll
      for (int r = 0; r < R; ++r) q[p] += fix_word(v[p][r], e[p] + 3);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int p = 0; p < Q; ++p) q[p] += __shfl_xor_sync(0xffffffffu, q[p], o);
#pragma unroll
    for (int p = 0; p < Q; ++p)
      if (lane == p && t0 + p * GW < nk)
        out[t0 + p * GW] = e[p] == 0x7ff ? __longlong_as_double(0x7ff8000000000000LL)
                           : Small       ? fix_scale((double)q[p], e[p] - 1076, 0.0)
                                         : (double)q[p] * fix_pow2(e[p] - 1076);
  }
  __syncthreads();
}

// Coefficients c_t, t < k, against the own slices of the basis (FP64), for up to CE own elements from
// q0 on: per element one exponent for all c_t 2^(exponent of its slice of V_t).
template <int NB>
__device__ __forceinline__ void set_coefficients(GShared<NB, double>& sh, const double* c, int k, const int* Vexp,
                                                 size_t lde, int q0, int nel) {
  constexpr int CE = Rows<NB, double>::CE;
  if (q0 % CE != 0) return;
  const int n = min(CE, nel - q0);
  __syncthreads();
  if (threadIdx.x < CE) sh.ce[threadIdx.x] = 0;
  __syncthreads();
  for (int p = threadIdx.x; p < n * k; p += GALL) {
    const int el = p / k, t = p - el * k;
    const int ex = fix_exponent(c[t]), ev = Vexp[(size_t)t * lde + q0 + el];
    if (ex != 0 && ev != 0) atomicMax(&sh.ce[el], ex == 0x7ff || ev == 0x7ff ? (1 << 20) : ex + ev);
  }
  __syncthreads();
  for (int p = threadIdx.x; p < n * k; p += GALL) {
    const int el = p / k, t = p - el * k;
    const int ex = fix_exponent(c[t]), ev = Vexp[(size_t)t * lde + q0 + el];
    sh.cq[el * GM + t] = ex != 0 && ev != 0 ? fix_shift(c[t], sh.ce[el] - ex - ev) : Fix{0, 0};
  }
  __syncthreads();
}
template <int NB>
__device__ __forceinline__ void set_coefficients(GShared<NB, float>&, const double*, int, const int*, size_t, int,
                                                 int) {}

// sum_t c_t V_t at one own row (of own element el, word i of the own slices)
template <int NB>
__device__ __forceinline__ double combine(const GShared<NB, double>& sh, const double*, int k, const Fix* V,
                                          size_t ldv, int el, int i) {
  static_assert(GM <= kFixTerms, "the vectors of a cycle are one exact sum");
  FixDot acc;
  acc.clear();
  el %= Rows<NB, double>::CE;
  const Fix* c = sh.cq + el * GM;
  const Fix* p = V + i;
#pragma unroll 16
  for (int t = 0; t < k; ++t) acc.add(c[t], p[(size_t)t * ldv]);
  return acc.result(sh.ce[el], sh.ce[el] >= (1 << 20), 0.0);
}
template <int NB>
__device__ __forceinline__ float combine(const GShared<NB, float>&, const double* c, int k, const float* V,
                                         size_t ldv, int, int i) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  int t = 0;
  for (; t + 3 < k; t += 4) {
    const float* p = V + (size_t)t * ldv + i;
    s[0] += float(c[t]) * p[0];
    s[1] += float(c[t + 1]) * p[ldv];
    s[2] += float(c[t + 2]) * p[2 * ldv];
    s[3] += float(c[t + 3]) * p[3 * ldv];
  }
  for (; t < k; ++t) s[0] += float(c[t]) * V[(size_t)t * ldv + i];
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// word i of a basis slot
__device__ __forceinline__ double entry(const Fix* slot, const int* slot_e, int el, int i) {
  return fix_decode(slot[i], slot_e[el]);
}
__device__ __forceinline__ float entry(const float* slot, const int*, int, int i) { return slot[i]; }

// Givens update of column j (coefficients in coef, norm of the new vector from nrm2 and inv) by one
// warp.  The rotations carry one number through the column, carry_{i+1} = c_i h_{i+1} - s_i carry_i:
// a composition of affine maps, taken as a scan over the lanes (two columns each), 5 dependent steps
// instead of j (an FP64 operation takes 64 clocks).
template <int NB, class S>
__device__ __forceinline__ void givens(GShared<NB, S>& sh, int j, bool last) {
  const int lane = threadIdx.x & 31;
  double* col = sh.H + j * (j + 1) / 2;
  const double hn = sh.nrm2 * sh.inv;
  auto h = [&](int i) { return i <= j ? sh.coef[i] + (i == j ? 1.0 : 0.0) : 0.0; };
  double c[2], s[2], nx[2], b[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = 2 * lane + q;
    const bool on = i < j;
    c[q] = on ? sh.cs[i] : 0.0;
    s[q] = on ? sh.sn[i] : -1.0;  // the identity map beyond the column
    nx[q] = on ? h(i + 1) : 0.0;
    b[q] = c[q] * nx[q];
  }
  // inclusive scan of the lanes' maps x -> m x + t
  double m = s[0] * s[1], t = fma(-s[1], b[0], b[1]);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double pm = __shfl_up_sync(0xffffffffu, m, o), pt = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) {
      t = fma(m, pt, t);
      m *= pm;
    }
  }
  double pm = __shfl_up_sync(0xffffffffu, m, 1), pt = __shfl_up_sync(0xffffffffu, t, 1);
  if (lane == 0) {
    pm = 1.0;
    pt = 0.0;
  }
  const double c0 = h(0);
  const double x0 = fma(pm, c0, pt), x1 = fma(-s[0], x0, b[0]);
  if (2 * lane < j) col[2 * lane] = fma(c[0], x0, s[0] * nx[0]);
  if (2 * lane + 1 < j) col[2 * lane + 1] = fma(c[1], x1, s[1] * nx[1]);
  const double carry = fma(__shfl_sync(0xffffffffu, m, 31), c0, __shfl_sync(0xffffffffu, t, 31));
  if (lane == 0) {
    const double rr2 = fma(carry, carry, hn * hn);
    const double ir = rr2 > 0.0 ? rsqrt(rr2) : 0.0;
    const double cj = rr2 > 0.0 ? carry * ir : 1.0, sj = hn * ir;
    const double gj = sh.g[j], gn = -sj * gj;
    sh.cs[j] = cj;
    sh.sn[j] = sj;
    col[j] = rr2 * ir;
    sh.g[j + 1] = gn;
    sh.g[j] = cj * gj;
    int stop = 0;
    if (fabs(gn) <= sh.tol) stop = 1;
    if (hn == 0.0) stop = 2;
    if (!isfinite(hn) || !isfinite(gn)) stop = 4;
    if (stop == 0 && last) stop = 3;
    sh.stop = stop;
  }
}

// the kernel's arguments: as they are, or a copy whose exchange buffers are replaced
template <class S, int MODE>
struct ArgsOf {
  using T = const GArgs<S>&;
};
template <class S>
struct ArgsOf<S, kSingle> {
  using T = GArgs<S>;
};

// VS: the own slices of the basis lie in shared memory
template <int NB, class S, int MODE, bool VS>
__global__ void __launch_bounds__(GALL, 1) k_stage_gmres(const __grid_constant__ GArgs<S> args) {
  constexpr int ST = VS ? 3 : Rows<NB, S>::DEEP;
  __shared__ GShared<NB, S> sh;
  extern __shared__ __align__(16) unsigned char dyn[];
  typename ArgsOf<S, MODE>::T a = args;
  if (__ldcg(a.rec) != 0.0) return;  // an earlier solve of the sweep failed
  const int tid = threadIdx.x, G = gridDim.x, bi = blockIdx.x;
  const int wt = tid < GT ? tid : (1 << 30);  // first index of a worker's loop
  const int nR = a.nR, nI = a.ne - a.nR;
  const int r0 = (int)((long long)nR * bi / G), r1 = (int)((long long)nR * (bi + 1) / G);
  const int i0 = nR + (int)((long long)nI * bi / G), i1 = nR + (int)((long long)nI * (bi + 1) / G);
  const int nel = r1 - r0;
  const size_t nv = (size_t)nR * NB;
  constexpr int E = Rows<NB, S>::E;
  using W = typename Wire<S>::T;
  // own slices of the basis and their exponents: shared memory, or the slices of V itself
  const Ring<NB, S, ST> ring(dyn);
  W* const Vo = VS ? reinterpret_cast<W*>(dyn) + Ring<NB, S, ST>::WORDS : a.V + (size_t)r0 * NB;
  const size_t ldv = VS ? (size_t)a.own_max * NB : nv;
  int* const Ve = VS ? reinterpret_cast<int*>(Vo + (a.m + 1) * ldv) : a.Vexp + r0;
  const size_t lde = VS ? (size_t)a.own_max : (size_t)nR;
  if constexpr (MODE == kSingle) {
    // one CTA: the exchanged operand and the partials stay in shared memory behind the basis
    const size_t ve_words = sizeof(S) == 8 ? (a.m + 1) * lde + ((a.m + 1) * lde & 1) : 0;
    a.wire = reinterpret_cast<W*>(Ve + ve_words);
    a.wexp = reinterpret_cast<int*>(a.wire + (size_t)a.ne * NB);
  }
  Barrier<MODE> bar{a.bar, 0u, &sh.ok};
  // CTA partials, rs words from one output to the next
  constexpr int rs = MODE == kSingle ? 1 : GCTAS;
  double* const region0 = MODE == kSingle ? sh.single[0] : a.partial;
  double* const region1 = MODE == kSingle ? sh.single[1] : a.partial + (size_t)GLD * GCTAS;
  S* const yo = a.y + (size_t)r0 * NB;
  const Lane<NB> ln;
  const W* const rowI = first_row_of<NB, S>(a, i0, i1);
  const W* const rowR = first_row_of<NB, S>(a, r0, r1);
  auto wait = [&] { return bar.wait(); };
  auto idle = [] {};
  auto raw = [&](int pos, int row) { return a.b[(size_t)a.list[pos] * NB + row]; };
  auto rhs = [&](int pos, int row) {
    if constexpr (sizeof(S) == 8) return raw(pos, row) * fix_pow2(a.scale[row / (NB / 4)]);
    else return raw(pos, row);
  };
  // f(on, own element, word of the own slices) over passes of the own kept elements
  auto passes = [&](auto&& before, auto&& f) {
    for (int q = 0; q < nel; q += E) {
      before(q);
      f(ln.el < E && q + ln.el < nel, q + ln.el, (q + ln.el) * NB + slice_at<NB, VS>(ln.row));
    }
  };
  auto none = [](int) {};
  bool alive = true;
  bool guess = a.ywarm && a.warm;
  int total = 0, flag = 0, turn = 0;
  if (tid < 3 * E) sh.emax[tid / E][tid % E] = 0;
  __syncthreads();

  {
    const W* const start = guess ? rowI : rowR;
    ring.prime(start, start != nullptr);
  }
  // the initial guess (zero without one) to the exchanged operand
  passes(none, [&](bool on, int oe, int) {
    S v = S(0);
    if (on) {
      const int i = oe * NB + ln.row;
      if (guess) v = a.ywarm[(size_t)r0 * NB + i];
      yo[i] = v;
    }
    publish<NB, S, VS>(a, sh, turn, on, ln.el, ln.row, r0 + oe, v, true);
  });
  bar.arrive();
  for (bool first = true; alive; first = false) {
    // ---- residual of the reduced system: z = b_I - B_IR y, r = b_R - y - B_RR y - B_RI z
    if (guess) {
      alive = rows_product<NB, S, ST, MODE>(a, sh, ring, i0, i1, rowI, rowR, wait, idle, [&](bool on, int el, int row, int pos, S s) {
        publish<NB, S, VS>(a, sh, turn, on, el, row, pos, on ? rhs(pos, row) - s : S(0), true);
      });
    } else {
      alive = bar.wait();
      for (int q = i0; alive && q < i1; q += E) {
        const bool on = ln.el < E && q + ln.el < i1;
        publish<NB, S, VS>(a, sh, turn, on, ln.el, ln.row, q + ln.el, on ? rhs(q + ln.el, ln.row) : S(0), true);
      }
    }
    if (!alive) break;
    double bb = 0.0;
    if (first) {
      // |b|^2 over all own rows
      S s = S(0);
      for (int i = wt; i < (nel + i1 - i0) * NB; i += GT) {
        const int pos = i < nel * NB ? r0 + i / NB : i0 + i / NB - nel;
        const S v = raw(pos, i % NB);
        s += v * v;
      }
      S t[1] = {s};
      warp_reduce_scatter<1, S>(t, tid & 31);
      bb = (double)t[0];
    }
    bar.arrive();
    alive = rows_product<NB, S, ST, MODE>(a, sh, ring, r0, r1, rowR, rowI, wait, idle, [&](bool on, int el, int row, int pos, S s) {
      publish<NB, S, VS>(a, sh, turn, on, el, row, pos, on ? rhs(pos, row) - yo[(pos - r0) * NB + row] - s : S(0), false,
                     Vo, Ve, pos - r0);
    });
    if (!alive) break;
    if (first && (tid & 31) == 0 && tid < GT) sh.coef[tid >> 5] = bb;
    __syncthreads();
    if (first && tid == 0) {
      double s = 0.0;
      for (int w = 0; w < GW; ++w) s += sh.coef[w];
      region0[rs + bi] = s;
    }
    cta_dots<NB, VS, true>(Vo, Ve, a.scale, ldv, lde, 0, 0, nel, region0, rs, sh.dpart);
    bar.arrive();
    if (!(alive = bar.wait())) break;
    sum_partials<MODE, true>(first ? 2 : 1, region0, sh.red);
    if (tid == 0) {
      const double beta = sqrt(fmax(sh.red[0], 0.0));
      if (first) sh.tol = fmax(a.rtol * sqrt(fmax(sh.red[1], 0.0)), a.atol);
      sh.inv = beta > 0.0 ? 1.0 / beta : 0.0;
      sh.g[0] = beta;
      sh.stop = !isfinite(sh.red[0]) || (first && !isfinite(sh.red[1])) ? 4 : (beta <= sh.tol ? 1 : 0);
    }
    __syncthreads();
    flag = sh.stop;
    int k = 0;  // columns of this cycle
    if (flag == 0) {
      const S inv0 = S(sh.inv);
      passes(none, [&](bool on, int oe, int i) {
        publish<NB, S, VS>(a, sh, turn, on, ln.el, ln.row, r0 + oe, on ? entry(Vo, Ve, oe, i) * inv0 : S(0), true, Vo, Ve,
                       oe);
      });
      bar.arrive();
      bool ended = false;
      for (int j = 0; j < a.m; ++j) {
        W* const slot = Vo + (size_t)(j + 1) * ldv;   // w, then v_{j+1}
        int* const slot_e = Ve + (size_t)(j + 1) * lde;
        // ---- z = -B_IR v_j; the Givens update of the step before on the scalar warp meanwhile
        alive = rows_product<NB, S, ST, MODE>(
            a, sh, ring, i0, i1, rowI, rowR, wait,
            [&] {
              if (j > 0) givens<NB, S>(sh, j - 1, total + j >= a.maxit);
            },
            [&](bool on, int el, int row, int pos, S s) { publish<NB, S, VS>(a, sh, turn, on, el, row, pos, -s, true); });
        if (!alive) break;
        bar.arrive();
        // ---- w = B_RR v_j + B_RI z, unless the step before was the last
        bool stopped = false;
        alive = rows_product<NB, S, ST, MODE>(
            a, sh, ring, r0, r1, rowR, rowI,
            [&] {
              if (!bar.wait()) return false;
              if constexpr (MODE == kClusters) __syncthreads();
              stopped = j > 0 && sh.stop != 0;
              return !stopped;
            },
            idle, [&](bool on, int el, int row, int pos, S s) {
              publish<NB, S, VS>(a, sh, turn, on, el, row, pos, s, false, slot, slot_e, pos - r0);
            });
        if (stopped) {
          alive = ended = true;
          k = j;
          // the ring holds the rows of the product that is not taken
          ring.drain();
          ring.prime(rowI, rowI != nullptr);
          break;
        }
        if (!alive) break;
        k = j + 1;
        __syncthreads();
        // ---- projections and |w|^2
        cta_dots<NB, VS>(Vo, Ve, a.scale, ldv, lde, k, 0, nel, region1, rs, sh.dpart);
        bar.arrive();
        if (!(alive = bar.wait())) break;
        sum_partials<MODE>(k + 1, region1, sh.red);
        bool again = false;
        for (int pass = 0;; ++pass) {
          // coefficients so far, |h|^2 of this pass, and the norm it leaves
          if (tid < 32) {
            double s = 0.0;
            for (int t = tid; t < k; t += 32) {
              const double h = sh.red[t];
              sh.coef[t] = pass == 0 ? h : sh.coef[t] + h;
              s += h * h;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (tid == 0) {
              const double w2 = sh.red[k], n2 = w2 - s;
              sh.need = !(s <= 0.5 * w2);
              sh.nrm2 = fmax(n2, 0.0);
              sh.inv = n2 > 0.0 ? rsqrt(n2) : (isfinite(n2) ? 0.0 : n2);
            }
          }
          __syncthreads();
          // more than half of |w|^2 cancelled: the projections are taken once more from what is left
          // (and the norm from a sum of its own should that cancel again)
          again = sh.need != 0 && pass < 2;
          if (!again) break;
          passes([&](int q) { set_coefficients<NB>(sh, sh.red, k, Ve, lde, q, nel); },
                 [&](bool on, int oe, int i) {
                   const S s = on && pass < 2 ? entry(slot, slot_e, oe, i) - combine<NB>(sh, sh.red, k, Vo, ldv, oe, i)
                                              : S(0);
                   publish<NB, S, VS>(a, sh, turn, on, ln.el, ln.row, r0 + oe, s, false, slot, slot_e, oe);
                 });
          __syncthreads();
          double* region = pass == 0 ? region0 : region1;
          if (pass == 0) cta_dots<NB, VS>(Vo, Ve, a.scale, ldv, lde, k, 0, nel, region, rs, sh.dpart);
          else cta_dots<NB, VS>(Vo, Ve, a.scale, ldv, lde, k, k, nel, region + (size_t)k * rs, rs, sh.dpart);
          bar.arrive();
          if (!(alive = bar.wait())) break;
          if (pass == 0) {
            sum_partials<MODE>(k + 1, region, sh.red);
          } else {
            for (int t = wt; t < k; t += GT) sh.red[t] = 0.0;
            sum_partials<MODE>(1, region + (size_t)k * rs, sh.red + k);
          }
        }
        if (!alive) break;
        // ---- v_{j+1} = (w - V h) / |w - V h| with the last pass's h
        const S inv = S(sh.inv);
        passes([&](int q) { set_coefficients<NB>(sh, sh.red, k, Ve, lde, q, nel); },
               [&](bool on, int oe, int i) {
                 const S s = on ? (entry(slot, slot_e, oe, i) - combine<NB>(sh, sh.red, k, Vo, ldv, oe, i)) * inv
                                : S(0);
                 publish<NB, S, VS>(a, sh, turn, on, ln.el, ln.row, r0 + oe, s, true, slot, slot_e, oe);
               });
        bar.arrive();
      }
      if (!alive) break;
      if (!ended) {
        // a full cycle: its last column is still to be rotated (and its barrier to be waited for)
        if (!(alive = bar.wait())) break;
        if (tid >= GT) givens<NB, S>(sh, k - 1, total + k >= a.maxit);
      }
      __syncthreads();
      flag = sh.stop;
      total += k;
    }
    if (flag == 4) break;
    // ---- y_R += V c, c = H^{-1} g (one warp, column oriented)
    __syncthreads();
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
    passes([&](int q) { set_coefficients<NB>(sh, sh.coef, k, Ve, lde, q, nel); },
           [&](bool on, int oe, int i) {
             S s = S(0);
             if (on) {
               const int r = oe * NB + ln.row;
               s = yo[r] + combine<NB>(sh, sh.coef, k, Vo, ldv, oe, i);
               yo[r] = s;
               if (a.ywarm) a.ywarm[(size_t)r0 * NB + r] = s;
             }
             publish<NB, S, VS>(a, sh, turn, on, ln.el, ln.row, r0 + oe, s, true);
           });
    bar.arrive();
    guess = true;
    if (flag != 0 || total >= a.maxit) break;
  }
  if (alive && flag != 4) {
    // ---- y_I = b_I - B_IR y_R, then x = D y element by element
    alive = rows_product<NB, S, ST, MODE>(a, sh, ring, i0, i1, rowI, nullptr, wait, idle, [&](bool on, int, int row, int pos, S s) {
      if (on) a.y[(size_t)pos * NB + row] = rhs(pos, row) - s;
    });
  }
  ring.drain();
  if (alive && flag != 4) {
    S* ys = reinterpret_cast<S*>(sh.xs[0]);
    const int nown = nel + (i1 - i0);
    for (int q0 = 0; q0 < nown; q0 += E) {
      __syncthreads();
      for (int idx = wt; idx < E * NB && q0 + idx / NB < nown; idx += GT) {
        const int q = q0 + idx / NB, pos = q < nel ? r0 + q : i0 + q - nel;
        S y = a.y[(size_t)pos * NB + idx % NB];
        if constexpr (sizeof(S) == 8) y *= fix_pow2(-a.scale[idx % NB / (NB / 4)]);
        ys[idx] = y;
      }
      __syncthreads();
      if (ln.el < E && q0 + ln.el < nown) {
        const int q = q0 + ln.el, pos = q < nel ? r0 + q : i0 + q - nel;
        const size_t e = a.list[pos];
        const S* d = a.D + e * (NB * NB) + (size_t)ln.row * a.d_row;
        S acc[4] = {S(0), S(0), S(0), S(0)};
#pragma unroll(NB % 20 == 0 ? 20 : 12)
        for (int c = 0; c < NB; ++c) acc[c & 3] += __ldg(d + (size_t)c * a.d_col) * ys[ln.el * NB + c];
        a.x[e * NB + ln.row] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
      }
    }
  }
  if (tid == 0) {
    if (bi == 0) a.rec[1] += (double)total;
    // codes are positive doubles, which order as their bits do
    if (const int code = solve_code(alive, flag, a.need_conv != 0, bi == 0))
      atomicMax(reinterpret_cast<unsigned long long*>(a.rec), (unsigned long long)__double_as_longlong((double)code));
  }
  if (alive) bar.leave();
}

struct GSetup {
  cudaError_t err = cudaSuccess;
  int sms = 0;
  int dyn[4] = {0, 0, 0, 0};  // dynamic shared memory of the four variants
};

template <int NB, class S>
cudaError_t launch_gmres(GArgs<S>& a, cudaStream_t st) {
  const void* const kernels[4] = {(const void*)k_stage_gmres<NB, S, kGrid, true>,
                                  (const void*)k_stage_gmres<NB, S, kGrid, false>,
                                  (const void*)k_stage_gmres<NB, S, kClusters, true>,
                                  (const void*)k_stage_gmres<NB, S, kSingle, true>};
  // one device per process (see pp_create); thread-safe static initialization
  static const GSetup setup = [&] {
    GSetup s;
    int dev = 0;
    s.err = cudaGetDevice(&dev);
    if (s.err == cudaSuccess) s.err = cudaDeviceGetAttribute(&s.sms, cudaDevAttrMultiProcessorCount, dev);
    for (int k = 0; k < 4; ++k) {
      cudaFuncAttributes at;
      if (s.err == cudaSuccess) s.err = cudaFuncGetAttributes(&at, kernels[k]);
      if (s.err != cudaSuccess) break;
      s.dyn[k] = kSmemMax - (int)at.sharedSizeBytes;
      s.err = cudaFuncSetAttribute(kernels[k], cudaFuncAttributeMaxDynamicSharedMemorySize, s.dyn[k]);
    }
    return s;
  }();
  if (setup.err != cudaSuccess) return setup.err;
  const size_t short_bytes = sizeof(S) * Ring<NB, S, 3>::WORDS, deep_bytes = sizeof(S) * Ring<NB, S, Rows<NB, S>::DEEP>::WORDS;
  // the short ring and the basis slices of `own` elements
  auto basis_bytes = [&](int own) {
    return short_bytes + (size_t)(a.m + 1) * own * (sizeof(S) * NB + (sizeof(S) == 8 ? sizeof(int) : 0)) + 8;
  };
  // One CTA while the kept rows are one pass and everything fits its shared memory: a step then has no
  // barrier but the CTA's own (32 triangles, p = 1: 11.6 us a step against 13.0 us with the cluster; 64
  // triangles would take two passes, 15.1 us against 11.9 us).  A cluster of 8 up to kClusterRows, one
  // pass each.  Otherwise all SMs, the basis beside the short ring when both fit, else the deep ring.
  const size_t single_bytes = basis_bytes(a.nR) + (size_t)a.ne * (sizeof(S) * NB + sizeof(int));
  const int cl_own = (a.nR + kCluster - 1) / kCluster;
  int k, G;
  if (a.nR <= Rows<NB, S>::E && single_bytes <= (size_t)setup.dyn[3]) {
    k = 3;
    G = 1;
  } else if ((int64_t)a.nR * NB <= kClusterRows && basis_bytes(cl_own) <= (size_t)setup.dyn[2]) {
    k = 2;
    G = kCluster;
  } else {
    G = std::min(std::min(setup.sms, GCTAS), a.nR);
    k = basis_bytes((a.nR + G - 1) / G) <= (size_t)setup.dyn[0] ? 0 : 1;
  }
  a.own_max = (a.nR + G - 1) / G;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(GALL);
  cfg.dynamicSmemBytes = k == 3 ? single_bytes : k == 1 ? deep_bytes : basis_bytes(a.own_max);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = k == 2 ? cudaLaunchAttributeClusterDimension : cudaLaunchAttributeCooperative;
  if (k == 2) {
    at.val.clusterDim.x = kCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
  } else {
    at.val.cooperative = 1;
  }
  cfg.attrs = &at;
  cfg.numAttrs = k == 3 ? 0 : 1;
  void* params[] = {&a};
  return cudaLaunchKernelExC(&cfg, kernels[k], params);
}

}  // namespace

template <class S>
cudaError_t launch_stage_gmres(const DevMesh& m, int nb, const StageGmres<S>& q, cudaStream_t st) {
  if (q.m < 1 || q.m > GM || m.n_kept < 1) return cudaErrorInvalidValue;
  ProfScope ps(sizeof(S) == 8 ? PP_K_STAGE_GMRES : PP_K_STAGE_GMRES32, st);
  using W = typename Wire<S>::T;
  GArgs<S> a{};
  a.ne = m.ne;
  a.nR = m.n_kept;
  a.list = m.order;
  a.src = m.order_nbr;
  a.B = reinterpret_cast<const W*>(q.B);
  a.Bexp = q.Bexp;
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
  a.V = reinterpret_cast<W*>(q.V);
  a.Vexp = q.wexp + m.ne;
  a.y = q.y;
  a.wire = reinterpret_cast<W*>(q.wire);
  a.wexp = q.wexp;
  a.partial = q.partial;
  a.bar = q.bar;
  a.rec = q.rec;
  a.scale = q.scale;
  switch (nb) {
    case 12: return launch_gmres<12, S>(a, st);
    case 24: return launch_gmres<24, S>(a, st);
    case 40: return launch_gmres<40, S>(a, st);
    case 60: return launch_gmres<60, S>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pp
