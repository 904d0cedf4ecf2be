// How a one-launch stage solve ends, as the code that stays in its record (rec[0]).
#pragma once

#ifdef __CUDACC__
#define PP_SR_HD __host__ __device__
#else
#define PP_SR_HD
#endif

namespace pp {

constexpr int kSolveOk = 0, kSolveCap = 1, kSolveNonFinite = 4, kSolveBarrier = 8;

// The code that one CTA reports; the record keeps the largest.  Every CTA whose barrier wait expired
// reports that itself: the others need not notice (at the last barrier a late CTA can still arrive in
// time for all but one, which then leaves its rows of x unwritten and the barrier count standing).  What
// all CTAs know alike, the first one reports.  flag: 0 restart, 1 converged, 2 breakdown, 3 cap, 4 non-finite.
PP_SR_HD inline int solve_code(bool alive, int flag, bool need_conv, bool first_cta) {
  if (!alive) return kSolveBarrier;
  if (!first_cta) return kSolveOk;
  if (flag == 4) return kSolveNonFinite;
  return need_conv && flag != 1 && flag != 2 ? kSolveCap : kSolveOk;
}

}  // namespace pp
