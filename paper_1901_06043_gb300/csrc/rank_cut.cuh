// Rank cut of Eq. Un on n descending eigenvalues, by one CTA of RANK_CUT_NT
// threads: R = min{R in 1..n : tail(R) <= thr}, tail(R) = sum_{i >= R} w_i summed
// in FP64 from the smallest eigenvalue up, one after the other (the order fixes
// the rounding, and with thr = 0 the cut); fixed_R > 0: R = fixed_R.  The chain of
// additions is one thread's (~64 cycles each); loads, stores and comparisons
// are the others'.  (One thread for everything: 21 us at n = 200, 122 us at
// n = 1500.)
#pragma once
#include <cstdint>

namespace tk {

constexpr int RANK_CUT_NT = 128;

__device__ __forceinline__ void rank_cut_cta(const double* __restrict__ w, int n, double thr,
                                             int fixed_R, int64_t* out_R, double* out_d) {
  constexpr int CH = 1024;
  __shared__ double s_t[CH];
  __shared__ int s_best;
  __shared__ double s_tail;
  if (threadIdx.x == 0) { s_best = fixed_R > 0 ? fixed_R : n; s_tail = 0.0; }
  double t = 0.0;                                   // thread 0: tail of the last chunk
  for (int hi = n; hi > 0; hi -= CH) {              // s_t[k]: w, then the tail, of index lo + k
    const int lo = hi > CH ? hi - CH : 0;
    __syncthreads();
    for (int k = threadIdx.x; k < hi - lo; k += RANK_CUT_NT) s_t[k] = w[lo + k];
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll 8
      for (int k = hi - lo - 1; k >= 0; --k) {
        t += s_t[k];
        s_t[k] = t;
      }
    }
    __syncthreads();
    if (fixed_R > 0) {
      if (threadIdx.x == 0 && fixed_R >= lo && fixed_R < hi) s_tail = s_t[fixed_R - lo];
      continue;
    }
    int best = n;
    for (int k = threadIdx.x; k < hi - lo; k += RANK_CUT_NT)
      if (lo + k >= 1 && s_t[k] <= thr) { best = lo + k; break; }
    if (best < n) atomicMin(&s_best, best);
    __syncthreads();
    if (threadIdx.x == 0 && s_best >= lo && s_best < hi) s_tail = s_t[s_best - lo];
  }
  if (threadIdx.x == 0) {
    *out_R = s_best;
    *out_d = s_tail;
  }
}

}  // namespace tk
