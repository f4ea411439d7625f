// FP64 symmetric eigensolver for the truncation step of ST-HOSVD (Section
// 5.2 computes the eigenpairs of the I_n x I_n Gram matrix with LAPACK's
// syev, whose first stage is a Householder reduction to tridiagonal form).
// Only what Algorithm 1 consumes is computed: all eigenvalues (the rank cut
// of Eq. Un sums their tail) and the leading R eigenvectors (U_n).
//
//   1. Householder tridiagonalization  Q^T S Q = T          (k_tridiag)
//   2. all eigenvalues of T by bisection on Sturm counts    (k_bisect)
//   3. the rank cut (k_rank_cut of jacobi.cu)
//   4. eigenvectors of T for the leading R eigenvalues by
//      inverse iteration                                     (k_invit)
//   5. their Cholesky QR in descending eigenvalue order, two passes:
//      Gram (gram kernels), L^-1 and Z L^-T           (k_chol_*, k_apply_*)
//   6. back-transformation U = Q Z                           (k_backtransform)
//
// Every stage is FP64.  Work is ~(4/3) n^3 for stage 1 and O(n^2 R) for the
// rest, against ~4 n^3 per sweep (matrix plus vectors) of a cyclic Jacobi
// method, which needs ~15 sweeps on the graded Gram matrices of a Tucker
// tensor; on this part FP64 runs at 1/64 of the FP32 rate, so the FP64
// operation count decides.
//
// Stage 1 runs on a team of CTAs: the whole grid (one matrix) or a share of it
// (batched matrices), a cooperative launch.  Rows are owned cyclically (row i by
// team rank i mod G), so each CTA keeps a balanced share of the shrinking
// trailing matrix.  Step k (reflector H_k = I - tau_k v_k v_k^T on indices
// k+1..n-1) needs p_k = tau_k A v_k (rows spread over the team) and the next
// pivot row r = A[k+1][:], both published by the rows' owners; every CTA then forms
// v_{k+1} itself and, in one pass over its own rows, applies step k's update
// A <- A - v_k w_k^T - w_k v_k^T, w = p - (tau/2)(p . v) v, and its part of
// A v_{k+1}.
//   A step is a chain of latencies (an FP64 instruction takes 64 cycles, and a
// warp's occupies its sub-partition's pipe for as long), so the chain is kept
// short:
// - No barrier up to kTridiagWordsMax.  Every published value is a 16-byte word {value, step}, written
//   and read by single 128-bit accesses; a reader polls the word until it
//   carries the step it waits for.  Two buffers in turn: a CTA publishes for
//   step k+1 only after all its threads have read step k.  (A grid barrier and
//   then the loads: two more round trips to L2 per step.)
// - Short sums: warp_sum adds in integers.  (Forming the norm of the next pivot
//   row from sums taken together with p . v, one reduction less, cancels in
//   most steps of a graded matrix: not kept.)
// - Unscaled reflectors: v = x - beta e_1, tau = 2 / (v . v).  One warp computes beta,
//   v's first entry and tau while the others form A x without its first column;
//   p = tau (the sums + v_1 the first column) follows.  (The
//   matrix is scaled by a power of two first, so that squares neither overflow
//   nor underflow where they matter.)  The update goes by w, though a_ij - v_i p_j -
//   (p_i - tau (p . v) v_i) v_j needs one FMA less on the chain: its first product
//   is larger, and the vectors of close eigenvalues came out 1.3 times as far off.
// Measured, whole reduction: n = 50 0.26 -> 0.16 ms, n = 200 1.20 -> 0.74 ms, n = 500
// 3.48 -> 2.62 ms, n = 1500 18.2 -> 16.2 ms (a barrier, normalized reflectors and FP64
// sums before; 0.81, 2.77 and 17.3 with the reflector ahead of A v).
#include <algorithm>
#include <cfloat>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "rank_cut.cuh"

namespace tk {
namespace {

constexpr int TNT = 256;            // threads per CTA of k_tridiag / k_chol_*
constexpr int TNW = TNT / 32;

__device__ __forceinline__ double warp_sum_fp64(double v) {
  // xor butterfly: every lane adds the same two operands at every level
  // (addition commutes exactly), so all lanes end with the same value
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the warp, the same in every lane: the values as 58-bit fixed point
// under the largest exponent E of the warp (bits below 2^-57 of 2^E are
// dropped, a 32nd of the largest value's last bit each), split into three
// fields that redux.sync adds in integers, and the exact sum rounded to FP64
// once.  ~230 cycles; five FP64 additions with their shuffles take ~1,000 and a
// share of the FP64 pipe.  Exponents near the ends of the range, Inf and NaN
// take those.
__device__ __forceinline__ double warp_sum(double v) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  const int E = __reduce_max_sync(0xffffffffu, e);
  if (E < 70 || E > 2040) {
    if (E == 0) return __reduce_or_sync(0xffffffffu, (unsigned)__double2loint(v) | (unsigned)(hi & 0xfffff)) == 0u
                           ? 0.0 : warp_sum_fp64(v);
    return warp_sum_fp64(v);
  }
  const unsigned lo = (unsigned)__double2loint(v);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;     // (a zero or denormal v: shifted out)
  unsigned long long q;
  asm("{\n .reg .u64 m;\n mov.b64 m, {%1, %2};\n shr.u64 %0, m, %3;\n}"
      : "=l"(q) : "r"(lo << 5), "r"((mh << 5) | (lo >> 27)), "r"(E - e));
  const long long n = (long long)(hi >> 31);
  const long long s = (long long)((q ^ (unsigned long long)n)) - n;
  const unsigned L = __reduce_add_sync(0xffffffffu, (unsigned)s & 0xfffffu);
  const unsigned M = __reduce_add_sync(0xffffffffu, (unsigned)(s >> 20) & 0xfffffu);
  const int H = __reduce_add_sync(0xffffffffu, (int)(s >> 40));
  const long long S = ((long long)H << 40) + ((long long)M << 20) + (long long)L;
  if (S == 0) return 0.0;
  unsigned long long a = (unsigned long long)(S < 0 ? -S : S);
  const int z = __clzll((long long)a);
  a <<= z;
  const unsigned long long mant = (a >> 11) + ((a >> 10) & 1ull);
  const unsigned long long r = ((unsigned long long)(E + 5 - z) << 52) + mant;   // exponent field E + 6 - z
  return __longlong_as_double((long long)(r | (S < 0 ? 1ull << 63 : 0ull)));
}

// FP64 instructions occupy a sub-partition's FP64 pipe for ~64 cycles per
// warp whatever they compute, so scalar work that every thread needs is done
// by warp 0 and broadcast through shared memory.

// 1/x for a normal x with |x| in [2^-1000, 2^1000]: the FP32 reciprocal of
// x's mantissa (moved into FP32 by integer operations), rescaled by the
// exponent, then two Newton-Raphson steps.
__device__ __forceinline__ double rcp64(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex < 24 || ex > 2022) return 1.0 / x;
  const float mf = __uint_as_float(0x3f800000u | (unsigned)((b >> 29) & 0x7fffff));   // [1, 2)
  float rf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(mf));                              // (0.5, 1]
  const unsigned rb = __float_as_uint(rf);
  const int re = (int)((rb >> 23) & 0xff) - 127 + 1023 - (ex - 1023);
  double r = __longlong_as_double((long long)((b >> 63) << 63 | (unsigned long long)re << 52 |
                                              (unsigned long long)(rb & 0x7fffff) << 29));
  double e = fma(-x, r, 1.0);
  r = fma(r, e, r);
  e = fma(-x, r, 1.0);
  return fma(r, e, r);
}

// sqrt(x) for x in [2^-1000, 2^1000]: an FP32 estimate of 1 / sqrt of x's mantissa
// (exponent made even), then Goldschmidt's iteration on g ~ sqrt(x), h ~ 1 / (2
// sqrt(x)) and one correction by the residual x - g^2.
__device__ __forceinline__ double sqrt64(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff) - 1023, odd = e & 1;
  const float mf = __uint_as_float((unsigned)(127 + odd) << 23 | (unsigned)((b >> 29) & 0x7fffff));
  float rf;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(mf));          // (0.5, 1]
  const unsigned rb = __float_as_uint(rf);
  const int re = (int)(rb >> 23) - 127 + 1023 - (e - odd) / 2;
  const double y = __longlong_as_double((long long)((unsigned long long)re << 52 |
                                                    (unsigned long long)(rb & 0x7fffff) << 29));
  double g = x * y, h = 0.5 * y;
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  return fma(fma(-g, g, x), h, g);
}

// A value published for a step, and its step number.
__device__ __forceinline__ void put_word(ulonglong2* p, double v, unsigned long long step) {
  asm volatile(
      "{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(p),
      "l"(__double_as_longlong(v)), "l"(step)
      : "memory");
}
__device__ __forceinline__ double get_word(const ulonglong2* p, unsigned long long& step) {
  long long v;
  asm volatile(
      "{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}"
      : "=l"(v), "=l"(step) : "l"(p) : "memory");
  return __longlong_as_double(v);
}

}  // namespace

// ---------------------------------------------------------------- stage 1
// Largest n whose team exchanges words; above, plain values and a barrier.  Whole
// solves, words and barrier: n = 200 2.04 and 2.15 ms, n = 500 5.58 and 5.63, n = 800
// 10.54 and 10.18, n = 1500 33.5 and 29.3.
constexpr int kTridiagWordsMax = 640;

// A copy of S (one problem; NULL: A holds the matrix) and the largest biased
// exponent of A's entries, into info[2].
__global__ void __launch_bounds__(TNT) k_eig_load(const EigProblem* probs, const double* S) {
  const EigProblem P = probs[blockIdx.y];
  const int64_t nn = (int64_t)P.n * P.n;
  int m = 0;
  for (int64_t e = (int64_t)blockIdx.x * TNT + threadIdx.x; e < nn; e += (int64_t)gridDim.x * TNT) {
    const double v = S ? S[e] : P.A[e];
    if (S) P.A[e] = v;
    m = max(m, (__double2hiint(v) >> 20) & 0x7ff);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(P.info + 2, m);
}

// One team of P.team_size CTAs per problem (teams back to back in the grid); a
// team of one exchanges through its shared memory.  P.srows: the CTA's own
// rows live in shared memory; otherwise they are read and written in place in
// A (L2-resident).  v_k goes into row k of V, columns k+1.. .
__global__ void __launch_bounds__(TNT, 1) k_tridiag(const EigProblem* probs, int count,
                                                    unsigned* err, unsigned long long poll_limit) {
  extern __shared__ __align__(16) double tsm[];
  __shared__ double s_red[2][TNW], s_c[4], s_tau;
  int pidx = 0;
  while (pidx + 1 < count && probs[pidx + 1].team_off <= (int)blockIdx.x) ++pidx;
  const EigProblem P = probs[pidx];
  const int n = P.n;
  const int G = P.team_size;
  const int c = (int)blockIdx.x - P.team_off;
  if (c < 0 || c >= G) return;
  const bool SROWS = P.srows != 0, solo = G == 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double* A = P.A;
  ulonglong2* const xp = reinterpret_cast<ulonglong2*>(P.xch);   // p: 2 x n words
  ulonglong2* const xr = xp + 2 * (size_t)n;                     // next pivot row: 2 x n words
  // long rows: plain values behind a barrier of the team
  const bool plain = n > kTridiagWordsMax;
  double* const dp = P.xch;               // p: 2 x n
  double* const dr = dp + 2 * (size_t)n;  // next pivot row: 2 x n
  const GridBarrier bar{reinterpret_cast<unsigned*>(P.xch + 8 * (size_t)n), nullptr, err};
  unsigned gen = 0;
  double* vk = tsm;                       // v_k by global index
  double* vn = tsm + n;                   // the pivot row, then v_{k+1}
  double* sp = tsm + 2 * n;               // p_k, then w_k
  // own rows t = 0, 1, ... (row c + G t): A x without the first column (solo: then
  // p_{k+1}), the first column
  const int nown = (n + G - 1) / G;
  double* sq = tsm + 3 * n;
  double* const sa = sq + nown;
  double* const sr = sa + nown;           // solo: next pivot row
  double* const srows = sr + (solo ? n : 0);   // the own rows when SROWS
  auto row = [&](int i) -> double* {
    return SROWS ? srows + (size_t)((i - c) / G) * n : A + (int64_t)i * n;
  };

  if (n <= 2) {
    if (c == 0 && tid == 0) {
      P.d[0] = A[0];
      if (n == 2) { P.e[0] = A[1]; P.d[1] = A[3]; }
    }
    return;
  }
  // entries scaled by sc = 2^-floor(log2 max|a|) (1 for a zero or non-finite matrix)
  const int mexp = P.info[2];
  const bool scaled = mexp > 0 && mexp < 0x7ff;
  const int dex = scaled ? max(-1022, min(1022, mexp - 1023)) : 0;
  const double sc = __longlong_as_double((long long)(1023 - dex) << 52);
  const double isc = __longlong_as_double((long long)(1023 + dex) << 52);
  for (int i = c; i < n; i += G) {
    if (i == 0) continue;                 // row 0 is read as it is, below
    const double* src = A + (int64_t)i * n;
    double* dst = row(i);
    for (int j = tid; j < n; j += TNT) dst[j] = src[j] * sc;
  }

  // By the last warp, with the row x in vn[lo..] and the partial sums of
  // |x[lo+1..]|^2 in s_red[1]: beta into s_c[2], v = x - beta e_lo (its first entry
  // into vn[lo] and s_c[3]), 2 / (v . v) into s_tau; a zero (or negligible) rest: no
  // reflector, tau = 0.
  auto reflector = [&](int lo) {
    const double ss = warp_sum(lane < TNW ? s_red[1][lane] : 0.0);
    const double alpha = vn[lo], tot = fma(alpha, alpha, ss);
    __syncwarp();
    double be = alpha, v1 = 1.0;
    const bool on = !(ss == 0.0) && !(tot < 0x1p-900);
    if (on) {
      const double g = sqrt64(tot);
      be = alpha > 0.0 ? -g : g;
      v1 = alpha - be;
    }
    const double t = on ? 2.0 * rcp64(fma(v1, v1, ss)) : 0.0;
    if (lane == 0) { s_c[2] = be; s_c[3] = v1; s_tau = t; vn[lo] = v1; }
  };
  // ---- v_0 from row 0
  {
    double ss = 0.0;
    for (int j = 1 + tid; j < n; j += TNT) {
      const double a = A[j] * sc;
      vn[j] = a;
      if (j >= 2) ss = fma(a, a, ss);
    }
    ss = warp_sum(ss);
    if (lane == 0) s_red[1][warp] = ss;
  }
  // Largest own row.  A CTA without rows in the trailing matrix publishes nothing,
  // so nobody would wait until it has read its words: it leaves.  Results of a
  // step are written by the owner of row lo, which is still there.
  const int last = n - 1 - (n - 1 - c) % G;

  int i0 = c > 0 ? c : G, t0 = c > 0 ? 0 : 1;   // smallest own row of the trailing matrix, and where it is
  double* own0 = row(i0 < n ? i0 : c);
  const int64_t rstep = SROWS ? n : (int64_t)G * n;               // to the next own row
  double tau = 0.0;
  for (int k = -1; k <= n - 3; ++k) {
    const int lo = k + 2;                 // first row and column of the trailing matrix after step k
    if (k >= 0 && last < lo && !plain) return;        // (a barrier counts every CTA)
    const bool more = k < n - 3;
    if (i0 < lo) { i0 += G; ++t0; own0 += rstep; }
    const bool scribe = i0 == lo;
    if (k >= 0) {
      // ---- p_k into sp and the pivot row r into vn; p . v
      const double v1 = vk[k + 1];
      double s1 = 0.0;
      bool fail = false;
      const unsigned long long want = (unsigned long long)k + 1ull;
      const ulonglong2* pw = xp + (size_t)(k & 1) * n;
      const ulonglong2* rw = xr + (size_t)(k & 1) * n;
      constexpr int JPT = 4;              // entries in flight per thread and array
      for (int j0 = k + 1 + tid; j0 < n; j0 += JPT * TNT) {
        double pj[JPT], rj[JPT];
        if (solo) {
#pragma unroll
          for (int q = 0; q < JPT; ++q) {
            const int j = j0 + q * TNT;
            pj[q] = j < n ? sp[j] : 0.0;
            rj[q] = j < n ? sr[j] : 0.0;
          }
        } else if (plain) {
#pragma unroll
          for (int q = 0; q < JPT; ++q) {
            const int j = j0 + q * TNT;
            pj[q] = j < n ? __ldcg(dp + (size_t)(k & 1) * n + j) : 0.0;
            rj[q] = j < n ? __ldcg(dr + (size_t)(k & 1) * n + j) : 0.0;
            if (j < n) sp[j] = pj[q];
          }
        } else {
          unsigned long long tp[JPT], tr[JPT];
#pragma unroll
          for (int q = 0; q < JPT; ++q) {
            const int j = j0 + q * TNT;
            tp[q] = tr[q] = want;
            pj[q] = rj[q] = 0.0;
            if (j < n) { pj[q] = get_word(pw + j, tp[q]); rj[q] = get_word(rw + j, tr[q]); }
          }
          unsigned long long it = 0;
#pragma unroll
          for (int q = 0; q < JPT; ++q) {
            const int j = j0 + q * TNT;
            while (tp[q] != want || tr[q] != want) {
              if (++it >= poll_limit) { atomicOr(err, DEV_ERR_BARRIER_TIMEOUT); fail = true; break; }
              if ((it & 1023) == 0 && (ld_acquire_u32(err) & DEV_ERR_BARRIER_TIMEOUT)) { fail = true; break; }
              if (it > 4096) __nanosleep(64);
              if (tp[q] != want) pj[q] = get_word(pw + j, tp[q]);
              if (tr[q] != want) rj[q] = get_word(rw + j, tr[q]);
            }
            if (fail) break;
            if (j < n) sp[j] = pj[q];
          }
        }
        if (fail) break;
#pragma unroll
        for (int q = 0; q < JPT; ++q) {
          const int j = j0 + q * TNT;
          if (j < n) {
            vn[j] = rj[q];
            s1 = fma(pj[q], vk[j], s1);
          }
        }
      }
      s1 = warp_sum(s1);
      if (lane == 0) s_red[0][warp] = s1;
      if (__syncthreads_or(fail)) return;
      // the last warp does the scalars (it has no rows, see below)
      if (warp == TNW - 1) {
        const double K = 0.5 * tau * warp_sum(lane < TNW ? s_red[0][lane] : 0.0);
        if (lane == 0) {
          s_c[0] = K;
          s_c[1] = fma(-K, v1, sp[k + 1]);
        }
      }
      __syncthreads();
      const double K = s_c[0], w1 = s_c[1];
      if (scribe && tid == 0) {
        P.d[k + 1] = fma(-w1, v1, fma(-v1, w1, vn[k + 1])) * isc;
        if (!more) {                      // the last off-diagonal and the last entry (lo = n - 1)
          const double vl = vk[lo], wl = fma(-K, vl, sp[lo]);
          P.e[n - 2] = fma(-w1, vl, fma(-v1, wl, vn[lo])) * isc;
          P.d[lo] = fma(-wl, vl, fma(-vl, wl, own0[lo])) * isc;
        }
      }
      if (more) {
        // w_k into sp, the pivot row x after step k, and its norm
        double ss = 0.0;
        for (int j = lo + tid; j < n; j += TNT) {
          const double v = vk[j], w = fma(-K, v, sp[j]);
          const double x = fma(-w1, v, fma(-v1, w, vn[j]));
          sp[j] = w;
          vn[j] = x;
          if (j > lo) ss = fma(x, x, ss);
        }
        ss = warp_sum(ss);
        if (lane == 0) s_red[1][warp] = ss;
      }
    }
    if (!more) break;
    __syncthreads();                      // x is complete
    if (k < 0 && c == 0 && tid == 0) P.d[0] = A[0];
    // ---- own rows: the update of step k and A x without its first column; v and tau
    // by the last warp meanwhile
    if (warp == TNW - 1) {
      reflector(lo);
    } else {
      constexpr int nw = TNW - 1;
      ulonglong2* rw = xr + (size_t)((k + 1) & 1) * n;
      // PIV: the next pivot row, also published
      auto do_row = [&](int i, int t, double* Ai, auto UPD, auto PIV) {
        double vi = 0.0, wi = 0.0, acc = 0.0, alo = 0.0;
        if constexpr (decltype(UPD)::value) {
          vi = vk[i];
          wi = sp[i];
        }
#pragma unroll 4
        for (int j = lo + lane; j < n; j += 32) {
          double a = Ai[j];
          if constexpr (decltype(UPD)::value) {
            a = fma(-wi, vk[j], fma(-vi, sp[j], a));
            Ai[j] = a;
          }
          if constexpr (decltype(PIV)::value) {
            if (solo) sr[j] = a;
            else if (plain) dr[(size_t)((k + 1) & 1) * n + j] = a;
            else put_word(rw + j, a, (unsigned long long)k + 2ull);
          }
          if (j == lo) alo = a;
          acc = fma(a, j == lo ? 0.0 : vn[j], acc);       // (vn[lo] is being replaced)
        }
        acc = warp_sum(acc);
        if (lane == 0) { sq[t] = acc; sa[t] = alo; }
      };
      using yes = std::true_type;
      using no = std::false_type;
      int i = i0 + G * warp, t = t0 + warp;
      double* Ai = own0 + rstep * warp;
      for (; i < n; i += G * nw, t += nw, Ai += rstep * nw) {
        if (k < 0) {
          if (i == lo) do_row(i, t, Ai, no(), yes());
          else do_row(i, t, Ai, no(), no());
        } else {
          if (i == lo) do_row(i, t, Ai, yes(), yes());
          else do_row(i, t, Ai, yes(), no());
        }
      }
    }
    __syncthreads();                      // the sums, v and tau are there
    tau = s_tau;
    {
      const double v1 = s_c[3];
      ulonglong2* pw = xp + (size_t)((k + 1) & 1) * n;
      for (int i = i0 + G * tid, t = t0 + tid; i < n; i += G * TNT, t += TNT) {
        const double p = fma(sa[t], v1, sq[t]) * tau;
        if (solo) sq[t] = p;
        else if (plain) dp[(size_t)((k + 1) & 1) * n + i] = p;
        else put_word(pw + i, p, (unsigned long long)k + 2ull);
      }
    }
    if (scribe) {
      double* Vr = P.V + (int64_t)(k + 1) * n;
      for (int j = lo + tid; j < n; j += TNT) Vr[j] = vn[j];
      if (tid == 0) { P.e[k + 1] = s_c[2] * isc; P.tau[k + 1] = tau; }
    }
    { double* t = vk; vk = vn; vn = t; }
    if (solo) {
      double* t = sp; sp = sq; sq = t;
      __syncthreads();
    } else if (plain) {
      if (!grid_sync(bar, gen, poll_limit, (unsigned)G)) return;
    }
  }
}

// ---------------------------------------------------------------- stage 2
// Sturm count: the number of eigenvalues of T below x = the number of sign
// changes in the leading principal minors p_0 = 1, p_1, ..., p_n of T - x I,
// from the three-term recurrence p_i = (d_{i-1} - x) p_{i-1} -
// e_{i-2}^2 p_{i-2} (Wilkinson, The Algebraic Eigenvalue Problem, Ch. 5: the
// computed signs are exact for a matrix within a few ulps of T).  The FP64 pipe
// takes 64 cycles per warp instruction, so the recurrence is scaled to two of
// them a step: with q_i = p_i / c_i, c_i = e_{i-2}^2 c_{i-2}, it reads
// q_i = (d_{i-1} - x) r_i q_{i-1} - q_{i-2}, r_i = c_{i-1} / c_i, and (d - x) r is one FMA
// of d r and r.  c_i > 0, so the signs are those of p_i, and each coefficient
// is off by a few ulps, as rounding does to T's entries.
//   The c start at 1 every SB = 8 steps.  T arrives scaled by a power of two to
// entries of magnitude <= 1, and e_i^2 below 2^-112 counts as 2^-112 (e_i = 2^-56:
// below the rounding of entries of magnitude 1), so c >= 2^-448.  In 8 steps the
// larger of two neighbouring |p| grows by at most 3^8 and, solving the
// recurrence for p_{i-2}, falls by at most (3 2^112)^8 < 2^909; it is set to about
// 1 (a power of two) at the end of the 8, so nothing overflows or vanishes.  One
// of the pair may be 0, exactly or by underflow: the next q is then minus the one
// before it, and one sign change is counted whichever sign the zero has.
//   Per step: one shared load, two FMAs and a shift of the sign into a register,
// whose changes are counted by 8 at the block's end; ~210 cycles a step, of which
// the FP64 pipe 160 (the block's rescale included).  n = 200 397 -> 203 us,
// n = 1500 4.97 -> 2.62 ms against (d - x) p - e^2 p with a test for zero and a sign
// count in each step.
constexpr int SB = 8;
__device__ __forceinline__ int exp_bits(double v) {
  return (int)((__double_as_longlong(v) >> 52) & 0x7ff);
}
// t[i] = {d_i r_{i+1}, r_{i+1}}, c[b] = the last two c of block b of SB steps
__device__ __forceinline__ int sturm_count(const double2* t, const double2* c, int n, double x) {
  double pm = 0.0, pc = 1.0;          // q_{i-1}, q_i
  unsigned sg = 0;                    // signs of the q, the last in bit 0
  int cnt = 0;
  // a step ahead: the coefficient, two steps ahead: the table (both padded)
  double a = fma(-x, t[0].y, t[0].x);
  double2 v = t[1];
  auto step = [&](int i) {
    const double pn = fma(a, pc, -pm);
    a = fma(-x, v.y, v.x);
    v = t[i + 2];
    sg = __funnelshift_l((unsigned)__double2hiint(pn), sg, 1);
    pm = pc;
    pc = pn;
  };
  int i = 0;
  for (; i + SB <= n; i += SB) {
#pragma unroll
    for (int q = 0; q < SB; ++q) step(i + q);
    cnt += __popc((sg ^ (sg >> 1)) & ((1u << SB) - 1u));
    const double2 cb = c[i / SB];
    pm *= cb.x;
    pc *= cb.y;
    const int em = min(max(max(exp_bits(pc), exp_bits(pm)), 1), 2045);
    const double f = __longlong_as_double((long long)(2046 - em) << 52);     // 2^(1023 - em)
    pc *= f;
    pm *= f;
  }
  const int rest = n - i;
  for (; i < n; ++i) step(i);
  return cnt + __popc((sg ^ (sg >> 1)) & ((1u << rest) - 1u));
}

// Doubles as integers of the same order, and back.
__device__ __forceinline__ long long order_key(double v) {
  const long long b = __double_as_longlong(v);
  return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}
__device__ __forceinline__ double from_key(long long k) {
  return __longlong_as_double(k ^ (long long)((unsigned long long)(k >> 63) >> 1));
}

// Bisection by multisection: L lanes (a power of two up to 128: up to four
// warps) work on one eigenvalue, each round counting at L interior points of
// [lo, hi] and keeping the sub-interval that holds eigenvalue number a
// (ascending), until its width is below 2 eps ||T|| (the accuracy of the
// counts).  A warp issues one FP64 instruction per step whatever its lanes do, so
// L trades rounds (53 / log2(L + 1)) against warps: wide L for a few
// eigenvalues, narrow L for many.  CTA = BNW warps of one problem.
constexpr int BNW = 4;
__global__ void __launch_bounds__(BNW * 32) k_bisect(const EigProblem* probs, int L) {
  extern __shared__ __align__(16) double bsm[];
  const EigProblem P = probs[blockIdx.y];
  const int n = P.n;
  const int per_cta = BNW * 32 / L;
  if ((int)blockIdx.x * per_cta >= n) return;
  double2* t = reinterpret_cast<double2*>(bsm);        // {d r, r}
  double2* tc = t + n + 2;                             // the last two c per SB steps
  if (threadIdx.x < 2) t[n + threadIdx.x] = make_double2(0.0, 0.0);
  __shared__ long long s_lo[BNW], s_hi[BNW];
  __shared__ int s_first[BNW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Gershgorin's bounds
  long long klo = 0x7fffffffffffffffll, khi = -0x7fffffffffffffffll;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double di = P.d[i];
    const double r = (i > 0 ? fabs(P.e[i - 1]) : 0.0) + (i < n - 1 ? fabs(P.e[i]) : 0.0);
    klo = min(klo, order_key(di - r));
    khi = max(khi, order_key(di + r));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    klo = min(klo, __shfl_xor_sync(0xffffffffu, klo, o));
    khi = max(khi, __shfl_xor_sync(0xffffffffu, khi, o));
  }
  if (lane == 0) { s_lo[warp] = klo; s_hi[warp] = khi; }
  __syncthreads();
  for (int w = 0; w < BNW; ++w) { klo = min(klo, s_lo[w]); khi = max(khi, s_hi[w]); }
  double glo = from_key(klo), ghi = from_key(khi);
  const double tnorm = fmax(fabs(glo), fabs(ghi));
  // scale by 2^-ex (exact) so that ||T|| / 2^ex is in [0.5, 1)
  const int ex = (tnorm > 0.0) ? exp_bits(tnorm) - 1022 : 0;
  const double sc = __longlong_as_double((long long)(1023 - ex) << 52);
  const double isc = __longlong_as_double((long long)(1023 + ex) << 52);
  for (int b0 = threadIdx.x * SB; b0 < n; b0 += blockDim.x * SB) {
    double ca = 1.0, cb = 1.0;                         // c_{i-2}, c_{i-1}
#pragma unroll
    for (int q = 0; q < SB; ++q) {
      const int i = b0 + q;
      if (i < n) {
        const double ei = i > 0 ? P.e[i - 1] * sc : 1.0;
        const double e2 = ei * ei;
        const double c = ca * (e2 > 0x1p-112 ? e2 : 0x1p-112);
        const double r = cb * rcp64(c);
        t[i] = make_double2(P.d[i] * sc * r, r);
        ca = cb;
        cb = c;
      }
    }
    tc[b0 / SB] = make_double2(ca, cb);
  }
  __syncthreads();
  const double tn = tnorm * sc;
  const double atol = 2.0 * DBL_EPSILON * tn + DBL_MIN;
  glo = glo * sc - (2.0 * DBL_EPSILON * tn * n + DBL_MIN);
  ghi = ghi * sc + (2.0 * DBL_EPSILON * tn * n + DBL_MIN);
  const int g = threadIdx.x / L, l = threadIdx.x % L;           // group, lane in group
  const int j = blockIdx.x * per_cta + g;                       // descending index
  const bool valid = j < n;
  const int a = n - 1 - (valid ? j : n - 1);                    // ascending index
  const double part = 1.0 / (double)(L + 1);
  double lo = glo, hi = ghi;
  auto point = [&](int m) { return fma(hi - lo, (double)(m + 1) * part, lo); };
  if (L <= 32) {
    const int base = lane & ~(L - 1);
    const unsigned gmask = (L == 32) ? 0xffffffffu : (((1u << L) - 1u) << base);
    for (int round = 0; round < 64; ++round) {
      const bool active = valid && (hi - lo > atol);
      if (!__any_sync(0xffffffffu, active)) break;
      const int cnt = active ? sturm_count(t, tc, n, point(l)) : 0;
      const unsigned above = __ballot_sync(0xffffffffu, active && cnt > a) & gmask;
      const int m = above ? (__ffs(above) - 1 - base) : L;       // first point above, in group
      if (active) {
        const double xm = point(m), xl = point(m - 1);
        if (m < L) hi = xm;
        if (m > 0) lo = xl;
      }
    }
  } else {
    const int wpg = L / 32, w0 = warp - warp % wpg;
    for (int round = 0; round < 64; ++round) {
      const bool active = valid && (hi - lo > atol);
      if (!__syncthreads_or(active)) break;
      const int cnt = active ? sturm_count(t, tc, n, point(l)) : 0;
      const unsigned above = __ballot_sync(0xffffffffu, active && cnt > a);
      if (lane == 0) s_first[warp] = above ? __ffs(above) - 1 : 32;
      __syncthreads();
      int m = L;
      for (int w = wpg - 1; w >= 0; --w)
        if (s_first[w0 + w] < 32) m = 32 * w + s_first[w0 + w];
      if (active) {
        const double xm = point(m), xl = point(m - 1);
        if (m < L) hi = xm;
        if (m > 0) lo = xl;
      }
    }
  }
  if (valid && l == 0) P.w[j] = 0.5 * (lo + hi) * isc;
  if (blockIdx.x == 0 && threadIdx.x == 0) P.tau[n - 1] = tnorm;      // for k_invit
}

// ---------------------------------------------------------------- stage 4
// Inverse iteration: Gaussian elimination with partial pivoting of T - lambda I,
// then two solves, the first from a pseudo-random right-hand side.  Two lanes
// per wanted eigenvector: one eliminates from the first row down, the other
// from the last row up ("burning at both ends"), the 2 x 2 system where they
// meet gives the two middle entries, and both substitute back outwards, so the
// dependent chain is n / 2 steps long.  In local indices (s = 0 at the lane's end)
// both lanes run the same code; a row swap gives U a second superdiagonal.
// Pivots below 2^-92 ||T|| are raised to that size (the shift is an eigenvalue, so
// one pivot is ~0; raised to eps ||T||, which shifts the eigenvalue by as much, the
// vectors of close eigenvalues came out up to 4 times as far off); a running power-of-two rescale (|z| <= 2^400, so the sum of
// squares stays finite) keeps the back substitution finite.  Output column j
// of Z (n x R, row-major: Z[i*R + j]), a unit vector.
//   The FP64 pipe is the limit (a warp instruction takes 64 cycles of it whatever
// its lanes do), so what need not be FP64 is not: the right-hand side's bits
// are hashed directly, pivots are compared as integers, nothing is scaled
// that need not be.  18 FP64 instructions a step, n / 2 steps: 186 us at n = 200, 489 us at
// n = 500 (34 and n with one lane per vector: 371 and 975 us).  The factorization runs
// fused with the first forward elimination, and the pivots are stored as
// reciprocals (rcp64), so the only reciprocal on the chain is the factorization's.
__device__ __forceinline__ uint32_t hash_u32(uint32_t i, uint32_t j) {
  uint32_t h = i * 0x9E3779B1u ^ (j + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; h ^= h >> 15;
  return h;
}
// +-[1, 2)
__device__ __forceinline__ double hash_unit(uint32_t i, uint32_t j) {
  const uint32_t h = hash_u32(i, j);
  return __hiloint2double((int)(0x3ff00000u | (h & 0x800fffffu)), (int)(h * 0x9E3779B1u));
}

// OP 0: rcp64, 1: sqrt64, 2: f64_to_f32
template <int OP, typename TOut>
__global__ void k_scalar_probe(const double* x, TOut* y, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if constexpr (OP == 0) y[i] = rcp64(x[i]);
  else if constexpr (OP == 1) y[i] = sqrt64(x[i]);
  else y[i] = f64_to_f32(x[i]);
}

__global__ void __launch_bounds__(32) k_invit(const EigProblem* probs, int nprob, int total) {
  // flattened (problem, vector): probs[p].zoff is the first vector of p; lanes
  // 0-15 from the top, 16-31 from the bottom (past the last vector: no rows)
  const bool up = threadIdx.x >= 16;
  const int tv = (int)(blockIdx.x * 16 + (threadIdx.x & 15)), t = min(tv, total - 1);
  int p = 0;
  while (p + 1 < nprob && probs[p + 1].zoff <= t) ++p;
  const EigProblem P = probs[p];
  const int j = t - P.zoff;
  const int n = P.n, R = P.R;
  const int len = tv >= total ? 0 : (up ? n / 2 : n - n / 2);      // rows of this lane
  const double lam = P.w[j];
  const double* __restrict__ d = P.d + (up ? n - 1 : 0);
  const double* __restrict__ e = P.e + (up ? n - 2 : 0);
  const int dir = up ? -1 : 1;
  const int64_t o0 = (int64_t)(up ? n - 1 : 0) * R + j, step = (int64_t)dir * R;
  double* __restrict__ RI = P.lu + o0;                   // 1 / pivot
  double* __restrict__ U1 = RI + (int64_t)n * R;
  double* __restrict__ U2 = U1 + (int64_t)n * R;
  double* __restrict__ M = U2 + (int64_t)n * R;
  unsigned char* __restrict__ flag = reinterpret_cast<unsigned char*>(P.lu + 4 * (int64_t)n * R) + o0;
  unsigned char* __restrict__ scnt = flag + (int64_t)n * R;
  double* __restrict__ Z = P.z + o0;
  auto at = [&](int s) { return s * step; };
  const double ptol = fmax(0x1p-92 * P.tau[n - 1], 0x1p-990);      // tau[n - 1]: ||T|| (k_bisect)
  const unsigned long long ptol_bits = (unsigned long long)__double_as_longlong(ptol);
  auto absb = [](double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  };
  auto floored = [&](double v) { return absb(v) < ptol_bits ? (v < 0.0 ? -ptol : ptol) : v; };
  // factorization fused with the forward elimination of b (random); y -> Z.
  // The pending row is p0 z(s) + p1 z(s + 1) = pb.
  double p0 = 1.0, p1 = 0.0, pb = 0.0;
  if (len > 0) {
    p0 = d[0] - lam;
    p1 = n > 1 ? e[0] : 0.0;
    pb = hash_unit(up ? n - 1 : 0, j);
  }
  for (int s = 0; s + 1 < len; ++s) {
    const double es = e[dir * s];
    const double a1 = d[dir * (s + 1)] - lam;
    // (local s + 1 couples to s + 2, at the end to the other lane's last row)
    const int ie = up ? n - 2 - (s + 1) : s + 1;
    const double e1 = ie >= 0 && ie < n - 1 ? e[dir * (s + 1)] : 0.0;
    const double bs1 = hash_unit(up ? n - 2 - s : s + 1, j);
    const bool swap = absb(es) > absb(p0);
    if (!swap) p0 = floored(p0);
    const double r = rcp64(swap ? es : p0);
    const double m = (swap ? p0 : es) * r;
    RI[at(s)] = r;
    U1[at(s)] = swap ? a1 : p1;
    U2[at(s)] = swap ? e1 : 0.0;
    M[at(s)] = m;
    flag[at(s)] = swap ? 1 : 0;
    double ys;
    if (swap) {
      ys = bs1;
      pb = fma(-m, bs1, pb);
      p0 = fma(-m, a1, p1);
      p1 = -m * e1;
    } else {
      ys = pb;
      pb = fma(-m, pb, bs1);
      p0 = fma(-m, p1, a1);
      p1 = e1;
    }
    Z[at(s)] = ys;
  }
  // The 2 x 2 system of the two pending rows, unknowns (top's last, bottom's
  // last), factored once, the same in both lanes.
  double t0, t1, b0, b1;
  {
    const double q0 = __shfl_xor_sync(0xffffffffu, p0, 16), q1 = __shfl_xor_sync(0xffffffffu, p1, 16);
    t0 = up ? q0 : p0;  t1 = up ? q1 : p1;                // top's row
    b0 = up ? p1 : q1;  b1 = up ? p0 : q0;                // bottom's row, same unknowns
    if (n == 1) { t1 = 0.0; b0 = 0.0; b1 = 1.0; }
  }
  const bool mswap = absb(b0) > absb(t0);
  const double piv = floored(mswap ? b0 : t0), piv_x = mswap ? b1 : t1;
  const double rp = rcp64(piv), mm = (mswap ? t0 : b0) * rp;
  const double rq = rcp64(floored(fma(-mm, piv_x, mswap ? t1 : b1)));
  const double SMALL = 0x1p-400;
  // (1 / pivot may be near overflow: the first solution is scaled to about 1)
  const bool tiny = P.tau[n - 1] < 0x1p-400;
  double ss = 0.0;
  int nres = 0;
  // the passes below prefetch the operands of the next PF steps into
  // registers before working through the current ones, which keeps the L2
  // latency off the dependent chain (each step stores into Z, so the
  // compiler cannot move the next loads ahead by itself)
  constexpr int PF = 8;
  for (int it = 0; it < 2; ++it) {
    if (it == 1 && len > 0) {
      // forward elimination of the previous solution
      double pv = Z[at(0)];
      double nb_[PF], nm_[PF];
      unsigned char nf_[PF];
      auto load_f = [&](int s0) {
#pragma unroll
        for (int q = 0; q < PF; ++q) {
          const int s = s0 + q;
          const bool ok = s + 1 < len;
          nb_[q] = ok ? Z[at(s + 1)] : 0.0;
          nm_[q] = ok ? M[at(s)] : 0.0;
          nf_[q] = ok ? flag[at(s)] : 0;
        }
      };
      load_f(0);
      for (int s0 = 0; s0 + 1 < len; s0 += PF) {
        double cb[PF], cm[PF];
        unsigned char cf[PF];
#pragma unroll
        for (int q = 0; q < PF; ++q) { cb[q] = nb_[q]; cm[q] = nm_[q]; cf[q] = nf_[q]; }
        if (s0 + PF + 1 < len) load_f(s0 + PF);
#pragma unroll
        for (int q = 0; q < PF; ++q) {
          const int s = s0 + q;
          if (s + 1 < len) {
            const double ys = cf[q] ? cb[q] : pv;
            pv = cf[q] ? fma(-cm[q], cb[q], pv) : fma(-cm[q], pv, cb[q]);
            Z[at(s)] = ys;
          }
        }
      }
      pb = pv;
    }
    // the middle entries: z1 this lane's last, z2 the other's
    double z1, z2;
    {
      const double o = __shfl_xor_sync(0xffffffffu, pb, 16);
      const double bt = up ? o : pb, bb = n == 1 ? 0.0 : (up ? pb : o);
      const double rhs = mswap ? bb : bt;
      const double zb = fma(-mm, rhs, mswap ? bt : bb) * rq;          // bottom's last
      const double zt = fma(-piv_x, zb, rhs) * rp;                    // top's last
      z1 = up ? zb : zt;
      z2 = up ? zt : zb;
    }
    // back substitution with rescaling; scnt[s] = rescales before z(s) was
    // stored; the sum of squares is kept at the running scale
    nres = 0;
    double sc = 1.0;             // 2^(-400 nres): the scale of z1, z2 and zk
    ss = 0.0;
    if (len > 0) {
      for (int q = 0; q < 3 && max(absb(z1), absb(z2)) > 0x58F0000000000000ull; ++q) {   // > 2^400
        z1 *= SMALL; z2 *= SMALL; sc *= SMALL;
        ++nres;
      }
      Z[at(len - 1)] = z1;
      scnt[at(len - 1)] = (unsigned char)nres;
      ss = z1 * z1;
    }
    double ny[PF], n1[PF], n2[PF], nr[PF];
    auto load_b = [&](int s0) {   // steps s0, s0 - 1, ..., s0 - PF + 1
#pragma unroll
      for (int q = 0; q < PF; ++q) {
        const int s = s0 - q;
        const bool ok = s >= 0;
        ny[q] = ok ? Z[at(s)] : 0.0;
        n1[q] = ok ? U1[at(s)] : 0.0;
        n2[q] = ok ? U2[at(s)] : 0.0;
        nr[q] = ok ? RI[at(s)] : 0.0;
      }
    };
    load_b(len - 2);
    for (int s0 = len - 2; s0 >= 0; s0 -= PF) {
      double cy[PF], c1[PF], c2[PF], cr[PF];
#pragma unroll
      for (int q = 0; q < PF; ++q) { cy[q] = ny[q]; c1[q] = n1[q]; c2[q] = n2[q]; cr[q] = nr[q]; }
      if (s0 - PF >= 0) load_b(s0 - PF);
#pragma unroll
      for (int q = 0; q < PF; ++q) {
        const int s = s0 - q;
        if (s >= 0) {
          double rr = cy[q];
          if (nres) rr *= sc;
          if (absb(c2[q]) != 0) rr = fma(-c2[q], z2, rr);
          rr = fma(-c1[q], z1, rr);
          double zk = rr * cr[q];
          if (absb(zk) > 0x58F0000000000000ull) {   // |zk| > 2^400: rescale by 2^-400
            zk *= SMALL; z1 *= SMALL; z2 *= SMALL; sc *= SMALL; ss *= 0x1p-800;
            ++nres;
          }
          Z[at(s)] = zk;
          scnt[at(s)] = (unsigned char)(nres > 255 ? 255 : nres);
          if (it == 1) ss = fma(zk, zk, ss);
          z2 = z1;
          z1 = zk;
        }
      }
    }
    // one scale for both ends
    const int nmax = max(nres, __shfl_xor_sync(0xffffffffu, nres, 16));
    if (nmax > 0) {
      for (int s = 0; s < len; ++s) {
        double zk = Z[at(s)];
        for (int q = scnt[at(s)]; q < nmax; ++q) zk *= SMALL;
        Z[at(s)] = zk;
      }
      for (int q = nres; q < nmax; ++q) ss *= 0x1p-800;
    }
    if (it == 0 && __any_sync(0xffffffffu, tiny)) {
      unsigned long long mx = 1ull << 52;
      for (int s = 0; s < len; ++s) mx = max(mx, absb(Z[at(s)]));
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
      const double f = __longlong_as_double((long long)(2046 - min((int)(mx >> 52), 2045)) << 52);
      for (int s = 0; s < len; ++s) Z[at(s)] *= f;
    }
  }
  ss += __shfl_xor_sync(0xffffffffu, ss, 16);
  const double bscale = (ss > 0.0) ? rcp64(sqrt(ss)) : 1.0;
  for (int s = 0; s < len; ++s) Z[at(s)] *= bscale;
}

// ---------------------------------------------------------------- stage 5
// Cholesky QR: with G = Z^T Z = L L^T, Q = Z L^-T.  Every diagonal block of 32
// columns (64: the whole matrix, when R <= 64) is factored by one CTA as
// W G W^T = D, W unit lower triangular, by eliminating [G | I] in shared memory:
// a column costs one reciprocal of a pivot on the chain and one barrier, and
// the inverse comes out with the factor, so that Q is a product (no chain of
// divisions per row).  L^-1 = D^-1/2 W.
//   R <= 64: k_chol_small leaves L^-1 in P.gram, k_apply_small forms Q.
//   R > 64: per block of 32 columns k_chol_diag (L_pp^-1 into the diagonal
// block), k_chol_panel (L_ip = G_ip L_pp^-T), k_chol_trail (G_ij -= L_ip
// L_jp^T, lower blocks); k_apply_big substitutes block by block.
// Measured: R = 401 of n = 1500 took 17.9 ms for the factor in one CTA and 6.3 ms
// for the substitution in one thread per row; R = 28 of n = 200 53 and 54 us.
//   A pivot <= 0 (info[0] = 1) or a condition number of Z above 1e6 (info[0] =
// 2: inverse iteration returned nearly dependent vectors, and the QR would
// lose orthogonality) marks the problem as failed; the host then takes
// another solver for it.
//   The second pass restores orthogonality to rounding when eigenvalues are
// clustered.  Z's columns are unit vectors; when their Gram is the identity
// to within 1/64 in norm (the first pass's k_chol_small / k_chol_far look), the
// first pass's Q is orthonormal to rounding already and the second is not run
// (info[1] stays 0: its kernels return).
constexpr int CB = 32;                       // columns per block, R > 64
constexpr int CS = 64;                       // largest R of the one-CTA factor

// Whether an off-diagonal or diagonal entry is too far from the identity's for
// the first pass to be enough: the sum of squares of all R^2 deviations within
// (1/64)^2 if each is within 1 / (64 R).
__device__ __forceinline__ bool far_from_identity(double g, bool diag, int R) {
  const double e = fabs(diag ? g - 1.0 : g);
  return !(e * (64.0 * R) <= 1.0);
}

// Eliminates [G | I] of the m x m block in sm (m <= CS): on return the lower
// triangle's diagonal holds D, and W's strict lower triangle sits transposed
// in the upper one (W[i][j] at sm[j][i]).  256 threads: four per row.  s_r: a
// shared word for the pivot's reciprocal.  Returns false on a pivot <= 0.
__device__ bool eliminate(double (*sm)[CS + 1], int m, double* s_r) {
  const int i = threadIdx.x >> 2, jg = threadIdx.x & 3;
  if (threadIdx.x == 0) *s_r = sm[0][0] > 0.0 ? rcp64(sm[0][0]) : 0.0;
  __syncthreads();
  for (int c = 0; c < m; ++c) {
    const double r = *s_r;
    if (!(r > 0.0)) return false;              // the same word for every thread
    const bool act = i > c && i < m;
    const bool piv = i == c + 1 && i < m && jg == ((c + 1) & 3);
    double f = 0.0, rn = 0.0;
    if (act) {
      f = sm[i][c] * r;
      if (piv) {                               // the next pivot first: its reciprocal is the chain
        const double p = fma(-f, sm[i][c], sm[i][i]);
        sm[i][i] = p;
        rn = p > 0.0 ? rcp64(p) : 0.0;
      }
      for (int j = jg; j < c; j += 4) sm[j][i] = fma(-f, sm[j][c], sm[j][i]);      // W[i][j] -= f W[c][j]
      for (int j = c + 1 + ((jg - c - 1) & 3); j <= i; j += 4)
        if (!(piv && j == i)) sm[i][j] = fma(-f, sm[j][c], sm[i][j]);
    }
    __syncthreads();                           // column c and the reciprocal are read
    if (act && jg == (c & 3)) sm[c][i] = -f;   // W[i][c] (over nothing: column c of G is used up)
    if (piv) *s_r = rn;
    __syncthreads();
  }
  return true;
}

__global__ void __launch_bounds__(TNT) k_chol_small(const EigProblem* probs, int pass) {
  const EigProblem P = probs[blockIdx.x];
  const int R = P.R;
  if (R > CS || P.info[0] || (pass > 0 && !P.info[1])) return;
  __shared__ double sm[CS][CS + 1];
  __shared__ double s_r, isq[CS];
  double* Gm = P.gram;
  bool far = false;
  for (int e = threadIdx.x; e < R * R; e += TNT) {
    const int i = e / R, j = e - i * R;
    const double g = Gm[e];
    sm[i][j] = j <= i ? g : 0.0;
    far |= far_from_identity(g, i == j, R);
  }
  if (pass == 0 && __syncthreads_or(far) && threadIdx.x == 0) P.info[1] = 1;
  __syncthreads();
  if (!eliminate(sm, R, &s_r)) {
    if (threadIdx.x == 0) P.info[0] = 1;
    return;
  }
  if (threadIdx.x < R) isq[threadIdx.x] = 1.0 / sqrt(sm[threadIdx.x][threadIdx.x]);
  __syncthreads();
  for (int e = threadIdx.x; e < R * R; e += TNT) {
    const int i = e / R, j = e - i * R;
    Gm[e] = j > i ? 0.0 : (j == i ? isq[i] : isq[i] * sm[j][i]);
  }
  if (threadIdx.x < 32) {
    double lo = INFINITY, hi = 0.0;            // of the pivots' 1 / sqrt
    for (int c = threadIdx.x; c < R; c += 32) { lo = fmin(lo, isq[c]); hi = fmax(hi, isq[c]); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (threadIdx.x == 0 && lo < 1e-6 * hi) P.info[0] = 2;
  }
}

// Q = Z L^-T, eight rows of Z per CTA (x) and problem (y), R <= 64.
constexpr int AR = 8;
__global__ void __launch_bounds__(TNT) k_apply_small(const EigProblem* probs, int pass) {
  const EigProblem P = probs[blockIdx.y];
  const int R = P.R, i0 = blockIdx.x * AR;
  if (R > CS || i0 >= P.n || P.info[0] || (pass > 0 && !P.info[1])) return;
  __shared__ double ws[CS][CS + 1], zs[AR][CS + 1];
  for (int e = threadIdx.x; e < R * R; e += TNT) ws[e / R][e % R] = P.gram[e];
  const int nr = min(AR, P.n - i0);
  for (int e = threadIdx.x; e < nr * R; e += TNT) zs[e / R][e % R] = P.z[(int64_t)i0 * R + e];
  __syncthreads();
  const int r = threadIdx.x >> 5;
  if (r >= nr) return;
  for (int c = threadIdx.x & 31; c < R; c += 32) {
    double s0 = 0.0, s1 = 0.0;
    int k = 0;
    for (; k + 1 <= c; k += 2) {
      s0 = fma(zs[r][k], ws[c][k], s0);
      s1 = fma(zs[r][k + 1], ws[c][k + 1], s1);
    }
    if (k <= c) s0 = fma(zs[r][k], ws[c][k], s0);
    P.z[(int64_t)(i0 + r) * R + c] = s0 + s1;
  }
}

// R > 64: is G far from the identity (first pass)?
__global__ void __launch_bounds__(TNT) k_chol_far(const EigProblem* P_) {
  const EigProblem P = *P_;
  const int64_t R = P.R;
  bool far = false;
  for (int64_t e = (int64_t)blockIdx.x * TNT + threadIdx.x; e < R * R; e += (int64_t)gridDim.x * TNT)
    far |= far_from_identity(P.gram[e], e / R == e % R, (int)R);
  if (__syncthreads_or(far) && threadIdx.x == 0) P.info[1] = 1;
}

// Diagonal block p: L_pp^-1 in place (lower); its pivots' 1 / sqrt into P.lu (free
// by now); the last block checks the condition.
__global__ void __launch_bounds__(TNT) k_chol_diag(const EigProblem* P_, int p, int pass) {
  const EigProblem P = *P_;
  if (P.info[0] || (pass > 0 && !P.info[1])) return;
  __shared__ double sm[CS][CS + 1];
  __shared__ double s_r, isq[CB], red[2][TNW];
  const int R = P.R, c0 = p * CB, m = min(CB, R - c0);
  for (int e = threadIdx.x; e < m * m; e += TNT) {
    const int i = e / m, j = e - i * m;
    sm[i][j] = j <= i ? P.gram[(int64_t)(c0 + i) * R + c0 + j] : 0.0;
  }
  __syncthreads();
  if (!eliminate(sm, m, &s_r)) {
    if (threadIdx.x == 0) P.info[0] = 1;
    return;
  }
  if (threadIdx.x < m) {
    isq[threadIdx.x] = 1.0 / sqrt(sm[threadIdx.x][threadIdx.x]);
    P.lu[c0 + threadIdx.x] = isq[threadIdx.x];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < m * m; e += TNT) {
    const int i = e / m, j = e - i * m;
    P.gram[(int64_t)(c0 + i) * R + c0 + j] = j > i ? 0.0 : (j == i ? isq[i] : isq[i] * sm[j][i]);
  }
  if (c0 + m < R) return;
  double lo = INFINITY, hi = 0.0;
  for (int c = threadIdx.x; c < R; c += TNT) {
    const double v = c < c0 ? P.lu[c] : isq[c - c0];
    lo = fmin(lo, v);
    hi = fmax(hi, v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = lo; red[1][threadIdx.x >> 5] = hi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < TNW; ++w) { lo = fmin(lo, red[0][w]); hi = fmax(hi, red[1][w]); }
    if (lo < 1e-6 * hi) P.info[0] = 2;
  }
}

// acc[q] += sum_k a[row][k] b[col][k], a thread's 4 outputs of a 32 x 32 tile:
// row = threadIdx.x / 8, columns threadIdx.x % 8 + 8 q.
__device__ __forceinline__ void tile_dot(const double (*a)[CB + 1], const double (*b)[CB + 1],
                                         double (&acc)[4]) {
  const int row = threadIdx.x >> 3, col = threadIdx.x & 7;
#pragma unroll 8
  for (int k = 0; k < CB; ++k) {
    const double v = a[row][k];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = fma(v, b[col + 8 * q][k], acc[q]);
  }
}
// Loads the 32 x 32 tile at (r0, c0) of the R x R matrix (zero outside).
__device__ __forceinline__ void tile_load(const double* G, int64_t R, int64_t r0, int64_t c0,
                                          double (*t)[CB + 1]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int row = (threadIdx.x >> 5) + 8 * q, col = threadIdx.x & 31;
    t[row][col] = (r0 + row < R && c0 + col < R) ? G[(r0 + row) * R + c0 + col] : 0.0;
  }
}

// L_ip = G_ip L_pp^-T, block i = p + 1 + blockIdx.x.
__global__ void __launch_bounds__(TNT) k_chol_panel(const EigProblem* P_, int p, int pass) {
  const EigProblem P = *P_;
  if (P.info[0] || (pass > 0 && !P.info[1])) return;
  __shared__ double a[CB][CB + 1], b[CB][CB + 1];
  const int64_t R = P.R, r0 = (int64_t)(p + 1 + blockIdx.x) * CB, c0 = (int64_t)p * CB;
  tile_load(P.gram, R, r0, c0, a);
  tile_load(P.gram, R, c0, c0, b);
  __syncthreads();
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  tile_dot(a, b, acc);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int64_t row = r0 + (threadIdx.x >> 3), col = c0 + (threadIdx.x & 7) + 8 * q;
    if (row < R && col < R) P.gram[row * R + col] = acc[q];
  }
}

// G_ij -= L_ip L_jp^T, blocks i >= j > p (blockIdx.x: the lower triangle in row order).
__global__ void __launch_bounds__(TNT) k_chol_trail(const EigProblem* P_, int p, int pass) {
  const EigProblem P = *P_;
  if (P.info[0] || (pass > 0 && !P.info[1])) return;
  __shared__ double a[CB][CB + 1], b[CB][CB + 1];
  const int t = (int)blockIdx.x;
  int bi = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
  while (bi * (bi + 1) / 2 > t) --bi;
  const int bj = t - bi * (bi + 1) / 2;
  const int64_t R = P.R, r0 = (int64_t)(p + 1 + bi) * CB, q0 = (int64_t)(p + 1 + bj) * CB;
  tile_load(P.gram, R, r0, (int64_t)p * CB, a);
  tile_load(P.gram, R, q0, (int64_t)p * CB, b);
  __syncthreads();
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  tile_dot(a, b, acc);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int64_t row = r0 + (threadIdx.x >> 3), col = q0 + (threadIdx.x & 7) + 8 * q;
    if (row < R && col < R) P.gram[row * R + col] -= acc[q];
  }
}

// Q = Z L^-T by blocks of columns, blockDim.x / 32 rows of Z per CTA: Q_p = (Z_p -
// sum_{q < p} Q_q L_pq^T) L_pp^-T.  A thread owns one row and one column of the block.
__global__ void __launch_bounds__(512) k_apply_big(const EigProblem* P_, int pass) {
  const EigProblem P = *P_;
  if (P.info[0] || (pass > 0 && !P.info[1])) return;
  __shared__ double ls[CB][CB + 1], zs[16][CB + 1];
  const int64_t R = P.R;
  const int nr = blockDim.x >> 5, r = threadIdx.x >> 5, c = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * nr + r;
  double* z = P.z + (i < P.n ? i : 0) * R;
  for (int64_t c0 = 0; c0 < R; c0 += CB) {
    double acc = (i < P.n && c0 + c < R) ? z[c0 + c] : 0.0;
    for (int64_t q0 = 0; q0 <= c0; q0 += CB) {
      __syncthreads();
      for (int e = threadIdx.x; e < CB * CB; e += blockDim.x) {
        const int64_t row = c0 + e / CB, col = q0 + e % CB;
        ls[e / CB][e % CB] = (row < R && col < R) ? P.gram[row * R + col] : 0.0;
      }
      zs[r][c] = q0 < c0 ? (i < P.n ? z[q0 + c] : 0.0) : acc;   // (blocks q0 < c0 are whole)
      __syncthreads();
      double s = 0.0, t = 0.0;
#pragma unroll
      for (int k = 0; k < CB; k += 2) {
        s = fma(zs[r][k], ls[c][k], s);
        t = fma(zs[r][k + 1], ls[c][k + 1], t);
      }
      acc = q0 < c0 ? acc - (s + t) : s + t;
    }
    if (i < P.n && c0 + c < R) z[c0 + c] = acc;
  }
}

// ---------------------------------------------------------------- stage 6
// U = Q_H Z with Q_H = H_0 H_1 ... H_{n-3}, in blocks of WYB reflectors: a
// block H_k0 ... H_{k0+m-1} equals I - V T V^T with V = [v_k0 ... v_{k0+m-1}]
// and T upper triangular (the compact WY form, Schreiber & Van Loan 1989:
// T_jj = tau_j, T[0:j, j] = -tau_j T[0:j, 0:j] (V[:, 0:j]^T v_j)).  The blocks
// are applied from the last to the first: z <- z - V (T (V^T z)).  U is
// I x R column-major.
constexpr int WYB = 32;
__host__ __device__ __forceinline__ int wy_blocks(int n) { return n > 2 ? (n - 2 + WYB - 1) / WYB : 0; }

// One CTA per block of reflectors: the T factor into wyT (WYB x WYB, row-major).
// probs NULL: the problem `one`.
__global__ void __launch_bounds__(256) k_wy_t(const EigProblem* probs, const EigProblem one) {
  const EigProblem P = probs ? probs[blockIdx.y] : one;
  const int n = P.n, b = blockIdx.x;
  if (b >= wy_blocks(n)) return;
  const int k0 = b * WYB, m = min(WYB, n - 2 - k0);
  __shared__ double W[WYB][WYB + 1];
  __shared__ double T[WYB][WYB + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // W[i][j] = v_{k0+i} . v_{k0+j} for i < j; v_{k0+j} is V[k0+j][c] from c = k0+j+1
  for (int q = warp; q < m * m; q += 8) {
    const int i = q / m, jj = q % m;
    if (i >= jj) continue;
    const double* vi = P.V + (int64_t)(k0 + i) * n;
    const double* vj = P.V + (int64_t)(k0 + jj) * n;
    const int s0 = k0 + jj + 1;
    double acc = 0.0;
    for (int c = s0 + lane; c < n; c += 32) acc = fma(vi[c], vj[c], acc);
    acc = warp_sum(acc);
    if (lane == 0) W[i][jj] = acc;
  }
  __syncthreads();
  if (warp == 0) {
    for (int jj = 0; jj < m; ++jj) {
      const double tj = P.tau[k0 + jj];
      if (lane < jj) {
        double s = 0.0;
        for (int l = lane; l < jj; ++l) s = fma(T[lane][l], W[l][jj], s);
        T[lane][jj] = -tj * s;
      } else if (lane == jj) {
        T[lane][jj] = tj;
      }
      __syncwarp();
    }
  }
  __syncthreads();
  double* To = P.wyT + (size_t)b * WYB * WYB;
  for (int q = threadIdx.x; q < WYB * WYB; q += 256) {
    const int i = q / WYB, jj = q % WYB;
    To[q] = (i < m && jj < m && i <= jj) ? T[i][jj] : 0.0;
  }
}

// One CTA per eigenvector (flattened over problems), the vector in shared memory.
__global__ void __launch_bounds__(256) k_backtransform(const EigProblem* probs, int nprob) {
  extern __shared__ __align__(16) double zs[];
  __shared__ double y[WYB], y2[WYB];
  const int t = blockIdx.x;
  int p = 0;
  while (p + 1 < nprob && probs[p + 1].zoff <= t) ++p;
  const EigProblem P = probs[p];
  const int j = t - P.zoff;
  if (j < 0 || j >= P.R || P.info[0]) return;
  const int n = P.n, R = P.R;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* V = P.V;
  for (int i = threadIdx.x; i < n; i += blockDim.x) zs[i] = P.z[(int64_t)i * R + j];
  __syncthreads();
  for (int b = wy_blocks(n) - 1; b >= 0; --b) {
    const int k0 = b * WYB, m = min(WYB, n - 2 - k0);
    // y = V^T z
    for (int q = warp; q < m; q += 8) {
      const double* v = V + (int64_t)(k0 + q) * n;
      const int s0 = k0 + q + 1;
      double acc = 0.0;
      for (int c = s0 + lane; c < n; c += 32) acc = fma(v[c], zs[c], acc);
      acc = warp_sum(acc);
      if (lane == 0) y[q] = acc;
    }
    __syncthreads();
    // y2 = T y
    if (warp == 0 && lane < m) {
      const double* Tb = P.wyT + (size_t)b * WYB * WYB + (size_t)lane * WYB;
      double s = 0.0;
      for (int l = lane; l < m; ++l) s = fma(Tb[l], y[l], s);
      y2[lane] = s;
    }
    __syncthreads();
    // z <- z - V y2 (entry i gets the reflectors q with k0 + q + 1 <= i)
    for (int i = k0 + 1 + threadIdx.x; i < n; i += blockDim.x) {
      const int qmax = min(m, i - k0);
      double s = 0.0;
      for (int q = 0; q < qmax; ++q) s = fma(V[(int64_t)(k0 + q) * n + i], y2[q], s);
      zs[i] -= s;
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) P.U[(int64_t)j * n + i] = zs[i];
}

// ---------------------------------------------------------------- batched helpers
// Rank cut of Eq. Un (or the given rank) for each problem, one CTA each.
__global__ void __launch_bounds__(RANK_CUT_NT) k_rank_cut_batched(const EigProblem* probs,
                                                                  const double* thr,
                                                                  const int* fixed, int64_t* R_out,
                                                                  double* disc_out) {
  const int p = blockIdx.x;
  rank_cut_cta(probs[p].w, probs[p].n, thr[p], fixed ? fixed[p] : 0, R_out + p, disc_out + p);
}

// G = Z^T Z (R x R, full) for each problem with R <= 64, one CTA each: rows of
// Z staged 16 at a time in shared memory, one thread per lower-triangle entry
// (several when R(R+1)/2 > 256), FP64 sums in row order.
constexpr int ZG_MAXR = 64, ZG_ROWS = 16, ZG_PPT = (ZG_MAXR * (ZG_MAXR + 1) / 2 + TNT - 1) / TNT;
__global__ void __launch_bounds__(TNT) k_zgram_batched(const EigProblem* probs, int pass) {
  const EigProblem P = probs[blockIdx.x];
  const int n = P.n, R = P.R;
  if (R > ZG_MAXR || P.info[0] || (pass > 0 && !P.info[1])) return;
  __shared__ double zs[ZG_ROWS][ZG_MAXR + 1];
  const int npair = R * (R + 1) / 2;
  int pa[ZG_PPT], pb[ZG_PPT];
  double acc[ZG_PPT];
#pragma unroll
  for (int q = 0; q < ZG_PPT; ++q) {
    const int t = threadIdx.x + TNT * q;
    int a = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while ((a + 1) * (a + 2) / 2 <= t) ++a;
    while (a * (a + 1) / 2 > t) --a;
    pa[q] = (t < npair) ? a : 0;
    pb[q] = (t < npair) ? t - a * (a + 1) / 2 : 0;
    acc[q] = 0.0;
  }
  for (int i0 = 0; i0 < n; i0 += ZG_ROWS) {
    __syncthreads();
    for (int c = threadIdx.x; c < ZG_ROWS * R; c += TNT) {
      const int r = c / R, a = c - r * R;
      zs[r][a] = (i0 + r < n) ? P.z[(int64_t)(i0 + r) * R + a] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < ZG_PPT; ++q) {
      if (threadIdx.x + TNT * q >= npair) break;
      double s = acc[q];
#pragma unroll
      for (int r = 0; r < ZG_ROWS; ++r) s = fma(zs[r][pa[q]], zs[r][pb[q]], s);
      acc[q] = s;
    }
  }
#pragma unroll
  for (int q = 0; q < ZG_PPT; ++q) {
    if (threadIdx.x + TNT * q >= npair) break;
    P.gram[(int64_t)pa[q] * R + pb[q]] = acc[q];
    P.gram[(int64_t)pb[q] * R + pa[q]] = acc[q];
  }
}

// ---------------------------------------------------------------- launchers
cudaError_t launch_rank_cut_batched(const EigProblem* probs_dev, int count, const double* thr,
                                    const int* fixed, int64_t* R_out, double* disc_out,
                                    cudaStream_t st) {
  k_rank_cut_batched<<<count, RANK_CUT_NT, 0, st>>>(probs_dev, thr, fixed, R_out, disc_out);
  count_launches(1);
  return cudaGetLastError();
}

int zgram_batched_max_r() { return ZG_MAXR; }

cudaError_t launch_zgram_batched(const EigProblem* probs_dev, int count, int pass,
                                 cudaStream_t st) {
  k_zgram_batched<<<count, TNT, 0, st>>>(probs_dev, pass);
  count_launches(1);
  return cudaGetLastError();
}

namespace {
int tridiag_rows_per_cta(int n, int G) { return (n + G - 1) / G; }
size_t tridiag_base_smem(int n, int G) {
  return sizeof(double) * (3 * (size_t)n + 2 * (size_t)tridiag_rows_per_cta(n, G) + (G == 1 ? n : 0));
}
constexpr size_t kTridiagSmemRowsCap = 120 * 1024;
}  // namespace

// ~6 rows per CTA at the first step (the step time is latency-bound: 2 to 8
// rows per CTA measured within 8% of each other at n = 500), at most one CTA
// per SM
int tridiag_team_size(int n, int num_sms) {
  int G = (n + 5) / 6;
  return G > num_sms ? num_sms : (G < 1 ? 1 : G);
}

void tridiag_batch_teams(const int* n, int count, int num_sms, int* team) {
  for (int p = 0; p < count; ++p) team[p] = 1;
  if (count >= num_sms) return;
  double tot = 0.0;
  for (int p = 0; p < count; ++p) tot += (double)n[p] * n[p] * n[p];
  const int extra = num_sms - count;
  for (int p = 0; p < count; ++p) {
    int g = 1 + (int)(extra * ((double)n[p] * n[p] * n[p]) / (tot > 0.0 ? tot : 1.0));
    const int cap = tridiag_team_size(n[p], num_sms);
    team[p] = g < cap ? g : cap;
  }
}

cudaError_t launch_tridiag(const EigProblem* probs_dev, EigProblem* probs_host, int count,
                           const double* S, unsigned* err, cudaStream_t st,
                           unsigned long long poll_limit) {
  int nmax = 0, grid = 0, multi = 0;
  // A team lays out its own vectors and rows only, so the launch takes the largest
  // team's sum (n <= 4096: at most 3 x 4096 doubles and the rows' 120 KB, or the 6 x
  // 4096 doubles of a team of one, which has no rows there above n = 123)
  size_t smem = 0;
  for (int p = 0; p < count; ++p) {
    EigProblem& P = probs_host[p];
    nmax = P.n > nmax ? P.n : nmax;
    const size_t rb = sizeof(double) * (size_t)tridiag_rows_per_cta(P.n, P.team_size) * P.n;
    P.srows = rb <= kTridiagSmemRowsCap;
    smem = std::max(smem, tridiag_base_smem(P.n, P.team_size) + (P.srows ? rb : 0));
    grid += P.team_size;
    multi |= P.team_size > 1;
  }
  cudaError_t e = allow_max_dyn_smem((const void*)k_tridiag);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(const_cast<EigProblem*>(probs_dev), probs_host, sizeof(EigProblem) * count,
                      cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;
  const int64_t nn = (int64_t)nmax * nmax;
  k_eig_load<<<dim3((unsigned)std::min<int64_t>((nn + 4 * TNT - 1) / (4 * TNT), 256), count), TNT, 0, st>>>(
      probs_dev, S);
  count_launches(2);
  if (multi) {
    // teams of several CTAs wait for each other: all CTAs must be resident
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tridiag, TNT, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorLaunchOutOfResources;
    void* args[] = {(void*)&probs_dev, (void*)&count, (void*)&err, (void*)&poll_limit};
    return cudaLaunchCooperativeKernel((void*)k_tridiag, dim3(grid), dim3(TNT), args, smem, st);
  }
  k_tridiag<<<grid, TNT, smem, st>>>(probs_dev, count, err, poll_limit);
  return cudaGetLastError();
}

cudaError_t launch_bisect(const EigProblem* probs_dev, int count, int nmax, int total_eigs,
                          int num_sms, cudaStream_t st) {
  // lanes per eigenvalue: about one warp per SM sub-partition in total
  int L = 32 * BNW;
  while (L > 1 && (int64_t)total_eigs * L > (int64_t)num_sms * 4 * 32) L >>= 1;
  const size_t smem = sizeof(double2) * (size_t)(nmax + 2 + (nmax + SB - 1) / SB);
  cudaError_t e = allow_max_dyn_smem((const void*)k_bisect);
  if (e != cudaSuccess) return e;
  const int per_cta = BNW * 32 / L;
  k_bisect<<<dim3((nmax + per_cta - 1) / per_cta, count), BNW * 32, smem, st>>>(probs_dev, L);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_invit(const EigProblem* probs_dev, int count, int total_vectors, cudaStream_t st) {
  if (total_vectors < 1) return cudaSuccess;
  k_invit<<<(total_vectors + 15) / 16, 32, 0, st>>>(probs_dev, count, total_vectors);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_cholqr(const EigProblem* probs_dev, const EigProblem* probs_host, int count,
                          int pass, int num_sms, cudaStream_t st, const int* info) {
  int nmax = 0;
  for (int p = 0; p < count; ++p)
    if (probs_host[p].R <= CS) nmax = probs_host[p].n > nmax ? probs_host[p].n : nmax;
  if (nmax > 0) {
    k_chol_small<<<count, TNT, 0, st>>>(probs_dev, pass);
    k_apply_small<<<dim3((nmax + AR - 1) / AR, count), TNT, 0, st>>>(probs_dev, pass);
    count_launches(2);
  }
  for (int p = 0; p < count; ++p) {
    const int R = probs_host[p].R, n = probs_host[p].n;
    if (R <= CS || (info && (info[3 * p] != 0 || info[3 * p + 1] == 0))) continue;
    const EigProblem* pd = probs_dev + p;
    if (pass == 0) {
      k_chol_far<<<(int)std::min<int64_t>(((int64_t)R * R + TNT - 1) / TNT, num_sms), TNT, 0, st>>>(pd);
      count_launches(1);
    }
    const int nb = (R + CB - 1) / CB;
    for (int b = 0; b < nb; ++b) {
      const int rest = nb - 1 - b;
      k_chol_diag<<<1, TNT, 0, st>>>(pd, b, pass);
      if (rest > 0) {
        k_chol_panel<<<rest, TNT, 0, st>>>(pd, b, pass);
        k_chol_trail<<<rest * (rest + 1) / 2, TNT, 0, st>>>(pd, b, pass);
      }
      count_launches(rest > 0 ? 3 : 1);
    }
    // one wave of CTAs where that leaves at most 16 rows each
    const int rows = std::max(4, std::min(16, (n + num_sms - 1) / num_sms));
    k_apply_big<<<(n + rows - 1) / rows, 32 * rows, 0, st>>>(pd, pass);
    count_launches(1);
  }
  return cudaGetLastError();
}

size_t eig_wy_doubles(int n) { return (size_t)wy_blocks(n) * WYB * WYB; }

cudaError_t launch_wy(const EigProblem* probs_dev, const EigProblem* one, int count, int nmax,
                      cudaStream_t st) {
  const int nb = wy_blocks(nmax);
  if (nb > 0) {
    k_wy_t<<<dim3(nb, count), 256, 0, st>>>(one ? nullptr : probs_dev, one ? *one : EigProblem{});
    count_launches(1);
  }
  return cudaGetLastError();
}

cudaError_t launch_backtransform(const EigProblem* probs_dev, int count, int total_vectors,
                                 int nmax, cudaStream_t st) {
  if (total_vectors < 1) return cudaSuccess;
  const size_t smem = sizeof(double) * (size_t)nmax;
  cudaError_t e = allow_max_dyn_smem((const void*)k_backtransform);
  if (e != cudaSuccess) return e;
  k_backtransform<<<total_vectors, 256, smem, st>>>(probs_dev, count);
  count_launches(1);
  return cudaGetLastError();
}

template <int OP, typename TOut>
static cudaError_t scalar_probe(const double* x, TOut* y, int64_t n, cudaStream_t st) {
  if (n > 0) k_scalar_probe<OP, TOut><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, y, n);
  count_launches(n > 0 ? 1 : 0);
  return cudaGetLastError();
}
cudaError_t launch_rcp64_probe(const double* x, double* y, int64_t n, cudaStream_t st) {
  return scalar_probe<0>(x, y, n, st);
}
cudaError_t launch_sqrt64_probe(const double* x, double* y, int64_t n, cudaStream_t st) {
  return scalar_probe<1>(x, y, n, st);
}
cudaError_t launch_f64_to_f32_probe(const double* x, float* y, int64_t n, cudaStream_t st) {
  return scalar_probe<2>(x, y, n, st);
}

}  // namespace tk
