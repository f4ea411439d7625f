// SIMT kernels of the ST-HOSVD path: FP64 sum of squares (Section 2.2.2),
// slab-batched Gram (Algorithm 2) and slab TTM (Algorithm 3) in FP64 or
// FP32 arithmetic, over the unfolding-free strided view (Rt, I, L) of
// Section 4.2: element (l, i, r) of the mode-n view sits at l + L*(i + I*r).
#include <algorithm>
#include <cstdio>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "gram_order.cuh"

namespace tk {

// ------------------------------------------------------------ sum of squares

// Block reduction of a thread's (sum, max|x|): partial[b] = sum of block b,
// partial[gridDim.x + b] = max of block b.  Any block size up to 1024.
__device__ __forceinline__ void block_store_sum_max(double acc, double mx, double* partial,
                                                    unsigned* nonfinite, bool bad) {
  for (int o = 16; o > 0; o >>= 1) {
    acc += __shfl_xor_sync(0xffffffffu, acc, o);
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  __shared__ double s[32], m[32];
  if ((threadIdx.x & 31) == 0) {
    s[threadIdx.x >> 5] = acc;
    m[threadIdx.x >> 5] = mx;
  }
  if (bad) atomicOr(nonfinite, 1u);
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0, tm = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      t += s[w];
      tm = fmax(tm, m[w]);
    }
    partial[blockIdx.x] = t;
    partial[gridDim.x + blockIdx.x] = tm;
  }
}

// FP64 input: one FP64 instruction per element (an FMA; it occupies the pipe for
// 64 cycles a warp, which bounds the pass: 0.69 ms for 4e8 elements against 0.47 ms
// of HBM).  max |x| and the non-finite test are integer maxima of the bit
// patterns, and four 16-byte loads are in flight per thread.  4e8 elements: 2.39 ms
// with FP64 maxima and one load, 1.53 ms with 64-bit integer ones, now 0.70 ms.
__device__ __forceinline__ void sumsq_f64(const double* __restrict__ y, int64_t n,
                                          double* __restrict__ partial,
                                          unsigned* __restrict__ nonfinite) {
  double a0 = 0.0, a1 = 0.0;
  Max64 mx;
  auto add = [&](double& acc, double v) {
    mx.add((unsigned)__double2hiint(v) & 0x7fffffffu, (unsigned)__double2loint(v));
    acc = fma(v, v, acc);
  };
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t head = (int64_t)(((uintptr_t)y & 15) / 8);      // to the first 16-byte boundary
  if (head > n) head = n;
  const int64_t nv = (n - head) / 2;
  const double2* yv = reinterpret_cast<const double2*>(y + head);
  int64_t v = tid;
  for (; v + 3 * stride < nv; v += 4 * stride) {
    double2 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = __ldcs(yv + v + u * stride);
#pragma unroll
    for (int u = 0; u < 4; ++u) { add(a0, q[u].x); add(a1, q[u].y); }
  }
  for (; v < nv; v += stride) {
    const double2 q = __ldcs(yv + v);
    add(a0, q.x);
    add(a1, q.y);
  }
  if (tid < head) add(a0, y[tid]);
  for (int64_t i = head + 2 * nv + tid; i < n; i += stride) add(a1, y[i]);
  const bool bad = mx.hi >= 0x7ff00000u;
  block_store_sum_max(a0 + a1, bad ? 0.0 : __longlong_as_double((long long)mx.get()), partial, nonfinite,
                      bad);
}

// Fixed-order reduction of `count` (sum, max) partials into out[0] (sum)
// and out[1] (max); block b: the b-th set.
__global__ void __launch_bounds__(256) k_reduce_sum(const double* __restrict__ partial, int count,
                                                    double* __restrict__ out) {
  double acc = 0.0, mx = 0.0;
  partial += 2 * (size_t)count * blockIdx.x;
  out += 2 * blockIdx.x;
  for (int i = threadIdx.x; i < count; i += blockDim.x) {
    acc += partial[i];
    mx = fmax(mx, partial[count + i]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    acc += __shfl_xor_sync(0xffffffffu, acc, o);
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  __shared__ double s[8], m[8];
  if ((threadIdx.x & 31) == 0) {
    s[threadIdx.x >> 5] = acc;
    m[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0, tm = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      t += s[w];
      tm = fmax(tm, m[w]);
    }
    out[0] = t;
    out[1] = tm;
  }
}

// Error-free FP32 sum: s + e == a + b exactly (Knuth's TwoSum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// FP32 input: x^2 = p + e exactly (p = fl(x*x), e = fma(x, x, -p)); the p
// are summed as an FP32 pair (hi, lo) with TwoSum and the pair is moved into
// the FP64 sum every 128 elements, so the result matches an FP64 sum of the
// exact squares to ~1e-15 while the kernel stays on the FP32 pipe and the
// HBM roofline.  Every FP64 instruction costs a sub-partition's FP64 pipe 64
// cycles per warp, so the per-element path has none: the moves into FP64
// convert on integer bits, max |x| and the non-finite test are integer
// maxima of the bit patterns, and a group of 16 whose largest |x| is at
// least 2^64 (an FP32 square could overflow) or nonzero and below 2^-60 (its
// squares would underflow FP32) is squared in FP64 on a warp-uniform branch
// (in a group with a larger value, squares below 2^-120 are ~2^-96 of it).
__device__ __forceinline__ double f32_bits_to_f64(float x) {
  // exact for normal x; zero and subnormals (below 1.2e-38) become 0
  const unsigned u = __float_as_uint(x);
  const unsigned ex = (u >> 23) & 0xffu;
  const unsigned long long b = (unsigned long long)(u >> 31) << 63 |
                               (unsigned long long)(ex + 1023u - 127u) << 52 |
                               (unsigned long long)(u & 0x7fffffu) << 29;
  return ex == 0u ? 0.0 : __longlong_as_double((long long)b);
}

struct SumSqF32 {
  double acc = 0.0;
  float hi = 0.f, lo = 0.f;
  unsigned mxb = 0;     // max |x| as bits; >= 0x7f800000: NaN or Inf seen
  __device__ __forceinline__ void add_fast(float x) {
    const float p = x * x;
    const float e = fmaf(x, x, -p);
    float s, err;
    two_sum(hi, p, s, err);
    hi = s;
    lo += err + e;
  }
  __device__ __forceinline__ void add(float x) {   // tails: per-element test
    const unsigned b = __float_as_uint(x) & 0x7fffffffu;
    mxb = max(mxb, b);
    if (b >= 0x5f800000u || (b != 0u && b < 0x21800000u)) acc = fma((double)x, (double)x, acc);
    else add_fast(x);
  }
  __device__ __forceinline__ void flush() {
    acc += f32_bits_to_f64(hi) + f32_bits_to_f64(lo);
    hi = lo = 0.f;
  }
};

__device__ __forceinline__ void sumsq_f32(const float* __restrict__ y, int64_t n,
                                          double* __restrict__ partial,
                                          unsigned* __restrict__ nonfinite) {
  SumSqF32 s;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t head = (int64_t)(((16 - ((uintptr_t)y & 15)) & 15) / 4);
  if (head > n) head = n;
  const int64_t nv = (n - head) / 4;
  const float4* yv = reinterpret_cast<const float4*>(y + head);
  // four independent 16-byte loads in flight per thread per iteration
  int64_t v = tid;
  int groups = 0;
  for (; v + 3 * stride < nv; v += 4 * stride) {
    float4 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = __ldcs(yv + v + u * stride);
    unsigned gm = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      gm = max(gm, __float_as_uint(q[u].x) & 0x7fffffffu);
      gm = max(gm, __float_as_uint(q[u].y) & 0x7fffffffu);
      gm = max(gm, __float_as_uint(q[u].z) & 0x7fffffffu);
      gm = max(gm, __float_as_uint(q[u].w) & 0x7fffffffu);
    }
    s.mxb = max(s.mxb, gm);
    if (__any_sync(__activemask(), gm >= 0x5f800000u || (gm != 0u && gm < 0x21800000u))) {
#pragma unroll
      for (int u = 0; u < 4; ++u) { s.add(q[u].x); s.add(q[u].y); s.add(q[u].z); s.add(q[u].w); }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        s.add_fast(q[u].x); s.add_fast(q[u].y); s.add_fast(q[u].z); s.add_fast(q[u].w);
      }
    }
    if (++groups == 8) { s.flush(); groups = 0; }
  }
  for (; v < nv; v += stride) {
    const float4 q = __ldcs(yv + v);
    s.add(q.x); s.add(q.y); s.add(q.z); s.add(q.w);
  }
  for (int64_t i = tid; i < head; i += stride) s.add(y[i]);
  for (int64_t i = head + 4 * nv + tid; i < n; i += stride) s.add(y[i]);
  s.flush();
  const bool bad = s.mxb >= 0x7f800000u;
  block_store_sum_max(s.acc, bad ? 0.0 : (double)__uint_as_float(s.mxb), partial, nonfinite, bad);
}

__global__ void __launch_bounds__(256) k_sumsq_f64(const double* __restrict__ y, int64_t n,
                                                   double* __restrict__ partial,
                                                   unsigned* __restrict__ nonfinite) {
  sumsq_f64(y, n, partial, nonfinite);
}
__global__ void __launch_bounds__(256) k_sumsq_f32(const float* __restrict__ y, int64_t n,
                                                   double* __restrict__ partial,
                                                   unsigned* __restrict__ nonfinite) {
  sumsq_f32(y, n, partial, nonfinite);
}
// The tensors of a batch side by side (blockIdx.y): one after the other, 64 of them with
// their reductions took 1.5 ms for 0.28 ms of HBM, 0.44 ms side by side.
template <typename T>
__global__ void __launch_bounds__(256) k_sumsq_batched(const NormItem* __restrict__ items,
                                                       double* __restrict__ partial,
                                                       unsigned* __restrict__ nonfinite) {
  const NormItem it = items[blockIdx.y];
  double* p = partial + 2 * (size_t)gridDim.x * blockIdx.y;
  if constexpr (sizeof(T) == 8) sumsq_f64(static_cast<const T*>(it.y), it.n, p, nonfinite + blockIdx.y);
  else sumsq_f32(static_cast<const T*>(it.y), it.n, p, nonfinite + blockIdx.y);
}

cudaError_t launch_sumsq_batched(const NormItem* items_dev, tucker_dtype dt, int count, int nblocks,
                                 double* partial, unsigned* nonfinite, double* out, cudaStream_t st) {
  const dim3 grid((unsigned)nblocks, (unsigned)count);
  if (dt == TUCKER_F64) k_sumsq_batched<double><<<grid, 256, 0, st>>>(items_dev, partial, nonfinite);
  else k_sumsq_batched<float><<<grid, 256, 0, st>>>(items_dev, partial, nonfinite);
  k_reduce_sum<<<count, 256, 0, st>>>(partial, nblocks, out);
  count_launches(2);
  return cudaGetLastError();
}

// Row maxima of the column-major I0 x ncols view (each row's max |x| as FP32
// bits, atomicMax into rowmax_bits[I0], zeroed by the caller), SUM: and the same
// sum of squares.  A thread owns W rows (VEC: 4, one 16-byte load, I0 % 4 == 0 and y
// 16-byte aligned; else 1), tq threads a column (and several rounds of tq when a
// block is not enough: `passes`), and a block takes `groups` columns at a time, so
// that short columns fill it as well: I0 = 256, 5.9 GB: 1.39 ms with one column a
// block, now 0.95 ms (0.87 ms of HBM).  The columns blockIdx.x * groups + group,
// + gridDim.x * groups, ...; U of them in flight per thread.  I0 <= 8192.
constexpr int kRmThreads = 256;               // block of several columns
template <bool VEC, bool SUM>
__global__ void __launch_bounds__(512) k_sumsq_rowmax_f32(const float* __restrict__ y, int64_t I0,
                                                           int64_t ncols, int passes, int tq,
                                                           int groups, double* __restrict__ partial,
                                                           unsigned* __restrict__ nonfinite,
                                                           unsigned* __restrict__ rowmax_bits) {
  constexpr int W = VEC ? 4 : 1, U = VEC ? 8 : 16;
  __shared__ unsigned s_max[kRmThreads / 2 * W];      // groups > 1: tq <= kRmThreads / 2
  SumSqF32 s;
  int done = 0;
  const int grp = (int)threadIdx.x / tq, t = (int)threadIdx.x - grp * tq;
  const int64_t cstep = (int64_t)gridDim.x * groups;
  if (groups > 1) {
    for (int i = threadIdx.x; i < kRmThreads / 2 * W; i += blockDim.x) s_max[i] = 0u;
    __syncthreads();
  }
  for (int pass = 0; pass < passes; ++pass) {
    const int64_t r = W * ((int64_t)t + (int64_t)pass * tq);
    const bool active = r < I0 && grp < groups;
    unsigned rm[W];
#pragma unroll
    for (int w = 0; w < W; ++w) rm[w] = 0u;
    struct Vals { float v[W]; };
    auto load = [&](int64_t c) {
      Vals q;
      const float* p = y + r + I0 * c;
      if constexpr (VEC) {
        const float4 f = __ldcs(reinterpret_cast<const float4*>(p));
        q.v[0] = f.x; q.v[1] = f.y; q.v[2] = f.z; q.v[3] = f.w;
      } else {
        q.v[0] = __ldcs(p);
      }
      return q;
    };
    int64_t c = active ? (int64_t)blockIdx.x * groups + grp : ncols;
    for (; c + (U - 1) * cstep < ncols; c += U * cstep) {
      Vals q[U];
#pragma unroll
      for (int u = 0; u < U; ++u) q[u] = load(c + u * cstep);
      unsigned gm = 0;
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const unsigned b = __float_as_uint(q[u].v[w]) & 0x7fffffffu;
          rm[w] = max(rm[w], b);
          if (SUM) gm = max(gm, b);
        }
      if constexpr (SUM) {
        s.mxb = max(s.mxb, gm);
        if (__any_sync(__activemask(), gm >= 0x5f800000u || (gm != 0u && gm < 0x21800000u))) {
#pragma unroll
          for (int u = 0; u < U; ++u)
#pragma unroll
            for (int w = 0; w < W; ++w) s.add(q[u].v[w]);
        } else {
#pragma unroll
          for (int u = 0; u < U; ++u)
#pragma unroll
            for (int w = 0; w < W; ++w) s.add_fast(q[u].v[w]);
        }
        if (++done == 128 / (U * W)) { s.flush(); done = 0; }
      }
    }
    for (; c < ncols; c += cstep) {
      const Vals q = load(c);
#pragma unroll
      for (int w = 0; w < W; ++w) {
        rm[w] = max(rm[w], __float_as_uint(q.v[w]) & 0x7fffffffu);
        if (SUM) s.add(q.v[w]);
      }
    }
    if (active) {
#pragma unroll
      for (int w = 0; w < W; ++w)
        if (rm[w]) atomicMax(groups > 1 ? s_max + r + w : rowmax_bits + r + w, rm[w]);
    }
  }
  if (groups > 1) {
    __syncthreads();
    for (int i = threadIdx.x; i < I0; i += blockDim.x)
      if (s_max[i]) atomicMax(rowmax_bits + i, s_max[i]);
  }
  if constexpr (SUM) {
    s.flush();
    const bool bad = s.mxb >= 0x7f800000u;
    block_store_sum_max(s.acc, bad ? 0.0 : (double)__uint_as_float(s.mxb), partial, nonfinite, bad);
  }
}

cudaError_t launch_sumsq_rowmax(const float* y, int64_t I0, int64_t ncols, double* partial,
                                int nblocks, unsigned* nonfinite, unsigned* rowmax_bits, double* out,
                                cudaStream_t st) {
  if (I0 > 8192 || I0 < 1 || ((uintptr_t)y & 3) != 0) return cudaErrorInvalidValue;
  const bool vec = I0 % 4 == 0 && ((uintptr_t)y & 15) == 0;
  // threads per column: as few passes as a 512-thread block allows, the rows
  // spread evenly over them
  const int64_t units = vec ? I0 / 4 : I0;
  const int passes = (int)((units + 511) / 512);
  const int tq = (int)((units + passes - 1) / passes);
  const int groups = tq <= 64 ? kRmThreads / tq : 1;
  const int threads = (tq * groups + 31) / 32 * 32;
  // fewer blocks rather than columns taken one by one
  const int64_t full = (ncols + (int64_t)groups * (vec ? 8 : 16) - 1) / ((int64_t)groups * (vec ? 8 : 16));
  nblocks = (int)std::min<int64_t>(nblocks, std::max<int64_t>(full, 1));
  auto run = [&](auto V, auto S) {
    k_sumsq_rowmax_f32<decltype(V)::value, decltype(S)::value><<<nblocks, threads, 0, st>>>(
        y, I0, ncols, passes, tq, groups, partial, nonfinite, rowmax_bits);
  };
  using yes = std::true_type;
  using no = std::false_type;
  count_launches(1);
  if (out) {
    if (vec) run(yes(), yes());
    else run(no(), yes());
    k_reduce_sum<<<1, 256, 0, st>>>(partial, nblocks, out);
    count_launches(1);
  } else {
    if (vec) run(yes(), no());
    else run(no(), no());
  }
  return cudaGetLastError();
}

cudaError_t launch_sumsq(const void* y, tucker_dtype dt, int64_t n, double* partial, int nblocks,
                         unsigned* nonfinite, double* out, cudaStream_t st) {
  count_launches(2);
  if (dt == TUCKER_F64)
    k_sumsq_f64<<<nblocks, 256, 0, st>>>((const double*)y, n, partial, nonfinite);
  else
    k_sumsq_f32<<<nblocks, 256, 0, st>>>((const float*)y, n, partial, nonfinite);
  k_reduce_sum<<<1, 256, 0, st>>>(partial, nblocks, out);
  return cudaGetLastError();
}

// b[i] += a[i] (FP64), grid-stride.
__global__ void k_add_f64(const double* __restrict__ a, double* __restrict__ b, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    b[i] += a[i];
}

cudaError_t launch_add_f64(const double* a, double* b, int64_t n, int num_sms, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int nb = (int)std::min<int64_t>((n + 255) / 256, (int64_t)num_sms * 4);
  count_launches(1);
  k_add_f64<<<nb, 256, 0, st>>>(a, b, n);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ Gram

constexpr int GT = 64;    // Gram output tile
constexpr int GBK = 16;   // K-block

// Loads the (GBK x GT) panel of rows [i0, i0+GT) for K-block kb into regs.
template <typename TIn, typename TC>
__device__ __forceinline__ void gram_load(const TIn* __restrict__ y, const KGeom& g, int64_t kb,
                                          int64_t i0, TC (&reg)[4]) {
  const int tid = threadIdx.x;
  if (g.L == 1) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int idx = tid + 256 * e;
      int ii = idx % GT, kk = idx / GT;
      int64_t r = kb * GBK + kk, i = i0 + ii;
      reg[e] = (r < g.Rt && i < g.I) ? (TC)y[i + g.I * r] : (TC)0;
    }
  } else {
    int64_t r = kb / g.nLB;
    int64_t lbeg, lend;
    lblock_range(g, kb - r * g.nLB, GBK, lbeg, lend);
    const TIn* base = y + g.L * g.I * r;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int idx = tid + 256 * e;
      int kk = idx % GBK, ii = idx / GBK;
      int64_t l = lbeg + kk, i = i0 + ii;
      reg[e] = (l < lend && i < g.I) ? (TC)base[l + g.L * i] : (TC)0;
    }
  }
}

template <typename TC>
__device__ __forceinline__ void gram_store(TC (*sm)[GT + 1], const KGeom& g, const TC (&reg)[4]) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    int idx = tid + 256 * e;
    int ii, kk;
    if (g.L == 1) { ii = idx % GT; kk = idx / GT; }
    else { kk = idx % GBK; ii = idx / GBK; }
    sm[kk][ii] = reg[e];
  }
}

// One CTA: lower-triangle tile (ta >= tb) of S over its K-blocks.  TC is the
// product type.  FP64 products are summed in FP64.  FP32 products are summed
// by FMA in FP32 within a chunk, and the chunk sums are combined as an exact
// FP32 pair (TwoSum), which keeps the FP64 pipe (1/62 of the FP32 rate on
// this part) out of the inner loop.  Writes the FP64 partial tile to
// part[(ks * ntiles + tile) * GT * GT].
template <typename TIn, typename TC>
__global__ void __launch_bounds__(256) k_gram_simt(const TIn* __restrict__ y, KGeom g, int ntiles,
                                                   int ksplit, double* __restrict__ part) {
  __shared__ TC As[GBK][GT + 1];
  __shared__ TC Bs[GBK][GT + 1];
  const int tile = blockIdx.x;
  const int ks = blockIdx.y;
  // tile -> (ta, tb), ta >= tb, row-major over the lower triangle
  int ta = (int)((sqrtf(8.f * tile + 1.f) - 1.f) * 0.5f);
  while ((ta + 1) * (ta + 2) / 2 <= tile) ++ta;
  while (ta * (ta + 1) / 2 > tile) --ta;
  const int tb = tile - ta * (ta + 1) / 2;
  const bool diag = (ta == tb);
  const int64_t ia0 = (int64_t)ta * GT, ib0 = (int64_t)tb * GT;
  const KOrder ord = make_korder(g, ks, ksplit);

  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  TC acc[4][4];
  float hi[4][4], lo[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) { acc[u][v] = (TC)0; hi[u][v] = 0.f; lo[u][v] = 0.f; }

  TC ra[4], rb[4];
  bool end_cur = false, end_next = false;
  int64_t kb = 0;
  if (ord.count > 0) {
    kb = korder_block(g, ord, 0, end_cur);
    gram_load<TIn, TC>(y, g, kb, ia0, ra);
    if (!diag) gram_load<TIn, TC>(y, g, kb, ib0, rb);
  }
  for (int64_t idx = 0; idx < ord.count; ++idx) {
    gram_store<TC>(As, g, ra);
    if (!diag) gram_store<TC>(Bs, g, rb);
    __syncthreads();
    if (idx + 1 < ord.count) {
      const int64_t kbn = korder_block(g, ord, idx + 1, end_next);
      gram_load<TIn, TC>(y, g, kbn, ia0, ra);
      if (!diag) gram_load<TIn, TC>(y, g, kbn, ib0, rb);
    }
    TC (*Bp)[GT + 1] = diag ? As : Bs;
    // FP32: the 16 products of a K-block are summed into a fresh register
    // first and only that block sum enters the chunk accumulator.  Squares
    // x^2 pile up near zero (chi-square), and adding them one by one to a
    // large FP32 sum rounds with a negative bias ~ (terms in the sum)^1.5;
    // 16-term block sums have a smooth density and round without bias.  The
    // block runs from its last K to its first: in row mode its 16 l are
    // consecutive indices of a truncated mode whose energy falls with l, so
    // the products are added in increasing size.
    TC t[4][4];
#pragma unroll
    for (int kq = 0; kq < GBK; ++kq) {
      const int kk = GBK - 1 - kq;
      TC a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = As[kk][ty + 16 * u];
#pragma unroll
      for (int v = 0; v < 4; ++v) b[v] = Bp[kk][tx + 16 * v];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          if constexpr (sizeof(TC) == 4)
            t[u][v] = (kq == 0) ? a[u] * b[v] : fma(a[u], b[v], t[u][v]);
          else
            acc[u][v] = fma(a[u], b[v], acc[u][v]);
        }
    }
    if constexpr (sizeof(TC) == 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] += t[u][v];
    }
    __syncthreads();
    if constexpr (sizeof(TC) == 4) {
      if (end_cur) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            float s, e;
            two_sum(hi[u][v], (float)acc[u][v], s, e);
            hi[u][v] = s;
            lo[u][v] += e;
            acc[u][v] = (TC)0;
          }
      }
    }
    end_cur = end_next;
  }
  double* out = part + ((int64_t)ks * ntiles + tile) * GT * GT;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v)
      out[(ty + 16 * u) * GT + tx + 16 * v] =
          (double)hi[u][v] + (double)lo[u][v] + (double)acc[u][v];
}

// S[i][j] = S[j][i] = sum over ks (fixed order) of the partial tiles.
__global__ void k_gram_reduce(const double* __restrict__ part, int ntiles, int ksplit, int64_t I,
                              double* __restrict__ S) {
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)ntiles * GT * GT) return;
  int tile = (int)(idx / (GT * GT));
  int e = (int)(idx % (GT * GT));
  int ta = (int)((sqrtf(8.f * tile + 1.f) - 1.f) * 0.5f);
  while ((ta + 1) * (ta + 2) / 2 <= tile) ++ta;
  while (ta * (ta + 1) / 2 > tile) --ta;
  int tb = tile - ta * (ta + 1) / 2;
  int64_t i = (int64_t)ta * GT + e / GT, j = (int64_t)tb * GT + e % GT;
  if (i >= I || j >= I) return;
  if (ta == tb && j > i) return;  // diagonal tile: write its lower half (and mirror)
  double s = 0.0;
  for (int k = 0; k < ksplit; ++k) s += part[((int64_t)k * ntiles + tile) * GT * GT + e];
  S[i * I + j] = s;
  S[j * I + i] = s;
}

GramPlan plan_gram_simt(int64_t L, int64_t I, int64_t Rt, int num_sms, int64_t L0) {
  GramPlan p;
  KGeom g = make_kgeom(L, I, Rt, GBK, L0);
  int T = (int)((I + GT - 1) / GT);
  p.ntiles = T * (T + 1) / 2;
  int64_t want = ((int64_t)num_sms * 4 + p.ntiles - 1) / p.ntiles;
  int64_t cap = (int64_t)(256ll << 20) / ((int64_t)p.ntiles * GT * GT * 8);
  if (want > cap) want = cap;
  if (want > g.NKB) want = g.NKB;
  if (want < 1) want = 1;
  p.ksplit = (int)want;
  p.scratch_bytes = (size_t)p.ksplit * p.ntiles * GT * GT * sizeof(double);
  return p;
}

// Same split as plan_gram_simt, with the partial-tile scratch held to at most
// max_bytes (fewer K-splits).  ok == 0 when even one split does not fit.
GramPlan plan_gram_simt_capped(int64_t L, int64_t I, int64_t Rt, int num_sms, size_t max_bytes,
                               int* ok, int64_t L0) {
  GramPlan p = plan_gram_simt(L, I, Rt, num_sms, L0);
  const size_t per_split = (size_t)p.ntiles * GT * GT * sizeof(double);
  *ok = per_split <= max_bytes;
  if (!*ok) return p;
  if (p.scratch_bytes > max_bytes) {
    p.ksplit = (int)(max_bytes / per_split);
    p.scratch_bytes = (size_t)p.ksplit * per_split;
  }
  return p;
}

cudaError_t launch_gram_simt(const void* y, tucker_dtype dt, bool fp64, int64_t L, int64_t I,
                             int64_t Rt, int64_t L0, const GramPlan& p, double* scratch, double* S,
                             cudaStream_t st) {
  KGeom g = make_kgeom(L, I, Rt, GBK, L0);
  dim3 grid(p.ntiles, p.ksplit);
  count_launches(2);
  if (dt == TUCKER_F64) {
    if (fp64) k_gram_simt<double, double><<<grid, 256, 0, st>>>((const double*)y, g, p.ntiles, p.ksplit, scratch);
    else k_gram_simt<double, float><<<grid, 256, 0, st>>>((const double*)y, g, p.ntiles, p.ksplit, scratch);
  } else {
    if (fp64) k_gram_simt<float, double><<<grid, 256, 0, st>>>((const float*)y, g, p.ntiles, p.ksplit, scratch);
    else k_gram_simt<float, float><<<grid, 256, 0, st>>>((const float*)y, g, p.ntiles, p.ksplit, scratch);
  }
  int64_t tot = (int64_t)p.ntiles * GT * GT;
  k_gram_reduce<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(scratch, p.ntiles, p.ksplit, I, S);
  return cudaGetLastError();
}

// ------------------------------------------------------------------- TTM
//
// Z (K x M) = A (K x I) * Y (I x M), M = the (l, r) pairs of the slab view, l
// fastest.  A block of four warps owns MT m and KT outputs, KT = 8, 16, 24 or 32
// (ttm_tile_outputs; few outputs are what a truncation leaves).  WK warps share the outputs and 4 / WK the m; a thread owns MM
// m (lane + 32 j) and KK = KT / WK outputs of each.  The sums run over i in order.
//   Stages of 32 i, two in turn, through registers a quarter at a time between the
// products (16-byte accesses where the view allows).  L > 1: Y as it lies, m fastest.
// L == 1: a row of 32 i per m, padded by 16 bytes, so that 16-byte reads of one m per
// lane do not conflict; zt writes Z transposed (z[m + M k]), else the block's Z
// goes through shared memory, k being fastest.
//   Bound: instructions (FP64: its pipe).  FP32 products go two outputs at a time
// (f32x2); addresses advance by additions, bounds are tested only in tiles that need
// it (64-bit comparisons run at the FP64 pipe's rate); four blocks per SM (two
// blocks of 256 m took 1.2 times as long).  Measured, with one 64 x 64 tile per block
// before: I = 301, M = 287,000, K = 20 (345 MB) 540 -> 183 us; I = 200, M = 56,000 82 -> 31;
// row view 3.5e6 x 32 to 10 638 -> 226; I = 54, M = 32,000 to 502 106 -> 81; FP64 I = 40,
// M = 1500, K = 5 55 -> 17.
constexpr int TNT = 128;                  // threads
constexpr int TIC = 32;                   // i per stage

// dynamic shared memory: two stages of Y, then (L == 1) the block's Z
template <typename TIn, typename TC, int KT, int MT, bool COL>
constexpr size_t ttm_smem() {
  return COL ? std::max(2 * (size_t)MT * (TIC * sizeof(TIn) + 16), (size_t)MT * (KT + 1) * sizeof(TC))
             : 2 * (size_t)MT * TIC * sizeof(TIn);
}

template <typename TIn, typename TOut, typename TC, int KT, int WK, int MM, bool COL>
__global__ void __launch_bounds__(TNT, sizeof(TC) == 4 ? 4 : 2)
    k_ttm(const TIn* __restrict__ y, int64_t L, int64_t I,
                                             int64_t M, const double* __restrict__ A, int64_t K,
                                             int64_t lda, int a_rowmajor,
                                             const float* __restrict__ A32, TOut* __restrict__ z,
                                             int zt) {
  constexpr int NW = TNT / 32, MT = NW / WK * 32 * MM, KK = KT / WK;
  constexpr int KP = KT + 16 / (int)sizeof(TC);                     // padded, 16-byte rows
  constexpr int VY = 16 / (int)sizeof(TIn), YP = TIC + VY;
  __shared__ __align__(16) TC As[2][TIC][KP];
  extern __shared__ __align__(16) unsigned char ttm_sm[];
  TIn* Ys = reinterpret_cast<TIn*>(ttm_sm);                         // COL: [2][MT][YP], else [2][TIC][MT]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // (tiles of outputs beyond the 65,535 that a grid's y counts go along z)
  const int64_t m0 = (int64_t)blockIdx.x * MT;
  const int64_t k0 = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * KT;
  if (k0 >= K) return;
  const int nk = (int)min((int64_t)KT, K - k0);

  // entries of A for i0..: threads along whichever index is contiguous
  constexpr int AE = TIC * KT / TNT;
  const bool ifast = A32 || a_rowmajor;
  auto load_a = [&](double (&v)[AE], int64_t i0) {
#pragma unroll
    for (int e = 0; e < AE; ++e) {
      const int idx = tid + TNT * e;
      const int ii = ifast ? idx % TIC : idx / KT, kk = ifast ? idx / TIC : idx % KT;
      const int64_t i = i0 + ii, k = k0 + kk;
      v[e] = 0.0;
      if (kk < nk && i < I) {
        if (sizeof(TC) == 4 && A32) v[e] = __hiloint2double(0, __float_as_int(A32[k * I + i]));   // bits
        else v[e] = a_rowmajor ? A[k * lda + i] : A[k + lda * i];
      }
    }
  };
  auto store_a = [&](const double (&v)[AE], int b) {
#pragma unroll
    for (int e = 0; e < AE; ++e) {
      const int idx = tid + TNT * e;
      const int ii = ifast ? idx % TIC : idx / KT, kk = ifast ? idx / TIC : idx % KT;
      if constexpr (sizeof(TC) == 4) As[b][ii][kk] = A32 ? __int_as_float(__double2loint(v[e])) : f64_to_f32(v[e]);
      else As[b][ii][kk] = v[e];
    }
  };
  // a stage of Y in four parts of PB values per thread; 16-byte accesses: chunk c of
  // the stage, CPR per row of it, by thread c % TNT
  constexpr int PB = MT * TIC / TNT / 4, CPR = (COL ? TIC : MT) / VY, ME = MT / TNT;
  const bool y16 = (COL ? I : L) % VY == 0 && ((uintptr_t)y & 15) == 0;
  const int cq = y16 ? tid % CPR * VY : (COL ? lane : tid);         // first column
  int64_t yo[COL ? 1 : ME] = {};                                    // ROW: offsets of this thread's m
  if constexpr (!COL) {
#pragma unroll
    for (int e = 0; e < ME; ++e) {
      const int64_t m = m0 + cq + (y16 ? 0 : TNT * e), r = m / L;
      yo[e] = m < M ? m - r * L + L * I * r : -1;
    }
  }
  auto row16 = [&](int q, int e) { return (q * (PB / VY) + e) * (TNT / CPR) + tid / CPR; };
  using V16 = typename std::conditional<sizeof(TIn) == 4, float4, double2>::type;
  const bool mfull = m0 + MT <= M;
  const int64_t step = COL ? I * (y16 ? TNT / CPR : NW) : L * (y16 ? TNT / CPR : 1);   // per row copied
  auto load_y = [&](TIn* v, int q, int64_t i0) {
    const bool full = mfull && i0 + TIC <= I;             // else every access is tested
    if (y16) {
      const int r0 = row16(q, 0);
      const TIn* p = COL ? y + I * (m0 + r0) + i0 + cq : y + yo[0] + L * (i0 + r0);
#pragma unroll
      for (int e = 0; e < PB / VY; ++e, p += step) {
        const int r = r0 + e * (TNT / CPR);
        const bool ok = full || (COL ? (i0 + cq < I && m0 + r < M) : (i0 + r < I && yo[0] >= 0));
        *reinterpret_cast<V16*>(v + VY * e) = ok ? __ldg(reinterpret_cast<const V16*>(p)) : V16{};
      }
    } else {
      const int r0 = COL ? warp + NW * q * PB : q * PB / ME;
      const TIn* p[COL ? 1 : ME];
#pragma unroll
      for (int c = 0; c < (COL ? 1 : ME); ++c)
        p[c] = COL ? y + I * (m0 + r0) + i0 + cq : y + yo[c] + L * (i0 + r0);
      if (full) {
#pragma unroll
        for (int e = 0; e < PB; ++e) {
          v[e] = __ldg(p[COL ? 0 : e % ME]);
          p[COL ? 0 : e % ME] += step;
        }
      } else {
#pragma unroll
        for (int e = 0; e < PB; ++e) {
          const int r = COL ? r0 + NW * e : r0 + e / ME;
          const bool ok = COL ? (i0 + cq < I && m0 + r < M) : (i0 + r < I && yo[e % ME] >= 0);
          v[e] = ok ? __ldg(p[COL ? 0 : e % ME]) : (TIn)0;
          p[COL ? 0 : e % ME] += step;
        }
      }
    }
  };
  auto store_y = [&](const TIn* v, int q, int b) {
    TIn* d = Ys + (size_t)b * (COL ? MT * YP : MT * TIC) + cq;
    constexpr int P = COL ? YP : MT;
    if (y16) {
#pragma unroll
      for (int e = 0; e < PB / VY; ++e)
        *reinterpret_cast<V16*>(d + row16(q, e) * P) = *reinterpret_cast<const V16*>(v + VY * e);
    } else {
#pragma unroll
      for (int e = 0; e < PB; ++e) {
        const int r = COL ? warp + NW * (q * PB + e) : (q * PB + e) / ME;
        d[r * P + (COL ? 0 : TNT * (e % ME))] = v[e];
      }
    }
  };

  // this thread's outputs kq.. and m (within the block) mq + 32 j
  const int kq = warp % WK * KK, mq = warp / WK * 32 * MM + lane;
  TC acc[MM][KK];
#pragma unroll
  for (int j = 0; j < MM; ++j)
#pragma unroll
    for (int k = 0; k < KK; ++k) acc[j][k] = (TC)0;
  auto mac = [&](const TC* a, const TC (&v)[MM]) {
    __align__(16) TC av[KK];
    constexpr int VB = KK * sizeof(TC) % 16 == 0 ? 16 : 8;
#pragma unroll
    for (int k = 0; k < KK; k += VB / (int)sizeof(TC)) {
      if constexpr (VB == 16) *reinterpret_cast<float4*>(av + k) = *reinterpret_cast<const float4*>(a + k);
      else *reinterpret_cast<float2*>(av + k) = *reinterpret_cast<const float2*>(a + k);
    }
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      if constexpr (sizeof(TC) == 4) {
#pragma unroll
        for (int k = 0; k < KK; k += 2) {
          const float2 r = fma2(make_float2(av[k], av[k + 1]), make_float2(v[j], v[j]),
                                make_float2(acc[j][k], acc[j][k + 1]));
          acc[j][k] = r.x;
          acc[j][k + 1] = r.y;
        }
      } else {
#pragma unroll
        for (int k = 0; k < KK; ++k) acc[j][k] = fma(av[k], v[j], acc[j][k]);
      }
    }
  };

  const int64_t nst = (I + TIC - 1) / TIC;
  {
    __align__(16) TIn v[2][PB];
    double av[AE];
    load_y(v[0], 0, 0);
    load_y(v[1], 1, 0);
    load_a(av, 0);
    store_y(v[0], 0, 0);
    store_y(v[1], 1, 0);
    load_y(v[0], 2, 0);
    load_y(v[1], 3, 0);
    store_a(av, 0);
    store_y(v[0], 2, 0);
    store_y(v[1], 3, 0);
  }
  for (int64_t s = 0; s < nst; ++s) {
    const int b = (int)(s & 1);
    const int ni = (int)min((int64_t)TIC, I - s * TIC);             // (past I: zeros)
    const bool more = s + 1 < nst;
    __syncthreads();                      // stage s is there, stage s - 1 is used up
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
      __align__(16) TIn nv[PB];
      double av[AE];
      if (more) {
        load_y(nv, q, (s + 1) * TIC);
        if (q == 0) load_a(av, (s + 1) * TIC);
      }
      constexpr int QI = TIC / 4;
      if (QI * q < ni) {
        if constexpr (COL) {
          const TIn* ys = Ys + ((size_t)b * MT + mq) * YP + QI * q;
#pragma unroll 1
          for (int i = 0; i < QI; i += VY) {
            __align__(16) TIn x[MM][VY];
#pragma unroll
            for (int j = 0; j < MM; ++j)
              *reinterpret_cast<V16*>(x[j]) = *reinterpret_cast<const V16*>(ys + 32 * j * YP + i);
#pragma unroll
            for (int w = 0; w < VY; ++w) {
              TC v[MM];
#pragma unroll
              for (int j = 0; j < MM; ++j) v[j] = (TC)x[j][w];
              mac(&As[b][QI * q + i + w][kq], v);
            }
          }
        } else {
          const TIn* ys = Ys + (size_t)b * MT * TIC + QI * q * MT + mq;
#pragma unroll 4
          for (int i = 0; i < QI; ++i) {
            TC v[MM];
#pragma unroll
            for (int j = 0; j < MM; ++j) v[j] = (TC)ys[i * MT + 32 * j];
            mac(&As[b][QI * q + i][kq], v);
          }
        }
      }
      if (more) {
        store_y(nv, q, b ^ 1);
        if (q == 0) store_a(av, b ^ 1);
      }
    }
  }
  if (COL && !zt) __syncthreads();

  if (COL && !zt) {
    // z[k + K m]: through shared memory, lanes along k
    TC* zs = reinterpret_cast<TC*>(ttm_sm);                         // [MT][KT + 1]
    constexpr int ZP = KT + 1;
#pragma unroll
    for (int j = 0; j < MM; ++j)
#pragma unroll
      for (int k = 0; k < KK; ++k) zs[(mq + 32 * j) * ZP + kq + k] = acc[j][k];
    __syncthreads();
    constexpr int RPW = KT >= 24 ? 1 : 32 / KT;                     // rows of m per warp
    const int k = KT >= 24 ? lane : lane % KT, sub = KT >= 24 ? 0 : lane / KT;
    const int mc = (int)min((int64_t)MT, M - m0);
    if (k < nk) {
      TOut* zr = z + K * m0 + k0 + k;
      for (int m = warp * RPW + sub; m < mc; m += NW * RPW) zr[K * m] = (TOut)zs[m * ZP + k];
    }
  } else {
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      const int64_t m = m0 + mq + 32 * j;
      if (m >= M) continue;
      const int64_t r = COL ? 0 : m / L;
      TOut* zr = z + (m - r * L) + (COL ? 0 : L * K * r) + (COL ? M : L) * (k0 + kq);
#pragma unroll
      for (int k = 0; k < KK; ++k)
        if (kq + k < nk) zr[(COL ? M : L) * k] = (TOut)acc[j][k];
    }
  }
}

constexpr int TT = 64;    // output tile (k and m)
constexpr int TBI = 16;   // contraction step

// FP32 arithmetic on FP64 input or output, and FP32 row views of few rows and many
// outputs (ttm_wide_tiles): a 64 x 64 tile per block.
// Z (K x M) = A (K x I) * Y (I x M), M = the (r, l) pairs of the slab view.
// Row mode (L > 1): an m-tile is 64 consecutive l of one slab.  Column mode
// (L == 1): an m-tile is 64 consecutive slabs; zt writes Z transposed
// (z[r + Rt k], slab fastest: the new mode last).
template <typename TIn, typename TOut, typename TC>
__global__ void __launch_bounds__(256) k_ttm_simt(const TIn* __restrict__ y, int64_t L, int64_t I,
                                                  int64_t Rt, int64_t nLT,
                                                  const double* __restrict__ A, int64_t K,
                                                  int64_t lda, int a_rowmajor,
                                                  const float* __restrict__ A32,
                                                  TOut* __restrict__ z, int zt) {
  __shared__ TC As[TBI][TT + 1];   // As[i][k]
  __shared__ TC Ys[TBI][TT + 1];   // Ys[i][m]
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  // output coordinates of this thread: the index that is contiguous in Z goes
  // to consecutive threads (k in column mode, l in row mode)
  const bool kfast = (L == 1) && !zt;
  const int kq = kfast ? tx : ty, mq = kfast ? ty : tx;
  const int64_t mt = blockIdx.x;
  const int64_t k0 = (int64_t)blockIdx.y * TT;
  int64_t r0, l0;
  if (L == 1) { r0 = mt * TT; l0 = 0; }
  else { r0 = mt / nLT; l0 = (mt - r0 * nLT) * TT; }
  const TIn* ybase = (L == 1) ? y : y + L * I * r0;

  TC acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = (TC)0;

  for (int64_t i0 = 0; i0 < I; i0 += TBI) {
    // A tile: 64 k x 16 i
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int idx = tid + 256 * e;
      int ii, kk;
      if (a_rowmajor) { ii = idx % TBI; kk = idx / TBI; }
      else { kk = idx % TT; ii = idx / TT; }
      int64_t k = k0 + kk, i = i0 + ii;
      TC v = (TC)0;
      if (k < K && i < I) {
        if (A32) v = (TC)A32[k * I + i];   // FP32 operator converted once (k_ttm_a32)
        else v = (TC)(a_rowmajor ? A[k * lda + i] : A[k + lda * i]);
      }
      As[ii][kk] = v;
    }
    // Y tile: 16 i x 64 m
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int idx = tid + 256 * e;
      int ii, mm;
      TC v = (TC)0;
      if (L == 1) {
        ii = idx % TBI; mm = idx / TBI;
        int64_t i = i0 + ii, r = r0 + mm;
        if (i < I && r < Rt) v = (TC)ybase[i + I * r];
      } else {
        mm = idx % TT; ii = idx / TT;
        int64_t i = i0 + ii, l = l0 + mm;
        if (i < I && l < L) v = (TC)ybase[l + L * i];
      }
      Ys[ii][mm] = v;
    }
    __syncthreads();
#pragma unroll
    for (int ii = 0; ii < TBI; ++ii) {
      TC a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = As[ii][kq + 16 * u];
#pragma unroll
      for (int v = 0; v < 4; ++v) b[v] = Ys[ii][mq + 16 * v];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
  // write Z: (k, m) -> l + L*(k + K*r)
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    int64_t k = k0 + kq + 16 * u;
    if (k >= K) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      int mm = mq + 16 * v;
      if (L == 1) {
        int64_t r = r0 + mm;
        if (r < Rt) {
          if (zt) z[r + Rt * k] = (TOut)acc[u][v];
          else z[k + K * r] = (TOut)acc[u][v];
        }
      } else {
        int64_t l = l0 + mm;
        if (l < L) z[l + L * (k + K * r0)] = (TOut)acc[u][v];
      }
    }
  }
}

// A (K x I, FP64, either layout) -> FP32 row-major K x I.  An FP64 -> FP32
// conversion runs on the FP64 pipe (64 cycles per warp instruction), so the
// FP32 TTM converts its operator once here instead of in every tile.
__global__ void k_ttm_a32(const double* __restrict__ A, int64_t K, int64_t I, int64_t lda,
                          int a_rowmajor, float* __restrict__ A32) {
  const int64_t n = K * I;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = e / I, i = e - k * I;
    A32[e] = (float)(a_rowmajor ? A[k * lda + i] : A[k + lda * i]);
  }
}

template <typename TIn, typename TOut, typename TC, int KT, bool COL>
static cudaError_t ttm_tile(const TIn* y, int64_t L, int64_t I, int64_t M, const double* A, int64_t K,
                            int64_t lda, int arow, const float* A32, TOut* z, int zt,
                            cudaStream_t st) {
  constexpr int WK = KT == 8 ? 2 : 4, MM = WK, MT = TNT;
  const int64_t gx = (M + MT - 1) / MT, tiles = (K + KT - 1) / KT, gz = (tiles + 65534) / 65535;
  if (gx > 0x7fffffffll || gz > 65535) return cudaErrorInvalidConfiguration;
  auto kern = k_ttm<TIn, TOut, TC, KT, WK, MM, COL>;
  cudaError_t e = allow_max_dyn_smem((const void*)kern);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)gx, (unsigned)((tiles + gz - 1) / gz), (unsigned)gz);
  kern<<<grid, TNT, ttm_smem<TIn, TC, KT, MT, COL>(), st>>>(y, L, I, M, A, K, lda, arow, A32, z, zt);
  return cudaGetLastError();
}

template <typename TIn, typename TOut, typename TC>
static cudaError_t ttm_new(const void* y, int64_t L, int64_t I, int64_t Rt, const double* A, int64_t K,
                           int64_t lda, int arow, const float* A32, void* z, int zt, int num_sms,
                           cudaStream_t st) {
  const int kt = ttm_tile_outputs(L * Rt, K, num_sms);
  auto tile = [&](auto KT) {
    return L == 1 ? ttm_tile<TIn, TOut, TC, decltype(KT)::value, true>(
                        (const TIn*)y, L, I, Rt, A, K, lda, arow, A32, (TOut*)z, zt, st)
                  : ttm_tile<TIn, TOut, TC, decltype(KT)::value, false>(
                        (const TIn*)y, L, I, L * Rt, A, K, lda, arow, A32, (TOut*)z, zt, st);
  };
  if (kt == 8) return tile(std::integral_constant<int, 8>());
  if (kt == 16) return tile(std::integral_constant<int, 16>());
  if (kt == 24) return tile(std::integral_constant<int, 24>());
  return tile(std::integral_constant<int, 32>());
}

// The smallest tile that divides K into tiles of at most 32; smaller ones while the grid
// still leaves half the SMs idle (a block's time grows with its outputs: 0.31, 0.57 and 1.08 us
// per i in FP64 for 8, 16 and 24 or 32): FP32 row view 300 x 3000 to 32 72 -> 49 us, FP64
// 64 x 1500 to 28 101 -> 52.
int ttm_tile_outputs(int64_t M, int64_t K, int num_sms) {
  const int64_t nt = (K + 31) / 32, per = (K + nt - 1) / nt;
  int kt = per <= 8 ? 8 : per <= 16 ? 16 : per <= 24 ? 24 : 32;
  while (kt > 8 && 2 * ((M + TNT - 1) / TNT) * ((K + kt - 1) / kt) <= num_sms) kt = kt > 16 ? 16 : 8;
  return kt;
}

// FP32 row views with more than 32 outputs whose I leaves half of k_ttm's last stage of 32
// unused, up to 16 rows, or 33 to 48 where the view allows no 16-byte loads: the 64 x 64 tiles
// of k_ttm_simt (stages of 16), where at least half of their entries are used.  k_ttm and
// there: 25000 x 12 x 10 to 310 235 and 190 us, x 16 to 50 76 and 61, x 16 to 33 67 and 60,
// x 17 to 310 254 and 274; 24999 x 48 x 10 to 50 118 and 103, 25000 x 48 x 10 to 310 435 and
// 431; 52 x 12 x 5000 to 65 89 and 106.
static bool ttm_wide_tiles(const void* y, int64_t L, int64_t I, int64_t K) {
  const int64_t l = (L + TT - 1) / TT, k = (K + TT - 1) / TT;
  const bool vec = L % 4 == 0 && ((uintptr_t)y & 15) == 0;
  return L > 1 && K > 32 && k <= 65535 && (I <= 16 || (!vec && I > 32 && I <= 48)) &&
         2 * (double)L * (double)K >= (double)(l * TT) * (double)(k * TT);
}

cudaError_t launch_ttm_simt(const void* y, tucker_dtype ydt, bool fp64, int64_t L, int64_t I,
                            int64_t Rt, const double* A, int64_t K, int64_t lda, int a_rowmajor,
                            float* a32_scratch, void* z, tucker_dtype zdt, int num_sms,
                            cudaStream_t st, bool zt) {
  if (zt && L != 1) return cudaErrorInvalidValue;
  if (L * Rt <= 0 || K <= 0) return cudaSuccess;
  const float* A32 = nullptr;
  if (!fp64 && a32_scratch) {
    const int64_t n = K * I;
    k_ttm_a32<<<(unsigned)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024), 256, 0, st>>>(
        A, K, I, lda, a_rowmajor, a32_scratch);
    count_launches(1);
    A32 = a32_scratch;
  }
  count_launches(1);
  const bool yd = ydt == TUCKER_F64, zd = zdt == TUCKER_F64;
  if (fp64) {
    if (yd) return zd ? ttm_new<double, double, double>(y, L, I, Rt, A, K, lda, a_rowmajor, A32, z, zt, num_sms, st)
                      : ttm_new<double, float, double>(y, L, I, Rt, A, K, lda, a_rowmajor, A32, z, zt, num_sms, st);
    return zd ? ttm_new<float, double, double>(y, L, I, Rt, A, K, lda, a_rowmajor, A32, z, zt, num_sms, st)
              : ttm_new<float, float, double>(y, L, I, Rt, A, K, lda, a_rowmajor, A32, z, zt, num_sms, st);
  }
  const int64_t nLT = L == 1 ? 1 : (L + TT - 1) / TT, nMT = L == 1 ? (Rt + TT - 1) / TT : Rt * nLT;
  if (!yd && !zd && !(ttm_wide_tiles(y, L, I, K) && nMT <= 0x7fffffffll))
    return ttm_new<float, float, float>(y, L, I, Rt, A, K, lda, a_rowmajor, A32, z, zt, num_sms, st);
  if (nMT > 0x7fffffffll) return cudaErrorInvalidConfiguration;
  const dim3 grid((unsigned)nMT, (unsigned)((K + TT - 1) / TT));
  if (!yd && !zd)
    k_ttm_simt<float, float, float><<<grid, 256, 0, st>>>((const float*)y, L, I, Rt, nLT, A, K, lda, a_rowmajor, A32, (float*)z, zt);
  else if (yd && zd)
    k_ttm_simt<double, double, float><<<grid, 256, 0, st>>>((const double*)y, L, I, Rt, nLT, A, K, lda, a_rowmajor, A32, (double*)z, zt);
  else if (yd)
    k_ttm_simt<double, float, float><<<grid, 256, 0, st>>>((const double*)y, L, I, Rt, nLT, A, K, lda, a_rowmajor, A32, (float*)z, zt);
  else
    k_ttm_simt<float, double, float><<<grid, 256, 0, st>>>((const float*)y, L, I, Rt, nLT, A, K, lda, a_rowmajor, A32, (double*)z, zt);
  return cudaGetLastError();
}

}  // namespace tk
