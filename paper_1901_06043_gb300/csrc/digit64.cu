// Double-precision contractions on the tensor cores by exact integer digits:
// the FP64 Gram S = sum_k x(i, k) x(j, k) of a slab view (Algorithm 2) and the
// FP64 TTM Z(m, k) = sum_i y(m, i) A(k, i) (Algorithm 3).
//
// Why.  FP64 instructions run at 1/64 of the FP32 rate on this part (1.19
// TFLOP/s measured), so an FP64 Gram was bound by the FP64 pipe at 30 to 60
// times the time its bytes take.  The tensor cores multiply FP16 integers
// exactly at 1.9 PFLOP/s; with seven 8-bit digits per value an FP64 product
// costs 34 FP16 products, still ~45 times the FP64 pipe's rate.  Measured
// (whole calls on a 200x200x200x50 tensor, the FP64 pipe first): mode-0 Gram 163 and
// 7.6 ms, mode-0 TTM to 28 rows 20.6 and 3.7 ms, the expansion 2e6 x 26 -> 200 of a row
// view (a 3.2 GB result) 23.6 and 3.8 ms.
//
// Arithmetic.  A row (an index that is not contracted) has one power-of-two
// scale 2^E, E = exponent of its largest magnitude + 1, so |x| < 2^E.  Every
// value becomes a 55-bit fixed-point number by integer operations (the FP64
// pipe is not used), |x| 2^(63 - E) rounded at 2^8, and with 0x80 added to the
// bytes below the top one its bytes are the balanced base-256 digits:
// |x| 2^(63 - E) = sum_j d_j 2^(8 (7 - j)) (+ the rounding), j = 0..6,
// |d_j| <= 128; the sign goes onto the digits.  Digits are exact in FP16.  For two operands the
// products are grouped by weight, D_c = sum_{p + q = c} d_p d'_q, c = 0..7 (34
// products), each class into its own FP32 accumulator in tensor memory.  A class
// sums at most 7 products of at most 2^14 per k; windows of 128 k keep every
// partial sum an integer below 2^24, so the accumulators are exact.  After
// each window the eight sums are combined as one integer sum_c D_c 2^(8 (7 - c))
// and added to a 96-bit integer per entry: nothing is rounded until the end,
// where the integer becomes one FP64 value, times 2^(E + E' - 70).
//   Errors: the fixed-point rounding, at most 2^-56 2^E (2^-55 of the row's
// largest magnitude, unbiased; values within a factor 4 of it are exact), and
// the classes c >= 8 left out, below 2^-63 of a product of the rows' maxima
// per k.  So an entry is off by at most 2^-55 (|x_i|_max |x_j|_1 + |x_j|_max
// |x_i|_1), where an FP64 sum is off by 2^-53 of each of its partial sums.
// Against the rows' norms that is no more than an FP64 sum has; against the entry
// itself it is more where the large values of one row meet small ones of the other
// (a value 2^-40 of its row's largest keeps 15 bits).  Hence TUCKER_OPT_FP64_KERNEL, and
// a TTM whose operator has a zero beside other values in a row (it may be there to leave
// out a fibre's large values: selections, differences) is computed on the FP64 pipe.
//   NaN, Inf, or a row whose largest magnitude is below 2^-958 (its exponents
// would need the denormal range): the exponent pass sets *bad and the caller
// computes the step on the FP64 pipe (the host reads the flag with the error
// word); a caller that does not wait gets NaN for NaN and Inf, and small rows in
// units of 2^-1013.
//   Splitting FP64 matrices into slices whose products are exact in a narrower
// arithmetic is the error-free transformation of Ozaki, Ogita, Oishi and Rump
// (Numerical Algorithms 59, 2012), used on integer and FP16 matrix units since.
//
// Tile and roles.  One CTA owns a 128 x 64 tile (M x N): eight classes of 64
// columns are all 512 tensor-memory columns.  The digit planes of the 64-row
// operand sit side by side along N, so digit plane q of the 128-row operand
// times [d'_0 .. d'_3] is one N = 256 MMA onto four adjacent classes: 11 MMAs
// per 16 k instead of 34.  A stage is 16 k (42 KB: 7 planes x (128 + 64) rows x
// 16 k, MN-major SW128), three stages.  Sixteen warps copy the raw values into shared
// memory (cp.async, four stages ahead), split them and write the planes, and drain a
// window as soon as it is complete (nothing can be issued onto the accumulators meanwhile, but
// the ring fills up); a seventeenth warp issues the MMAs (issuing a stage takes
// as long as its MMAs run: a producer that issues is 2,400 cycles late every
// 32 k).
//   The splitting is bound by the integer (ALU) pipe, which takes a warp
// instruction every two cycles, as is the FP64 rounding of a tile's results;
// so the digits are whole bytes (byte permutes; 7-bit digits took 47 ALU
// instructions a value against 13), the sign and the digit offset go through
// the FP16 pipe, and shifts to the left through multiplies.
//   TTM: the 128 rows are m (slabs, or l and slab), the 64 are outputs k; the
// operator's digit planes are prepared once per call as stage images and
// copied in by one bulk copy per stage.
//   What a 16-k stage takes (500 x 16-k stages of a 200 x 4e5 Gram, parts
// removed one at a time): 3,000 cycles with everything, 2,750 without the digit
// split, 2,550 without the drain, 1,100 for the MMAs issued back to back.  Counters of that
// Gram: tensor pipe 41 %, ALU pipe 49 %, issue 53 %, DRAM 6 %.
//
// Every wait is bounded: one that gives up sets DEV_ERR_MBAR_TIMEOUT and the
// kernel winds down; tensor memory is always released.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace tk {
namespace {

using namespace tc;

constexpr int ND = 7;                       // digits per value
constexpr int NC = 8;                       // weight classes
constexpr int MT = 128, NT = 64;            // tile
constexpr int BK = 16;                      // k per stage: one MMA step
constexpr int NST = 3;                      // stages
constexpr int NRAW = 4;                     // stages of raw values in flight
constexpr int WIN = 8;                      // stages per exact window (128 k)
constexpr int NPW = 16;                     // producer / drain warps
constexpr int MMA_WARP = NPW;
constexpr int NTHREADS = (NPW + 1) * 32;
constexpr uint32_t ATOM = 1024;             // 64 mn x 8 k, FP16
constexpr uint32_t KG_A = 2 * ND * ATOM;    // k-group (8 k) stride of the 128-row operand
constexpr uint32_t KG_B = ND * ATOM;
constexpr uint32_t A_BYTES = (BK / 8) * KG_A, B_BYTES = (BK / 8) * KG_B;
constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
// raw values: NRAW quads of the 128-row operand per thread, then NRAW / 2 of
// the 64-row one (Gram) or the exponents (TTM)
constexpr uint32_t RAW_A = NPW * 32 * 32, RAW_BYTES = NRAW * RAW_A + NRAW / 2 * RAW_A;
constexpr uint32_t SMEM_BYTES = NST * STAGE_BYTES + RAW_BYTES + 1024;
constexpr int TILE_ELEMS = MT * NT;
constexpr int BAD_EXP = 0x7ff, MIN_EXP = 64;   // biased exponents of a row: bad, smallest
constexpr int OUT_EXP = -2 * 1022 - 70;        // an entry is its sum times 2^(eb + eb' + OUT_EXP)
// Work from which a step comes here.  Gram: I^2 K >= 2e7 (whole calls, I = 200:
// 86 us on the FP64 pipe and 76 us here at 2e7; 66 and 75 us at 1e7; 235 and 89
// us at 1e8).
constexpr double kDigit64MinGram = 2e7;
// TTM: where the digits are the faster by the two models of a whole call below (us,
// FP64 data, one wave being num_sms blocks), fitted to 720 calls with I from 8 to 500, K from
// 4 to 200 and M from 300 to 4e5, column and row views: within 26 % (FP64 pipe and here, column
// views) and 35 % (row views).  On these calls the rule loses 0.3 % to the better of the two,
// and 31 % at worst (26 x 24000 to 28, row view, 103 us there and 78 here).  Both sides, there
// and here: 64 x 1500 to 4 52 and 71, to 28 52 and 78; 200 x 1500 to 28 95 and 94; 16 x 1e5
// to 16 84 and 107, to 28 135 and 114; 200 x 4e5 to 28 4242 and 807.
//   A block of the pipe's kernel takes 0.31, 0.57 or 1.08 us per i for 8, 16 or more
// outputs, a CTA here per item of 128 m and 64 outputs 2 (row views 1.6) us per stage of
// 16 i and its drain; 1.2 ps per value are the exponent pass.
//   And not below I = 64 and 2 K I M = 4e7, where the digits gain 25 us at most and a
// value keeps fewer bits there.
constexpr double kDigit64MinTtm = 4e7;
constexpr int kDigit64MinTtmI = 64;
inline double ceil_div(double a, double b) { return std::ceil(a / b); }
double ttm_pipe_us(double M, double I, double K, int sms) {
  const int kt = ttm_tile_outputs((int64_t)M, (int64_t)K, sms);
  const double blocks = ceil_div(M, 128.0) * ceil_div(K, kt);
  return 30.0 + (kt == 8 ? 0.31 : kt == 16 ? 0.57 : 1.08) * I * ceil_div(blocks, sms);
}
double ttm_digit_us(double M, double I, double K, double sms, bool col) {
  const double items = ceil_div(ceil_div(M, MT) * ceil_div(K, NT), sms), st = ceil_div(I, BK);
  const double k = std::min(K, (double)NT);
  return 62.0 + items * (col ? 2.0 * st + 3.0 + 0.1 * k : 1.6 * st + 4.0 + 0.04 * k) + 1.2e-6 * I * M;
}
// Modes below 64 (gram_small.cu otherwise, ~I^2 / 2 FP64 instructions per 32 k;
// here ~0.6 ns a k whatever I, one padded tile): K (I^2 - 565) >= 6.5e7.  Whole calls
// there and here: I = 28, K = 4e5 342 and 332 us (2e5 197 and 220); I = 40, 5e4 122 and
// 125 (1e5 193 and 155); I = 63, 2e4 136 and 113 (1e6 3.44 and 0.71 ms).
constexpr double kDigit64SmallII = 565, kDigit64SmallGram = 6.5e7;

// Byte offset of (mn, k) in plane 0 of an operand region with k-group stride kg.
__device__ __forceinline__ uint32_t mn_off(int mn, int k, uint32_t kg) {
  return (uint32_t)(k >> 3) * kg + (uint32_t)(mn >> 6) * ATOM + (uint32_t)(k & 7) * 128u +
         ((uint32_t)(((mn & 63) >> 3) ^ (k & 7)) << 4) + (uint32_t)(mn & 7) * 2u;
}

// kind::f16, FP16 A and B (both MN-major), FP32 D.
__device__ __forceinline__ uint32_t instr_desc(int N) {
  return (1u << 4) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(MT >> 4) << 24);
}

// The magnitude's high bits, ordered as the magnitudes are (0 only for x = 0),
// and the biased (1023) exponent of a row from their maximum.
__device__ __forceinline__ int mag_bits(double x) {
  return (__double2hiint(x) & 0x7fffffff) | (__double2loint(x) != 0 ? 1 : 0);
}
__device__ __forceinline__ int mag_bits(float x) { return (int)(__float_as_uint(x) & 0x7fffffffu); }
// MIN_EXP for a row of zeros; BAD_EXP for NaN, Inf and rows below MIN_EXP.  A
// caller that does not wait for the verdict (small = false) has such rows at
// MIN_EXP: their entries are then off by up to 2^-1013 each, below the rounding of a
// Gram's or a TTM's norm.
__device__ __forceinline__ int row_exp(int m, double, int small) {
  const int e = m >> 20;
  return m == 0 ? MIN_EXP : (e < MIN_EXP ? (small ? BAD_EXP : MIN_EXP) : e);
}
__device__ __forceinline__ int row_exp(int m, float, int) {
  const int e = m >> 23;
  return e == 0xff ? BAD_EXP : (e < 1 ? 1 : e) + 896;
}

// |x| 2^(63 - E) + 0x80 in bytes 0..6, E = eb - 1022: byte 7 (0..128) is the
// top digit, bytes 6..1 less 128 the others (byte 0 rounds).  es: the row's exponent as shift_base gives it.
__device__ __forceinline__ uint32_t shift_base(int eb, double) { return ((uint32_t)eb << 21) | 0x1fffffu; }
__device__ __forceinline__ uint32_t shift_base(int eb, float) {
  return ((uint32_t)(eb - 896) << 24) | 0xffffffu;
}
__device__ __forceinline__ uint2 fixed_of(uint32_t hi, uint32_t lo, uint32_t d) {
  uint32_t q0, q1;
  asm("{\n .reg .u64 m;\n mov.b64 m, {%2, %3};\n shr.u64 m, m, %4;\n"
      " add.u64 m, m, 0x0080808080808080;\n mov.b64 {%0, %1}, m;\n}"
      : "=r"(q0), "=r"(q1) : "r"(lo), "r"(hi), "r"(d));
  return make_uint2(q0, q1);
}
__device__ __forceinline__ uint2 fixed_of(double x, uint32_t es) {
  // (a zero or denormal x gets an implicit bit, but its exponent is 0 and es
  // at least MIN_EXP: it is shifted out)
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t d = (es - 2u * hi) >> 21;              // eb - exponent of x
  const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
  return fixed_of((mh << 10) | (lo >> 22), lo << 10, d);
}
__device__ __forceinline__ uint2 fixed_of(float x, uint32_t es) {
  const uint32_t u = __float_as_uint(x), t = u & 0x7fffffffu;
  const uint32_t d = (es - 2u * u) >> 24;
  const uint32_t m = t >= 0x800000u ? ((t & 0x7fffffu) | 0x800000u) : 2u * t;   // denormals: exponent 0
  return fixed_of(m << 7, 0u, d);
}
__device__ __forceinline__ uint32_t sign_word(double x) { return (uint32_t)__double2hiint(x); }
__device__ __forceinline__ uint32_t sign_word(float x) { return __float_as_uint(x); }

// Digit planes of two values as FP16 pairs, p[0] the top digit: a byte u under
// 0x64 is 1024 + u, and (1024 + u - 1152) s = d (top digit: - 1024), s = +-1
// per half.
template <typename T>
__device__ __forceinline__ void digits_pair(T xa, T xb, uint32_t ea, uint32_t eb,
                                            uint32_t (&p)[ND]) {
  const uint2 a = fixed_of(xa, ea), b = fixed_of(xb, eb);
  const uint32_t sg = (__byte_perm(sign_word(xa), sign_word(xb), 0x7632) & 0x80008000u) | 0x3c003c00u;
  const __half2 s = *reinterpret_cast<const __half2*>(&sg);
  const __half2 off0 = __hmul2(s, __halves2half2(__ushort_as_half(0xE400), __ushort_as_half(0xE400)));
  const __half2 off = __hmul2(s, __halves2half2(__ushort_as_half(0xE480), __ushort_as_half(0xE480)));
  const uint32_t w[4] = {__byte_perm(a.y, b.y, 0x7632), __byte_perm(a.y, b.y, 0x5410),
                         __byte_perm(a.x, b.x, 0x7632), __byte_perm(a.x, b.x, 0x5410)};
#pragma unroll
  for (int j = 0; j < ND; ++j) {
    // w[j / 2] = [a low, a high, b low, b high] digit bytes
    const uint32_t h = __byte_perm(w[j >> 1], 0x64646464u, (j & 1) ? 0x4240 : 0x4341);
    const __half2 d = __hfma2(*reinterpret_cast<const __half2*>(&h), s, j == 0 ? off0 : off);
    p[j] = *reinterpret_cast<const uint32_t*>(&d);
  }
}

// Four consecutive mn at one k: an 8-byte store per plane.
template <typename T>
__device__ __forceinline__ void store_quad(uint8_t* dst, uint32_t plane_step, const T (&v)[4],
                                           const uint32_t (&es)[4]) {
  uint32_t p01[ND], p23[ND];
  digits_pair(v[0], v[1], es[0], es[1], p01);
  digits_pair(v[2], v[3], es[2], es[3], p23);
#pragma unroll
  for (int q = 0; q < ND; ++q)
    *reinterpret_cast<uint2*>(dst + q * plane_step) = make_uint2(p01[q], p23[q]);
}

// A 96-bit two's complement sum.
struct Sum96 {
  uint32_t w0, w1, w2;
};

// s += sum_c D_c 2^(8 (7 - c)), the D_c integers of at most 2^24.
__device__ __forceinline__ void add_classes(Sum96& s, const uint32_t (&r)[NC]) {
  int d[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) d[c] = __float2int_rn(__uint_as_float(r[c]));
  // |D_0| <= 2^21, |D_2| <= 3 2^21: these pairs fit 32 bits
  const long long h = (long long)(d[0] * 256 + d[1]) * 65536ll + (long long)(d[2] * 256 + d[3]);
  const long long l = ((long long)d[4] << 24) + (long long)d[5] * 65536ll + (long long)d[6] * 256ll +
                      (long long)d[7];
  const uint32_t h0 = (uint32_t)h, h1 = (uint32_t)((unsigned long long)h >> 32);
  const uint32_t l0 = (uint32_t)l, l1 = (uint32_t)((unsigned long long)l >> 32);
  const uint32_t l2 = (uint32_t)((int)l1 >> 31);
  asm("{\n add.cc.u32 %0, %0, %3;\n addc.cc.u32 %1, %1, %4;\n addc.u32 %2, %2, %5;\n"
      " add.cc.u32 %1, %1, %6;\n addc.u32 %2, %2, %7;\n}"
      : "+r"(s.w0), "+r"(s.w1), "+r"(s.w2)
      : "r"(l0), "r"(l1), "r"(l2), "r"(h0), "r"(h1));
}

// The sum times 2^x, rounded to nearest in FP64, by integer operations.  (A
// negative sum is inverted without the carry, one unit of 2^-70 of the scales;
// bits below the top 64 do not break a tie.)
__device__ __forceinline__ double to_double(const Sum96& s, int x) {
  const uint32_t n = (uint32_t)((int)s.w2 >> 31);
  uint32_t a = s.w2 ^ n, b = s.w1 ^ n, c = s.w0 ^ n;
  int top = 1023 + 95 - 1 + x;                   // exponent field - 1 of bit 95
  if (a == 0u) { a = b; b = c; c = 0u; top -= 32; }
  if (a == 0u) { a = b; b = c; top -= 32; c = 0u; }
  if (a == 0u) return 0.0;
  const int z = __clz(a);
  top -= z;
  const uint32_t u1 = __funnelshift_l(b, a, z), u0 = __funnelshift_l(c, b, z);
  const uint32_t lo = __funnelshift_r(u0, u1, 11), hi = u1 >> 11;      // 53 bits, leading one at hi's bit 20
  uint32_t r0, r1;
  asm("{\n add.cc.u32 %0, %2, %4;\n addc.u32 %1, %3, 0;\n}"
      : "=r"(r0), "=r"(r1) : "r"(lo), "r"(hi), "r"((u0 >> 10) & 1u));
  if (top < 0 || top > 2044) {                    // out of the normal range
    const double v = __hiloint2double((int)((1022u << 20) + r1), (int)r0);
    const double w = scalbn(v, top - 1022);
    return n ? -w : w;
  }
  return __hiloint2double((int)((((uint32_t)top << 20) + r1) | (n & 0x80000000u)), (int)r0);
}

// Whether the barrier's phase with the given parity has completed.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done != 0;
}

struct Args {
  const void* x;
  int64_t L, I, Rt;
  int64_t nk;               // contracted length: L Rt (Gram), I (TTM)
  unsigned* err;
  const unsigned* bad;      // nonzero: NaN or Inf in an operand
  // Gram
  int ntiles, nkg;
  const unsigned* rexp;     // biased exponent of each row's largest magnitude
  double* part;
  // TTM
  int64_t M;                // L Rt
  int K, ntn, nks;          // outputs, N-tiles of 64, stages per tile
  int64_t nitems;           // M-tiles x N-tiles
  const uint16_t* mexp;     // per m
  const uint8_t* bimg;      // ntn x nks stage images of A
  const unsigned* kexp;     // per output (64 ntn entries)
  void* z;
  int zt;                   // L == 1: z[m + M k]
  int waits;                // the caller reads *bad and computes the step again
};

// Gram tile t -> (ta, tb): 128-row block ta, 64-row block tb <= 2 ta + 1.
__host__ __device__ __forceinline__ void tile_of(int t, int& ta, int& tb) {
  int a = (int)((sqrtf(4.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((a + 1) * (a + 2) <= t) ++a;
  while (a * (a + 1) > t) --a;
  ta = a;
  tb = t - a * (a + 1);
}

// Copies of N bytes (4, 8, 16) from global to shared memory without a register;
// ok = false writes zeros (src must be a valid address all the same).
template <int N>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, bool ok) {
  if (N == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(N), "r"(ok ? N : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A thread's quad of raw values: 16-byte chunks, chunk c of thread t at
// [c][t] (no bank conflicts).
constexpr uint32_t CHUNK = NPW * 32 * 16;
__device__ __forceinline__ void raw_quad(const uint8_t* p, double (&v)[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  const double2 b = *reinterpret_cast<const double2*>(p + CHUNK);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void raw_quad(const uint8_t* p, float (&v)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}

// The drain of one window (all classes of this warp's 16 columns of its 32
// rows) into the warp's sums.
__device__ __forceinline__ void drain(uint32_t taddr, Sum96 (&acc)[16]) {
#pragma unroll
  for (int cc = 0; cc < 16; cc += 4) {
    uint32_t r[NC][4];
#pragma unroll
    for (int c = 0; c < NC; ++c)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(r[c][0]), "=r"(r[c][1]), "=r"(r[c][2]), "=r"(r[c][3])
                   : "r"(taddr + 64u * (uint32_t)c + (uint32_t)cc));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t d[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) d[c] = r[c][j];
      add_classes(acc[cc + j], d);
    }
  }
}

// The MMAs of a stage: digit plane q of the 128-row operand times planes
// 0..3 and 4..min(6, 7 - q) of the 64-row one, onto classes q.. .  Plane p of
// the 64-row operand: its own region, or (diagonal Gram tiles) half `half` of
// the 128-row operand's plane.  acc0 = 0: the stage opens a window (its first
// product of every class overwrites).
__device__ __forceinline__ void issue_stage(uint32_t st, uint32_t tmem, bool diag, int half,
                                            uint32_t acc0) {
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t bstart = diag ? st + (uint32_t)half * ATOM : st + A_BYTES;
  const uint32_t bplane = diag ? 2 * ATOM : ATOM, bkg = diag ? KG_A : KG_B;
  const uint64_t a0 = smem_desc(st, ATOM, KG_A);
  const uint64_t b0 = smem_desc(bstart, bplane, bkg);
  const uint64_t b4 = b0 + (uint64_t)((4u * bplane) >> 4), b6 = b0 + (uint64_t)((6u * bplane) >> 4);
#pragma unroll
  for (int q = 0; q < ND; ++q) {
    const uint64_t a = a0 + (uint64_t)q * (2 * ATOM >> 4);
    const int np = q == 0 ? 7 : 8 - q;              // planes of the 64-row operand
    tc_mma(tmem + 64u * (uint32_t)q, a, b0, instr_desc(64 * (np < 4 ? np : 4)), q == 0 ? acc0 : 1u);
    if (q == 1 && acc0 == 0u) {                     // class 7 opens here
      tc_mma(tmem + 64u * 5u, a, b4, instr_desc(128), 1u);
      tc_mma(tmem + 64u * 7u, a, b6, instr_desc(64), 0u);
    } else if (np > 4) {
      tc_mma(tmem + 64u * (uint32_t)(q + 4), a, b4, instr_desc(64 * (np - 4)), q == 0 ? acc0 : 1u);
    }
  }
}

// MNC: the mn index is contiguous in memory (Gram of a column view, TTM of a
// row view), a lane holds four consecutive mn of one k; otherwise k is
// contiguous and lanes run along k.  VEC (MNC): quads start on 16 bytes (32
// for FP64 pairs) and never cross a slab.
template <typename T, typename TOut, bool TTM, bool MNC, bool VEC>
__global__ void __launch_bounds__(NTHREADS, 1) k_digit64(const Args g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t bar_full[NST], bar_empty[NST], bar_accf, bar_acce, bar_done;
  __shared__ uint32_t tmem_base_sh;
  if (*g.bad) {                                          // the same for the whole grid
    if (TTM && !g.waits) {
      TOut* z = static_cast<TOut*>(g.z);
      for (int64_t e = (int64_t)blockIdx.x * NTHREADS + threadIdx.x; e < g.M * g.K;
           e += (int64_t)gridDim.x * NTHREADS)
        z[e] = (TOut)__longlong_as_double(0x7ff8000000000000ll);
    }
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // this CTA's stages
  int ta = 0, tb = 0;
  int64_t s0 = 0;                                        // Gram: first stage of the K split
  int nst, wst;                                          // stages; per tile (Gram: all)
  if (!TTM) {
    tile_of((int)(blockIdx.x % g.ntiles), ta, tb);
    const int64_t kg = blockIdx.x / g.ntiles, stages = (g.nk + BK - 1) / BK;
    s0 = stages * kg / g.nkg;
    nst = wst = (int)(stages * (kg + 1) / g.nkg - s0);
  } else {
    const int64_t items =
        (g.nitems > (int64_t)blockIdx.x) ? (g.nitems - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    nst = (int)(items * g.nks);
    wst = g.nks;
  }
  const bool diag = !TTM && (tb >> 1) == ta;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(smem_u32(&bar_full[s]), NPW);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    mbar_init(smem_u32(&bar_accf), 1);
    mbar_init(smem_u32(&bar_acce), NPW);
    mbar_init(smem_u32(&bar_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
        smem_u32(&tmem_base_sh)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base_sh;

  if (warp == MMA_WARP) {
    // ---------------- MMA issue (one thread; issuing takes as long as the
    // MMAs run, so no producer can do it)
    if (lane == 0) {
      uint32_t w = 0, ph = 0;                              // windows begun; parity of the slot's fill
      int slot = 0, ws = 0, tend = wst;                    // start of the open window, end of the open tile
      for (int s = 0; s < nst; ++s) {
        const int we = ws + WIN < tend ? ws + WIN : tend;
        if (s == ws && w > 0 && !mbar_wait(smem_u32(&bar_acce), (w - 1) & 1u, g.err)) break;
        if (!mbar_wait(smem_u32(&bar_full[slot]), ph, g.err)) break;
        issue_stage(smem_u32(smem) + (uint32_t)slot * STAGE_BYTES, tmem, diag, tb & 1,
                    s == ws ? 0u : 1u);
        tc_commit(smem_u32(&bar_empty[slot]));
        if (++slot == NST) { slot = 0; ph ^= 1u; }
        if (s + 1 == we) {
          tc_commit(smem_u32(&bar_accf));
          ++w;
          ws = we;
          if (we == tend) tend += wst;
        }
      }
      // every tcgen05 op issued has completed once bar_done fires
      tc_commit(smem_u32(&bar_done));
    }
    __syncwarp();
  } else {
    // ---------------- producers, and drain
    const T* x = static_cast<const T*>(g.x);
    // this lane's quads: one of the 128-row operand every stage; one of the
    // 64-row operand (Gram) every second stage, warps 0-7 and 8-15 in turn
    const int wb = warp & 7;
    const int mnA = MNC ? 4 * lane : 8 * warp + 4 * (lane >> 4);
    const int mnB = MNC ? 4 * (lane & 15) : 8 * wb + 4 * (lane >> 4);
    const int kA = MNC ? warp : (lane & 15);
    const int kB = MNC ? 2 * wb + (lane >> 4) : (lane & 15);
    const uint32_t oA = mn_off(mnA, kA, KG_A);
    const uint32_t oB = A_BYTES + mn_off(mnB, kB, KG_B);
    const int64_t LI = g.L * g.I;

    uint32_t eA[4], eB[4];
    uint8_t* raw = smem + NST * STAGE_BYTES + threadIdx.x * 16;      // this thread's chunks
    unsigned maskA = 0, maskB = 0;
    const T* pA = x;
    const T* pB = x;
    // the next load of each quad: its address, and how many of this tile's
    // (Gram: this CTA's) loads are left; row views also the l of its k
    int cA = 0, cB = 0;
    int lA = 0, lB = 0;                                    // (L I < 2^31; 64-bit comparisons run on the FP64 pipe)
    const int Li = (int)g.L;
    int64_t item = blockIdx.x;
    int ks = 0;
    int mrel[4] = {0, 0, 0, 0};                            // TTM: offsets of the quad's m
    const uint16_t* mexp4 = g.mexp;                        // and their exponents
    const int64_t stepA = TTM ? BK * g.L : (MNC ? BK * g.I : BK);
    if (!TTM) {
      const int64_t rowA = (int64_t)ta * MT + mnA, rowB = (int64_t)tb * NT + mnB;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (rowA + j < g.I) maskA |= 1u << j;
        if (rowB + j < g.I) maskB |= 1u << j;
        eA[j] = shift_base(rowA + j < g.I ? (int)g.rexp[rowA + j] : 1023, T());
        eB[j] = shift_base(rowB + j < g.I ? (int)g.rexp[rowB + j] : 1023, T());
      }
      const int64_t ka = s0 * BK + kA, kb = (s0 + (warp >> 3)) * BK + kB;
      const int64_t rA = ka / g.L, rB = kb / g.L;
      lA = (int)(ka - rA * g.L);
      lB = (int)(kb - rB * g.L);
      pA = x + (maskA ? rowA * g.L : 0) + lA + LI * rA;
      pB = x + (maskB ? rowB * g.L : 0) + lB + LI * rB;
      const int64_t na = (g.nk - ka + BK - 1) / BK, nb = (g.nk - kb + 2 * BK - 1) / (2 * BK);
      cA = na > nst ? nst : (int)na;                       // (may be <= 0)
      cB = nb > nst ? nst : (int)nb;
    }
    auto tile_setup = [&]() {                              // TTM: pointers of the item's quad of m
      const int64_t m0 = (item / g.ntn) * MT + mnA;
      maskA = 0;
      const int64_t mc = m0 < g.M ? m0 : 0;
      const int64_t r = g.L == 1 ? mc : mc / g.L, l = mc - r * g.L;
      const int64_t moff = l + LI * r;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (m0 + j < g.M) {
          maskA |= 1u << j;
          if (MNC && !VEC) {
            const int64_t rj = (mc + j) / g.L;
            mrel[j] = (int)((mc + j - rj * g.L) + LI * rj - moff);
          }
        }
      }
      pA = x + moff + g.L * kA;
      mexp4 = g.mexp + m0;
      cA = kA < g.I ? (int)((g.I - kA + BK - 1) / BK) : 0;
    };
    auto load4 = [&](uint32_t dst, const T* p, unsigned m) {
      constexpr int PER = 16 / (int)sizeof(T);             // values per chunk
      if (VEC && (m == 15u || m == 0u)) {
#pragma unroll
        for (int c = 0; c < 4 / PER; ++c) cp_async<16>(dst + c * CHUNK, m ? p + PER * c : x, m != 0u);
        return;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool ok = m >> j & 1u;
        const T* q = p + (MNC ? (TTM && !VEC ? mrel[j] : j) : (TTM ? g.I : g.L) * j);
        cp_async<sizeof(T)>(dst + (j / PER) * CHUNK + (j % PER) * sizeof(T), ok ? q : x, ok);
      }
    };
    // Loads of the next stage to load (one group; nothing past the end), into
    // the raw slot `ro`; myB: the stage has this warp's quad of the 64-row operand.
    auto load = [&](bool any, uint32_t ro, bool myB, uint32_t rb) {
      if (any) {
        load4(smem_u32(raw) + ro, pA, cA > 0 ? maskA : 0u);
        --cA;
        pA += stepA;
        if (!TTM && !MNC) {
          lA += BK;
          while (lA >= Li) { lA -= Li; pA += LI - g.L; }
        }
        if (!TTM && myB) {
          load4(smem_u32(raw) + NRAW * RAW_A + rb, pB, cB > 0 ? maskB : 0u);
          --cB;
          pB += 2 * stepA;
          if (!MNC) {
            lB += 2 * BK;
            while (lB >= Li) { lB -= Li; pB += LI - g.L; }
          }
        }
        if (TTM) {
          cp_async<8>(smem_u32(raw) + NRAW * RAW_A + ro / 2, mexp4, true);
          if (++ks == g.nks) {
            ks = 0;
            item += gridDim.x;
            if (item < g.nitems) tile_setup();
          }
        }
      }
      cp_commit();
    };
    if (TTM) tile_setup();
    int bks = 0, bnt = TTM ? (int)(blockIdx.x % g.ntn) : 0;  // operator image of the next stage
    uint32_t rslot = 0, rbslot = 0;                        // raw slots of the next stage to split
#pragma unroll
    for (int t = 0; t < NRAW; ++t)
      load(t < nst, t * RAW_A, !diag && (warp >> 3) == (t & 1), (t >> 1) * RAW_A);

    Sum96 acc[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[j] = Sum96{0u, 0u, 0u};
    const uint32_t taddr = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 16u * (uint32_t)(warp >> 2);
    uint32_t wins = 0;                                     // windows drained
    int64_t oitem = blockIdx.x;                            // TTM: item of the next output
    int tend = wst;                                        // end of the tile of the next window to drain
    int wend = tend < WIN ? tend : WIN;                    // end of that window
    int slot = 0;
    uint32_t ph = 1;                                       // parity of the slot's next emptying
    bool ok = true;
    for (int s = 0; s < nst && ok; ++s) {
      if (s >= NST && !mbar_wait(smem_u32(&bar_empty[slot]), ph, g.err)) { ok = false; break; }
      uint8_t* st = smem + (size_t)slot * STAGE_BYTES;
      if (TTM) {
        if (threadIdx.x == 0) {
          mbar_expect_tx(smem_u32(&bar_full[slot]), B_BYTES);
          bulk_g2s(smem_u32(st + A_BYTES), g.bimg + ((size_t)bnt * g.nks + bks) * B_BYTES, B_BYTES,
                   smem_u32(&bar_full[slot]));
          if (++bks == g.nks) {
            bks = 0;
            bnt = (int)((bnt + gridDim.x) % g.ntn);
          }
        }
      }
      cp_wait<NRAW - 1>();
      T v[4];
      if (TTM) {
        const uint2 e = *reinterpret_cast<const uint2*>(raw + NRAW * RAW_A + rslot / 2);
        eA[0] = shift_base((int)(e.x & 0xffffu), T());
        eA[1] = shift_base((int)(e.x >> 16), T());
        eA[2] = shift_base((int)(e.y & 0xffffu), T());
        eA[3] = shift_base((int)(e.y >> 16), T());
      }
      raw_quad(raw + rslot, v);
      store_quad(st + oA, 2 * ATOM, v, eA);
      const bool myB = !TTM && !diag && (warp >> 3) == (s & 1);
      if (myB) {
        raw_quad(raw + NRAW * RAW_A + rbslot, v);
        store_quad(st + oB, ATOM, v, eB);
      }
      load(s + NRAW < nst, rslot, myB, rbslot);            // into the slots just read
      rslot = rslot == (NRAW - 1) * RAW_A ? 0u : rslot + RAW_A;
      if (myB) rbslot ^= RAW_A;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_full[slot]));
      if (++slot == NST) { slot = 0; ph ^= 1u; }
      // Drain the finished window.  Until the ring is full behind it (or the
      // stages end) the tensor cores may still be at it: go on producing.
      while (wend <= s + 1 && ok) {
        const bool last = s + 1 == nst || s + 1 - wend >= NST;
        if (last) {
          if (!mbar_wait(smem_u32(&bar_accf), wins & 1u, g.err)) { ok = false; break; }
        } else if (!__any_sync(0xffffffffu, mbar_test(smem_u32(&bar_accf), wins & 1u))) {
          break;                                           // (the whole warp takes one decision)
        }
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;");
        drain(taddr, acc);
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_acce));
        ++wins;
        const bool tile_done = wend == tend;
        if (TTM && tile_done) {
          // the tile's outputs
          const int64_t m = (oitem / g.ntn) * MT + 32 * (warp & 3) + lane;
          const int nt = (int)(oitem % g.ntn), k0 = nt * NT + 16 * (warp >> 2);
          if (m < g.M) {
            const int em = (int)g.mexp[m];
            const int64_t r = g.L == 1 ? m : m / g.L, l = m - r * g.L;
            const int64_t kst = g.zt ? g.M : g.L;
            TOut* z = static_cast<TOut*>(g.z) + (g.zt ? m : l + g.L * g.K * r) + kst * k0;
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (k0 + j < g.K)
                z[kst * j] = (TOut)to_double(acc[j], em + (int)__ldg(g.kexp + k0 + j) + OUT_EXP);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[j] = Sum96{0u, 0u, 0u};
          oitem += gridDim.x;
        }
        if (tile_done) tend += wst;
        wend = wend + WIN < tend ? wend + WIN : tend;
        if (wend > nst) break;
      }
    }
    if (!TTM) {
      // partial tile [col][row]
      double* pt = g.part + (size_t)blockIdx.x * TILE_ELEMS;
      const int row = 32 * (warp & 3) + lane, c0 = 16 * (warp >> 2);
#pragma unroll
      for (int j = 0; j < 16; ++j) pt[(c0 + j) * MT + row] = to_double(acc[j], 0);
    }
  }
  mbar_wait(smem_u32(&bar_done), 0, g.err);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

// S[i][j] = S[j][i] = 2^(E_i + E_j - 70) times the sum over the K splits (in
// order) of tile (ta, tb) at [col][row], i >= j; NaN when *bad.
__global__ void __launch_bounds__(256) k_digit64_reduce(const double* __restrict__ part, int ntiles,
                                                        int nkg, int64_t I,
                                                        const unsigned* __restrict__ rexp,
                                                        const unsigned* __restrict__ bad,
                                                        double* __restrict__ S) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t i = idx % I, j = idx / I;
  if (j > i || j >= I) return;
  const int ta = (int)(i / MT), tb = (int)(j / NT);
  const int t = ta * (ta + 1) + tb;
  const double* p = part + (size_t)t * TILE_ELEMS + (size_t)(j - (int64_t)tb * NT) * MT + (i - (int64_t)ta * MT);
  const size_t step = (size_t)ntiles * TILE_ELEMS;
  double s = 0.0;
  if (*bad) {
    s = __longlong_as_double(0x7ff8000000000000ll);
  } else {
    for (int k = 0; k < nkg; k += 8) {
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = k + q < nkg ? p[step * (k + q)] : 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) s += v[q];
    }
    s = scalbn(s, (int)rexp[i] + (int)rexp[j] + OUT_EXP);
  }
  S[i * I + j] = s;
  S[j * I + i] = s;
}

// Row maxima (magnitude bits) of the (L I) x Rt matrix of virtual rows
// q = l + L i (row i = q / L): a thread keeps one virtual row over a range of
// columns.  Blocks hold `cpb` columns of `rows` virtual rows at a time.
template <typename T>
__global__ void __launch_bounds__(256) k_rowexp_cols(const T* __restrict__ x, int64_t nrows,
                                                     int64_t L, int64_t ncols, int rows, int cpb,
                                                     unsigned* __restrict__ rexp) {
  const int tr = threadIdx.x % rows, tc = threadIdx.x / rows;
  const int64_t q = (int64_t)blockIdx.y * rows + tr;
  if (tc >= cpb || q >= nrows) return;
  const int64_t step = (int64_t)gridDim.x * cpb;
  int64_t c = (int64_t)blockIdx.x * cpb + tc;
  const T* p = x + q;
  int m = 0;
  for (; c + 7 * step < ncols; c += 8 * step) {
    T v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = __ldg(p + nrows * (c + u * step));
#pragma unroll
    for (int u = 0; u < 8; ++u) m = max(m, mag_bits(v[u]));
  }
  for (; c < ncols; c += step) m = max(m, mag_bits(__ldg(p + nrows * c)));
  atomicMax(rexp + q / L, (unsigned)m);
}

// The same for long runs: one warp per (row i, run of slabs), lanes along l.
template <typename T>
__global__ void __launch_bounds__(256) k_rowexp_runs(const T* __restrict__ x, int64_t L, int64_t I,
                                                     int64_t Rt, int nck,
                                                     unsigned* __restrict__ rexp) {
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (gw >= I * nck) return;
  const int64_t i = gw % I, ck = gw / I;
  const int64_t e0 = Rt * L * ck / nck, e1 = Rt * L * (ck + 1) / nck;   // range of (r, l), l fastest
  int m = 0;
  int64_t r = e0 / L, l = e0 - r * L;
  int64_t left = e1 - e0;
  while (left > 0) {
    const int64_t n = L - l < left ? L - l : left;
    const T* row = x + L * (i + I * r) + l;
    int64_t t = lane;
    for (; t + 96 < n; t += 128) {
      const T a = __ldg(row + t), b = __ldg(row + t + 32), c = __ldg(row + t + 64), d = __ldg(row + t + 96);
      m = max(m, max(max(mag_bits(a), mag_bits(b)), max(mag_bits(c), mag_bits(d))));
    }
    for (; t < n; t += 32) m = max(m, mag_bits(__ldg(row + t)));
    left -= n;
    l = 0;
    ++r;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) atomicMax(rexp + i, (unsigned)m);
}

// Row maxima (magnitude bits) to exponents, in place.
template <typename T>
__global__ void k_rowexp_final(unsigned* __restrict__ rexp, int64_t I, int small,
                               unsigned* __restrict__ bad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= I) return;
  const int e = row_exp((int)rexp[i], T(), small);
  rexp[i] = (unsigned)e;
  if (e == BAD_EXP) atomicOr(bad, 1u);
}

}  // namespace

GramPlan plan_gram_d64(int64_t L, int64_t I, int64_t Rt, int num_sms) {
  GramPlan p;
  if (I < 1 || I > 8192 || L < 1 || Rt < 1 || L * I >= ((int64_t)1 << 31)) return p;
  const double K = (double)L * (double)Rt, II = (double)I * (double)I;
  if (I < 64 ? (II - kDigit64SmallII) * K < kDigit64SmallGram : II * K < kDigit64MinGram) return p;
  const int64_t stages = (L * Rt + BK - 1) / BK;
  const int TA = (int)((I + MT - 1) / MT), TB = (int)((I + NT - 1) / NT);
  int ntiles = 0;
  for (int a = 0; a < TA; ++a) ntiles += std::min(2 * a + 2, TB);
  int64_t k = std::max(1, num_sms / ntiles);
  // at least four stages per CTA
  k = std::min<int64_t>(k, std::max<int64_t>(1, stages / 4));
  // the 96-bit sums hold 2^25 k of the largest products
  k = std::max<int64_t>(k, (stages + (1 << 20) - 1) >> 20);
  p.ntiles = ntiles;
  p.ksplit = (int)k;
  p.nctas = (int)(ntiles * k);
  p.scratch_bytes = (size_t)p.nctas * TILE_ELEMS * sizeof(double) + sizeof(unsigned) * (size_t)(I + 2);
  return p;
}

template <typename T>
static cudaError_t launch_rowexp(const T* x, int64_t L, int64_t I, int64_t Rt, int num_sms,
                                 int small, unsigned* rexp, unsigned* bad, cudaStream_t st) {
  // rexp[I], rexp[I + 1]: the verdict words
  cudaError_t e = cudaMemsetAsync(rexp, 0, sizeof(unsigned) * (size_t)(I + 2), st);
  if (e != cudaSuccess) return e;
  if (L < 32) {
    const int64_t nrows = L * I, gy = (nrows + 255) / 256;
    const int rows = (int)((nrows + gy - 1) / gy), cpb = 256 / rows;
    int64_t gx = std::max<int64_t>(1, (int64_t)num_sms * 8 / gy);
    gx = std::min<int64_t>(gx, (Rt + cpb - 1) / cpb);
    k_rowexp_cols<T><<<dim3((unsigned)gx, (unsigned)gy), 256, 0, st>>>(x, nrows, L, Rt, rows, cpb,
                                                                       rexp);
  } else {
    int64_t nck = ((int64_t)num_sms * 64 + I - 1) / I;
    nck = std::max<int64_t>(1, std::min<int64_t>(nck, L * Rt / 128));
    const int64_t warps = I * nck;
    k_rowexp_runs<T><<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(x, L, I, Rt, (int)nck, rexp);
  }
  k_rowexp_final<T><<<(unsigned)((I + 255) / 256), 256, 0, st>>>(rexp, I, small, bad);
  count_launches(2);
  return cudaGetLastError();
}

template <typename T, bool MNC, bool VEC>
static cudaError_t run_gram_d64(const Args& a, int nctas, cudaStream_t st) {
  cudaError_t e = allow_max_dyn_smem((const void*)k_digit64<T, double, false, MNC, VEC>);
  if (e != cudaSuccess) return e;
  k_digit64<T, double, false, MNC, VEC><<<(unsigned)nctas, NTHREADS, SMEM_BYTES, st>>>(a);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t gram_d64(const T* y, int64_t L, int64_t I, int64_t Rt, const GramPlan& p,
                            int num_sms, void* scratch, unsigned* err, double* S,
                            cudaStream_t st) {
  double* part = static_cast<double*>(scratch);
  unsigned* rexp = reinterpret_cast<unsigned*>(part + (size_t)p.nctas * TILE_ELEMS);
  unsigned* bad = rexp + I;
  cudaError_t e = launch_rowexp(y, L, I, Rt, num_sms, err == nullptr, rexp, bad, st);
  if (e != cudaSuccess) return e;
  Args a{};
  a.x = y;
  a.L = L;
  a.I = I;
  a.Rt = Rt;
  a.nk = L * Rt;
  a.err = err ? err : bad + 1;
  a.bad = bad;
  a.ntiles = p.ntiles;
  a.nkg = p.ksplit;
  a.rexp = rexp;
  a.part = part;
  const bool vec = L == 1 && I % (16 / sizeof(T)) == 0 && ((uintptr_t)y & 15) == 0;
  e = L > 1 ? run_gram_d64<T, false, false>(a, p.nctas, st)
            : vec ? run_gram_d64<T, true, true>(a, p.nctas, st)
                  : run_gram_d64<T, true, false>(a, p.nctas, st);
  if (e != cudaSuccess) return e;
  const int64_t tot = I * I;
  k_digit64_reduce<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(part, p.ntiles, p.ksplit, I, rexp,
                                                                 bad, S);
  count_launches(2);
  return cudaGetLastError();
}

const unsigned* gram_d64_verdict(const GramPlan& p, int64_t I, const void* scratch) {
  return reinterpret_cast<const unsigned*>(static_cast<const double*>(scratch) +
                                           (size_t)p.nctas * TILE_ELEMS) + I;
}

cudaError_t launch_gram_d64(const void* y, tucker_dtype dt, int64_t L, int64_t I, int64_t Rt,
                            const GramPlan& p, int num_sms, void* scratch, unsigned* err, double* S,
                            cudaStream_t st) {
  if (p.nctas <= 0) return cudaErrorInvalidValue;
  return dt == TUCKER_F64
             ? gram_d64((const double*)y, L, I, Rt, p, num_sms, scratch, err, S, st)
             : gram_d64((const float*)y, L, I, Rt, p, num_sms, scratch, err, S, st);
}

// ------------------------------------------------------------------ TTM

// Exponents of the largest magnitude over i of every m = (l, r): a thread per
// m when the m are contiguous (L > 1) ...
template <typename T>
__global__ void __launch_bounds__(256) k_mexp_rows(const T* __restrict__ y, int64_t L, int64_t I,
                                                   int64_t M, int small,
                                                   uint16_t* __restrict__ mexp,
                                                   unsigned* __restrict__ bad) {
  const int64_t m = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (m >= M || *bad) return;                            // (*bad: the operator's)
  const int64_t r = m / L, l = m - r * L;
  const T* p = y + l + L * I * r;
  int b = 0;
  int64_t i = 0;
  for (; i + 8 <= I; i += 8) {
    T v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = __ldg(p + L * (i + u));
#pragma unroll
    for (int u = 0; u < 8; ++u) b = max(b, mag_bits(v[u]));
  }
  for (; i < I; ++i) b = max(b, mag_bits(__ldg(p + L * i)));
  const int e = row_exp(b, T(), small);
  mexp[m] = (uint16_t)e;
  if (e == BAD_EXP) atomicOr(bad, 1u);
}

// ... and a warp per m (four at a time) when the contraction is (L == 1).
template <typename T>
__global__ void __launch_bounds__(256) k_mexp_cols(const T* __restrict__ y, int64_t I, int64_t M,
                                                   int small, uint16_t* __restrict__ mexp,
                                                   unsigned* __restrict__ bad) {
  const int64_t m0 = 4 * (((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (m0 >= M || __shfl_sync(0xffffffffu, *bad, 0)) return;   // (*bad: the operator's)
  int e[4] = {0, 0, 0, 0};
  const T* p = y + m0 * I;
  for (int64_t i = lane; i < I; i += 64) {
    T v[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        v[j][u] = (m0 + j < M && i + 32 * u < I) ? __ldg(p + j * I + i + 32 * u) : (T)0;
#pragma unroll
    for (int j = 0; j < 4; ++j) e[j] = max(e[j], max(mag_bits(v[j][0]), mag_bits(v[j][1])));
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e[j] = max(e[j], __shfl_xor_sync(0xffffffffu, e[j], o));
    if (lane == 0 && m0 + j < M) {
      const int x = row_exp(e[j], T(), small);
      mexp[m0 + j] = (uint16_t)x;
      if (x == BAD_EXP) atomicOr(bad, 1u);
    }
  }
}

// Stage images of the operator A (K x I FP64): block (ks, nt) writes the digit
// planes of rows k = 64 nt.., columns i = 32 ks.. (zero outside K x I) in the
// 64-row operand's layout; kexp[64 nt + row] = the row's exponent.
__global__ void __launch_bounds__(256) k_digit64_prep(const double* __restrict__ A, int K,
                                                      int64_t I, int64_t lda, int arow, int small,
                                                      uint8_t* __restrict__ img,
                                                      unsigned* __restrict__ kexp,
                                                      unsigned* __restrict__ bad) {
  __shared__ int eb[NT], zeros[NT];
  const int ks = blockIdx.x, nt = blockIdx.y, nks = gridDim.x;
  if (threadIdx.x < NT) eb[threadIdx.x] = zeros[threadIdx.x] = 0;
  __syncthreads();
  auto at = [&](int k, int64_t i) { return arow ? A[(int64_t)k * lda + i] : A[k + lda * i]; };
  if (arow) {                                       // i contiguous: a warp per row
    for (int row = threadIdx.x >> 5; row < NT; row += 8) {
      const int k = nt * NT + row;
      int e = 0;
      bool zero = false;
      if (k < K)
        for (int64_t i = threadIdx.x & 31; i < I; i += 32) {
          const int m = mag_bits(at(k, i));
          e = max(e, m);
          zero |= m == 0;
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
      zero = __any_sync(0xffffffffu, zero);
      if ((threadIdx.x & 31) == 0) { eb[row] = e; zeros[row] = zero; }
    }
  } else {
    const int row = threadIdx.x & (NT - 1), k = nt * NT + row;
    int e = 0;
    bool zero = false;
    if (k < K)
      for (int64_t i = threadIdx.x / NT; i < I; i += 256 / NT) {
        const int m = mag_bits(at(k, i));
        e = max(e, m);
        zero |= m == 0;
      }
    atomicMax(&eb[row], e);
    if (zero) zeros[row] = 1;
  }
  __syncthreads();
  // (a row of zeros gives zeros either way)
  if (ks == 0 && small && threadIdx.x < NT && zeros[threadIdx.x] && eb[threadIdx.x]) atomicOr(bad, 1u);
  __syncthreads();
  if (threadIdx.x < NT) eb[threadIdx.x] = row_exp(eb[threadIdx.x], 0.0, small);
  __syncthreads();
  if (ks == 0 && threadIdx.x < NT) {
    kexp[nt * NT + threadIdx.x] = (unsigned)eb[threadIdx.x];
    if (eb[threadIdx.x] == BAD_EXP) atomicOr(bad, 1u);
  }
  uint8_t* out = img + (size_t)(nt * nks + ks) * B_BYTES;
  for (int q = threadIdx.x; q < (NT / 4) * BK; q += 256) {
    // arow: threads along i, else along the rows
    const int mn = arow ? 4 * (q / BK) : 4 * (q % (NT / 4)), k = arow ? q % BK : q / (NT / 4);
    const int64_t i = (int64_t)ks * BK + k;
    double v[4];
    uint32_t e4[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = (nt * NT + mn + j < K && i < I) ? at(nt * NT + mn + j, i) : 0.0;
      e4[j] = shift_base(eb[mn + j], 0.0);
    }
    store_quad(out + mn_off(mn, k, KG_B), ATOM, v, e4);
  }
}

int ttm_d64_supported(int64_t L, int64_t I, int64_t Rt, int64_t K) {
  return I >= 1 && I <= 65536 && K >= 1 && K <= 65536 && L >= 1 && Rt >= 1 &&
         L * I < ((int64_t)1 << 31);
}

int ttm_d64_chosen(int64_t L, int64_t I, int64_t Rt, int64_t K, int num_sms) {
  if (!ttm_d64_supported(L, I, Rt, K)) return 0;
  const double M = (double)L * (double)Rt;
  if (I < kDigit64MinTtmI && 2.0 * (double)K * (double)I * M < kDigit64MinTtm) return 0;
  return ttm_digit_us(M, (double)I, (double)K, num_sms, L == 1) <
         ttm_pipe_us(M, (double)I, (double)K, num_sms);
}

namespace {
struct TtmScratch {
  size_t img, mexp, kexp, bad, bytes;
};
TtmScratch ttm_d64_layout(int64_t L, int64_t I, int64_t Rt, int64_t K) {
  const size_t ntn = (size_t)((K + NT - 1) / NT), nks = (size_t)((I + BK - 1) / BK);
  const size_t mpad = (size_t)((L * Rt + MT - 1) / MT) * MT;
  TtmScratch s;
  s.img = 0;
  s.mexp = ntn * nks * B_BYTES;
  s.kexp = s.mexp + mpad * sizeof(uint16_t);
  s.bad = s.kexp + ntn * NT * sizeof(unsigned);
  s.bytes = s.bad + 16;
  return s;
}
}  // namespace

size_t ttm_d64_scratch_bytes(int64_t L, int64_t I, int64_t Rt, int64_t K) {
  return ttm_d64_layout(L, I, Rt, K).bytes;
}

const unsigned* ttm_d64_verdict(int64_t L, int64_t I, int64_t Rt, int64_t K, const void* scratch) {
  return reinterpret_cast<const unsigned*>(static_cast<const uint8_t*>(scratch) +
                                           ttm_d64_layout(L, I, Rt, K).bad);
}

template <typename T, typename TOut>
static cudaError_t ttm_d64(const T* y, int64_t L, int64_t I, int64_t Rt, const double* A, int64_t K,
                           int64_t lda, int arow, TOut* z, bool zt, uint8_t* scr, unsigned* err,
                           int num_sms, cudaStream_t st) {
  const TtmScratch lay = ttm_d64_layout(L, I, Rt, K);
  uint16_t* mexp = reinterpret_cast<uint16_t*>(scr + lay.mexp);
  unsigned* kexp = reinterpret_cast<unsigned*>(scr + lay.kexp);
  unsigned* bad = reinterpret_cast<unsigned*>(scr + lay.bad);
  cudaError_t e = cudaMemsetAsync(bad, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  Args a{};
  a.x = y;
  a.L = L;
  a.I = I;
  a.Rt = Rt;
  a.nk = I;
  a.err = err ? err : bad + 1;
  a.bad = bad;
  a.M = L * Rt;
  a.K = (int)K;
  a.ntn = (int)((K + NT - 1) / NT);
  a.nks = (int)((I + BK - 1) / BK);
  a.nitems = (a.M + MT - 1) / MT * a.ntn;
  a.mexp = mexp;
  a.bimg = scr + lay.img;
  a.kexp = kexp;
  a.z = z;
  a.zt = zt ? 1 : 0;
  const int small = err == nullptr;                      // the caller reads the verdict
  a.waits = small;
  k_digit64_prep<<<dim3((unsigned)a.nks, (unsigned)a.ntn), 256, 0, st>>>(A, (int)K, I, lda, arow,
                                                                        small, scr + lay.img, kexp, bad);
  if (L > 1)
    k_mexp_rows<T><<<(unsigned)((a.M + 255) / 256), 256, 0, st>>>(y, L, I, a.M, small, mexp, bad);
  else
    k_mexp_cols<T><<<(unsigned)((a.M + 31) / 32), 256, 0, st>>>(y, I, a.M, small, mexp, bad);
  const unsigned grid = (unsigned)std::min<int64_t>(a.nitems, num_sms);
  const bool vec = L > 1 && L % 4 == 0 && ((uintptr_t)y & 15) == 0;
  auto go = [&](auto kern) -> cudaError_t {
    cudaError_t ee = allow_max_dyn_smem((const void*)kern);
    if (ee != cudaSuccess) return ee;
    kern<<<grid, NTHREADS, SMEM_BYTES, st>>>(a);
    return cudaGetLastError();
  };
  e = L == 1 ? go(k_digit64<T, TOut, true, false, false>)
             : vec ? go(k_digit64<T, TOut, true, true, true>)
                   : go(k_digit64<T, TOut, true, true, false>);
  count_launches(3);
  return e;
}

cudaError_t launch_ttm_d64(const void* y, tucker_dtype ydt, int64_t L, int64_t I, int64_t Rt,
                           const double* A, int64_t K, int64_t lda, int a_rowmajor, void* z,
                           tucker_dtype zdt, bool zt, void* scratch, unsigned* err, int num_sms,
                           cudaStream_t st) {
  if (!ttm_d64_supported(L, I, Rt, K) || (zt && L != 1)) return cudaErrorInvalidValue;
  uint8_t* scr = static_cast<uint8_t*>(scratch);
  if (ydt == TUCKER_F64)
    return zdt == TUCKER_F64
               ? ttm_d64((const double*)y, L, I, Rt, A, K, lda, a_rowmajor, (double*)z, zt, scr, err, num_sms, st)
               : ttm_d64((const double*)y, L, I, Rt, A, K, lda, a_rowmajor, (float*)z, zt, scr, err, num_sms, st);
  return zdt == TUCKER_F64
             ? ttm_d64((const float*)y, L, I, Rt, A, K, lda, a_rowmajor, (double*)z, zt, scr, err, num_sms, st)
             : ttm_d64((const float*)y, L, I, Rt, A, K, lda, a_rowmajor, (float*)z, zt, scr, err, num_sms, st);
}

}  // namespace tk
