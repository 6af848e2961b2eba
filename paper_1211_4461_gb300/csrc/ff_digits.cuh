// Stage 1 of the 2D far field on the tensor cores, exactly: both operands are
// cut into 8-bit digits of a fixed-point representation, every digit product
// and its sums are integers that FP32 accumulation holds without rounding, and
// the digit sums join in double-float arithmetic.
//
// Representation.  As in the double-float form, each row of either operand is
// scaled by a power of two per block of 32 nodes, so |x'| < 1 there.  Then
//   x' = sum_{s=1..n} d_s 2^-(8 s - 1) + r,   |d_s| <= 128,  |r| <= 2^-8n,
// n = 7 or 8, digits balanced (round to nearest), stored as BF16 integers.  A product
// of two digits is at most 2^14; a block's sum over 64 real terms (32 complex nodes)
// and the at most 8 digit pairs (s, t) of one diagonal s + t = D stays within
// 2^23, so the FP32 accumulators hold it exactly.  Diagonals D = 2..9 are kept (36
// of the 64 pairs of eight digits, 34 of seven's 49).  Cutting into slices whose
// products add up exactly is a published method (Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012).
//
// Error of a block, relative to the product 2^(ex + eg) of the two scales: seven
// (five) pairs of at most 2^14 at 2^-78 are dropped for each of 64 real products
// (2^-55.2; 2^-61 for digits of random signs), and seven digits leave remainders of up
// to 2^-56 (2^-54.8 rms for dense blocks, less where few values count).
//
// When it runs.  This error is relative to the block maxima, so the kernel is
// taken when for every block that a tile keeps the scales ex + eg lie at most
// MARGIN binades over L, the lower bound of the sum of the terms' magnitudes that
// the skip kernel forms (-3 to 2 for constant phases, more as they vary over a block:
// up to about k h sin(gamma) 32 = 9), with seven digits up to MARGIN_7 (4.5).  Up
// to either line the error stays below the double-float kernel's, which runs beyond
// the second.  Both restated on the CPU on single blocks against a longer sum,
// relative to the sum of the terms' magnitudes, by margin, as binades of the rms
// error over the double-float kernel's (2^-48.5 to 2^-45.7):
//                          seven digits, margin 6    8     9     10   eight, 10    13    15    16    17
//   random fields                          -3.3  -3.2                    -3.2  -3.0  -2.9  -2.9  -3.1
//   balanced against the phases            -3.7  -2.0  -1.4  -0.6        -4.3  -3.7  -2.3  -1.5  -0.5
//   falling three times as fast            -3.7  -1.9  -1.1  -0.6        -4.8  -3.6  -2.0  -0.9  +0.1
//   three nodes at the smallest phase      -2.2  -0.9  +0.1  +0.7        -2.6  -2.4  -0.8  +0.1  +0.8
//   a single node there                    -1.8  -0.8  +0.1  +1.0        -2.1  -1.9  -0.7  +0.3  +1.2
// (Seven digits with diagonals up to 8 and the line at 12 binades over a bound from
// single nodes, as before: up to 3.9 binades larger than the double-float kernel's.)
// On whole maps (129^2, fields at the small end of the phases, 2 to 14 binades a
// block) the eight digits lie 2^-50.3 of the terms from the FP64 contraction or less.
//
// Kernel.  D[rho][j] = sum_K A[rho][K] B[j][K], K = (re, im) of 32 nodes; a
// CTA takes 128 rows of g (A) and 16 phase rows (B: rows j < 16 give the real
// parts from (P_re, -P_im), 16 + j the imaginary parts from (P_im, P_re)).  The
// 32 rows of digit t of B are rows [32 (t - 1), 32 t) of one operand, and
// diagonal D accumulates in tensor-memory columns [32 (D - 2), 32 (D - 1)), so
// one MMA of digit s of A against digits 1..9-s of B (N = 32 (9 - s), at most all
// there are) adds to the right diagonals: one MMA a digit per 16 K values, each
// reading A once, and with seven digits one more where the last diagonal starts.
// One thread streams digit tiles (16 KB, pre-swizzled in global memory) into a
// ring with bulk copies, one issues the MMAs, sixteen warps read the two
// alternating sets of accumulators and join them, all handing over through
// mbarriers with bounded waits.
#pragma once

#include <cuda_bf16.h>

#include "csff_internal.h"
#include "df_bits.cuh"

namespace csff {
namespace digits {

constexpr int TM = 128, TK = 16;               // rows of g and phase rows of a tile
constexpr int KB = 32;                         // nodes of a block
constexpr int A_DIG = TM * 128;                // bytes of a digit of an A block (128-byte rows)
constexpr int B_DIG = 2 * TK * 128;
constexpr int MAX_NB = 1024;                   // blocks of a row
constexpr int EPI_WARPS = 16, NT = 32 * (EPI_WARPS + 2);
constexpr int EK = TK * 4 / EPI_WARPS;           // phase rows of an epilogue warp
constexpr int TMEM_COLS = 512, ACC = 256;      // columns of one set of accumulators, one diagonal in 32
constexpr int MARGIN = 15, MARGIN_7 = 8;

// A form of the contraction: NA A slots in the ring, SUB scale blocks in the 32 nodes
// of a row of B.
//  2D: one block, an A slot one digit of 32 nodes; seven or eight digits.
//  3D (the z and y contractions): two blocks, an A slot two digits of 16 nodes, eight
//  digits; each block's diagonals fill a set of accumulators.
constexpr int ND = 8;                          // digits at most, and diagonals kept
constexpr int B_SET = ND * B_DIG;
template <int NA_, int SUB_> struct Form {
  static constexpr int NA = NA_, SUB = SUB_;
  static constexpr int A_SLOTS = ND / SUB;     // slots of a block of eight digits
  static constexpr int OFF_BAR = NA * A_DIG + 2 * B_SET, OFF_ACT = OFF_BAR + 512;
  static constexpr int SMEM = OFF_ACT + MAX_NB * 2 + 1024;
  static_assert(SMEM <= 227 * 1024 && ND % SUB == 0 && 2 * TK * ND <= ACC, "shared and tensor memory");
};
using Form2 = Form<9, 1>;
using Form3 = Form<9, 2>;

// 128-byte-swizzled K-major row: byte offset of 16-byte chunk c of row r
__device__ __forceinline__ int sw(int r, int c) { return (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4); }

// x 2^(8 N - 1 - e) rounded to an integer, |x| < 2^e, from the IEEE fields
template <int N = ND> __device__ __forceinline__ long long fixed(double x, int e) {
  constexpr int BITS = 8 * N - 1;
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7ff);
  const long long m = (long long)((b & bits::MANT_MASK) | (E ? 1ull << 52 : 0));
  const int sh = max(E, 1) - 1075 + BITS - e;  // m 2^(max(E, 1) - 1075) 2^(BITS - e)
  long long q;
  if (sh >= 0) q = m << min(sh, 62);
  else if (sh < -54) q = 0;
  else q = (m + (1ll << (-sh - 1))) >> -sh;
  return E == 0x7ff ? 0 : (b >> 63) ? -q : q;
}
// e with |x| < 2^e from the exponent fields (zero and subnormal values: -1022;
// infinities and NaN, whose digits are zero: 1025)
__device__ __forceinline__ int scale_exp(double2 x) { return max(bits::exp_field(x.x), bits::exp_field(x.y)) - 1022; }

// the scale of a block of the 3D form that holds an infinity or a NaN: what it
// enters becomes NaN
constexpr int NONFINITE = 1 << 24;
__device__ __forceinline__ int block_scale(int e) { return e > 1024 ? NONFINITE : e; }

// the digits of two fixed-point values as pairs of BF16 integers, dig[0] the
// leading one.  Balanced digits are the bytes after adding 128 to every byte
// below the leading one, less 128; a byte becomes a float in the mantissa of
// 2^23 (a full-rate subtraction where a conversion runs at a quarter), whose
// upper half is the BF16 value.
__device__ __forceinline__ float byte_digit(unsigned v, int byte) {
  return __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7440 | byte)) - 8388736.f;      // 2^23 + 128
}
template <int N = ND> __device__ __forceinline__ void cut(long long p, long long q, uint32_t (&dig)[N]) {
  constexpr int SH = 8 * (N - 1);
  constexpr unsigned long long LOW = (1ull << SH) - 1, HALF = 0x8080808080808080ull & LOW;
  const unsigned long long lp = ((unsigned long long)p & LOW) + HALF, lq = ((unsigned long long)q & LOW) + HALF;
  auto pack = [](float a, float b) { return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632); };
#pragma unroll
  for (int s = 1; s < N; ++s) {
    const int byte = N - 1 - s;
    const unsigned a = (unsigned)(byte < 4 ? lp : lp >> 32), b = (unsigned)(byte < 4 ? lq : lq >> 32);
    dig[s] = pack(byte_digit(a, byte & 3), byte_digit(b, byte & 3));
  }
  auto top = [&](long long v, unsigned long long low) {
    return __int_as_float(0x4B400000 + (int)(v >> SH) + (int)(low >> SH)) - 12582912.f;
  };
  dig[0] = pack(top(p, lp), top(q, lq));
}
__device__ __forceinline__ uint32_t neg_hi(uint32_t v) { return v ^ 0x80000000u; }      // (a, b) -> (a, -b)
__device__ __forceinline__ uint32_t swap_pair(uint32_t v) { return (v >> 16) | (v << 16); }

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t desc(uint32_t a) {
  return (uint64_t)((a & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// bounded; gives up early when another thread of the CTA has
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, volatile int* abort,
                                         unsigned long long limit = FF_WAIT_NS) {
  unsigned long long t0 = 0;
  for (int it = 0; it < (1 << 28); ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 63) == 63) {
      if (*abort) return false;
      unsigned long long t;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
      if (t0 == 0) t0 = t;
      else if (t - t0 > limit) break;
    }
  }
  *abort = 1;
  return false;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
#define CSFF_TMEM_LD4(v, addr)                                                     \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"        \
               : "=r"((v)[0]), "=r"((v)[1]), "=r"((v)[2]), "=r"((v)[3])            \
               : "r"(addr))

// two sums at once (packed two-lane FP32): t + e = x + y exactly
__device__ __forceinline__ void two_sum(float2 x, float2 y, float2& t, float2& e) {
  const float2 m1 = make_float2(-1.f, -1.f);
  t = __fadd2_rn(x, y);
  const float2 v = __ffma2_rn(x, m1, t);
  e = __fadd2_rn(__ffma2_rn(__ffma2_rn(v, m1, t), m1, x), __ffma2_rn(v, m1, y));
}
// 2^d for d <= 0, zero from d = -127 on (terms that small add nothing)
__device__ __forceinline__ float pow2_or_0(int d) { return __int_as_float(max(d + 127, 0) << 23); }
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }

// h + l = sum_{d=0..7} p[d] 2^-8d: the six leading terms by exact sums (their digit
// sums reach 2^23, eight bits apart), the two trailing ones, whose roundings lie
// below 2^-49 of p[0]'s unit, the size of the last bits of a value 15 binades under
// the scales, by multiply-adds
__device__ __forceinline__ void join(const float2 (&p)[8], float2& h, float2& l) {
  const float2 w = both(0x1p-8f);
  float2 t = __ffma2_rn(p[7], w, p[6]), e, c;
  two_sum(p[5], __fmul2_rn(t, w), t, c);
#pragma unroll
  for (int d = 4; d >= 1; --d) {
    two_sum(p[d], __fmul2_rn(t, w), t, e);
    c = __ffma2_rn(c, w, e);
  }
  two_sum(p[0], __fmul2_rn(t, w), h, l);
  l = __fadd2_rn(l, __fmul2_rn(c, w));
}

// 3D form: sum_{d=0..7} p[d] 2^(43 - 8 d) as an integer (the block's sum times
// 2^57; its magnitude, at most 32, leaves a bit).  The digit sums are integers of
// at most 2^22 and pair up in 32 bits; the last two, below the integer, round.
__device__ __forceinline__ int exact_int(float x) { return __float_as_int(x + 12582912.f) - 0x4B400000; }
__device__ __forceinline__ long long join_fixed(const float (&p)[8]) {
  const int t0 = (exact_int(p[0]) << 8) + exact_int(p[1]), t1 = (exact_int(p[2]) << 8) + exact_int(p[3]);
  const int t2 = (exact_int(p[4]) << 8) + exact_int(p[5]);
  const int t3 = exact_int(__fmaf_rn(p[6], 256.f, p[7]) * 0x1p-13f);
  return (long long)t0 * (1ll << 35) + (long long)t1 * (1ll << 19) + (long long)t2 * 8 + t3;
}
// v 2^e rounded to FP64 (a subnormal result truncated), integer operations only
__device__ __forceinline__ double fixed_to_double(long long v, int e) {
  const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)u), ef = 1086 - lz + e;
  const unsigned long long n = u << min(lz, 63), mant = (n >> 11) + ((n >> 10) & 1);
  unsigned long long r = ((unsigned long long)(unsigned)(ef - 1) << 52) + mant;
  if (ef < 1) r = n >> min(12 - ef, 63);
  if (ef > 2045) r = 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(u == 0 ? 0ull : r | ((unsigned long long)(v < 0) << 63)));
}

}  // namespace digits
}  // namespace csff
