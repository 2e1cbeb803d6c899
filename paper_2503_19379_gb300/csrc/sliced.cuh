// Exact slicing of FP64-accurate values into FP16 integers for the tensor cores (the error-free splitting of
// Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 2012; on tensor cores: Mukunoki, Ozaki, Ogita and Imamura,
// ISC 2020).
//
// A value v is held against a common exponent E (biased as in FP64, at least that of every value it is summed with)
// as the integer m = round(v 2^(MB - 1 - (E - 1023))), |m| < 2^MB with MB = 8 (ND - 1) + 6, and m is written in ND
// balanced base-256 digits, m = sum_j d_j 256^(ND-1-j), |d_j| <= 128 (|d_0| <= 64). Digits are exact in FP16, a
// product of two is an integer of at most 2^14, and the products d_i d'_j of one level k = i + j (at most 8 pairs)
// over a sum of 128 terms stay within 2^24: the tensor core's FP32 accumulator holds them exactly, in any order. The
// level sums L_0 .. L_(NL-1) give sum m m' = 256^(2 ND - 1 - NL) sum_k L_k 256^(NL-1-k). A product is off by the
// dropped levels k >= NL (random digits have rms 74; a pair at level 8 is 2^-60 of the largest product) and by the
// rounding of its factors, 2^-(8 ND - 1.2) of the largest (rms); the additions do not round at all.
#pragma once
#include <cuda_fp16.h>

#include "dfloat.cuh"
#include "pc_internal.cuh"
#include "tc_ptx.cuh"

namespace pc {

template <int ND> constexpr int sl_bits() { return 8 * (ND - 1) + 6; }
constexpr int SL_NONFINITE = 0x7ff;
constexpr int SL_EMIN = 128;  // common exponents start here: FP64 values too small to reach their last digit become 0

// A key whose maximum over elements gives their common exponent (sl_exp_of): the larger part's magnitude, high bits
__device__ __forceinline__ int sl_key(double2 v) {
  return max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff);
}
__device__ __forceinline__ int sl_key(float4 v) {  // a pair's low part is normally far below its high part
  return max(max(__float_as_int(v.x) & 0x7fffffff, __float_as_int(v.z) & 0x7fffffff),
             max(__float_as_int(v.y) & 0x7fffffff, __float_as_int(v.w) & 0x7fffffff));
}
// biased FP64 exponent of a key (0x7ff for an infinity or a NaN)
template <typename T> __device__ __forceinline__ int sl_exp_of(int key) {
  if constexpr (std::is_same<T, double2>::value) return max(key >> 20, SL_EMIN);
  const int e = key >> 23;
  return e == 0xff ? SL_NONFINITE : max(e, 6) + 896;  // (not below 902: sl_scale stays an FP32 number)
}

__device__ __forceinline__ unsigned sl_shr(unsigned x, int s) {  // 0 for s >= 32
  unsigned r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
}
// (mh : ml) >> sh for sh >= 0 with the sign s (0 or -1) applied
__device__ __forceinline__ long long sl_shift(unsigned mh, unsigned ml, int sh, int s) {
  const unsigned lo = sl_shr(__funnelshift_rc(ml, mh, sh), max(sh - 32, 0)), hi = sl_shr(mh, sh);
  return (long long)(((unsigned long long)(hi ^ (unsigned)s) << 32) | (lo ^ (unsigned)s)) - s;
}
// 2 m, not yet rounded: v 2^(MB - (E - 1023)); E at least the exponent of v and SL_EMIN
template <int ND> __device__ __forceinline__ long long sl_raw(double x, int E) {
  constexpr int PS = sl_bits<ND>() - 52;  // the 53-bit significand's place in 2 m
  static_assert(PS > 0 && PS <= 10, "FP64 values take seven or eight digits");
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned mh = (__funnelshift_l(lo, hi, PS) & ((1u << (20 + PS)) - 1u)) | (1u << (20 + PS));
  // zeros and subnormals (e = 0) are shifted out, as E >= SL_EMIN
  return sl_shift(mh, lo << PS, E - (int)((hi >> 20) & 0x7ff), (int)hi >> 31);
}
// m with every digit moved up by 128, so that digit j is byte ND - 1 - j minus 128; with seven digits byte 7 holds 0x64
// (see sl_digits)
template <int ND> __device__ __forceinline__ unsigned long long sl_round(long long raw) {
  unsigned long long b = ND < 8 ? 0x64ull << 56 : 0ull;
#pragma unroll
  for (int k = 0; k < ND; ++k) b |= 0x80ull << (8 * k);
  if constexpr (ND < 8) return ((unsigned long long)raw + (2 * b + 1)) >> 1;
  return (unsigned long long)((raw + 1) >> 1) + b;
}
// rounded and biased m of the real and imaginary part of an element
template <int ND>
__device__ __forceinline__ void sl_split(double2 v, int E, unsigned long long &re, unsigned long long &im) {
  re = sl_round<ND>(sl_raw<ND>(v.x, E));
  im = sl_round<ND>(sl_raw<ND>(v.y, E));
}
// byte k of two biased values as FP16 digits (u0 low, u1 high): 0x6400 | byte is 1024 + byte
template <int ND> __device__ __forceinline__ unsigned sl_digits(unsigned long long u0, unsigned long long u1, int k) {
  unsigned x;
  if (ND == 8 || k < 4) {
    const int kk = k & 3;
    x = (__byte_perm(k < 4 ? (unsigned)u0 : (unsigned)(u0 >> 32), k < 4 ? (unsigned)u1 : (unsigned)(u1 >> 32),
                     kk | (kk << 4) | ((4 + kk) << 8) | ((4 + kk) << 12)) & 0x00ff00ffu) | 0x64006400u;
  } else  // the 0x64 of byte 7 comes along
    x = __byte_perm((unsigned)(u0 >> 32), (unsigned)(u1 >> 32), (k - 4) | (3 << 4) | (k << 8) | (7 << 12));
  const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&x), __half2half2(__ushort_as_half(0x6480)));
  return *reinterpret_cast<const unsigned *>(&h);
}

// Double-float pairs take digits in base 128 (seven: 48 bits, their precision), formed on the FP32 pipe: adding
// M_k = (1.5 2^23 + 0x6480) 2^-7k to the rest y rounds it to a multiple of 2^-7k and leaves the digit, |d_k| <= 64, plus
// 0x6480 in the low 16 bits of the sum: the FP16 number 1024 + 128 + d_k. (The integer route of the FP64 values costs
// twice the instructions for a pair, on the pipe of half the rate. Base 128, because a rest of exactly 1/2 would
// overflow a digit of base 256 here.)
// y = v f has |y| < 64 for |v| < 2^(E - 1022)
__device__ __forceinline__ float sl7_scale(int E) { return __int_as_float(max(1155 - E, 0) << 23); }
template <int ND> __device__ __forceinline__ void sl7_digits(float hi, float lo, float f, unsigned (&t)[ND]) {
  static_assert(ND <= 8, "at most eight digits");
  constexpr float M = 12582912.0f + 25728.0f;
  constexpr float Mk[8] = {M,           M * 0x1p-7f,  M * 0x1p-14f, M * 0x1p-21f,
                           M * 0x1p-28f, M * 0x1p-35f, M * 0x1p-42f, M * 0x1p-49f};
  float y = hi * f;
  // lo in two parts, each added where the sum with the rest of hi is exact
  const float l = lo * f, l1 = (l + Mk[4]) - Mk[4], l2 = l - l1;
#pragma unroll
  for (int k = 0; k < ND; ++k) {
    if (k == 3) y += l1;
    if (k == 5) y += l2;
    const float s = y + Mk[k];
    t[k] = (unsigned)__float_as_int(s);
    y -= s - Mk[k];
  }
}
// the FP16 digits of two values (a low, b high)
__device__ __forceinline__ unsigned sl7_pack(unsigned a, unsigned b) {
  const unsigned x = __byte_perm(a, b, 0x5410);
  const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&x), __half2half2(__ushort_as_half(0x6480)));
  return *reinterpret_cast<const unsigned *>(&h);
}

// Per element type: bits per digit, digits, levels of digit products, rows of K whose level sums FP32 holds exactly
template <typename T> struct SlForm;
template <> struct SlForm<double2> {  // sums over many rows
  static constexpr int RB = 8, ND = 7, NL = 8, KMAX = 128;
};
template <> struct SlForm<float4> {
  // (digits 3 and 5 take the low part's share: up to 72 and 128)
  static constexpr int RB = 7, ND = 7, NL = 7, KMAX = 256;
};
template <typename T> struct SlFormShort;  // sums over the columns of a block
template <> struct SlFormShort<double2> {
  static constexpr int RB = 8, ND = 8, NL = 8, KMAX = 128;
};
template <> struct SlFormShort<float4> {
  static constexpr int RB = 7, ND = 8, NL = 8, KMAX = 256;
};
// sum_k L_k 2^(RB (NL-1-k)) times this power of two is the sum of products of values held at exponents Ea and Eb
template <typename F> __device__ __forceinline__ int sl_weight(int Ea, int Eb) {
  return Ea + Eb - 2056 - F::RB * (F::NL - 1);
}
// The weighted level sum from the sum hi of the levels before the last four and the sum lo of the last four (each in
// units of its last level), as H 2^32 + low word
template <typename F> __device__ __forceinline__ void sl_join(long long hi, long long lo, long long &H, unsigned &Lw) {
  constexpr int S = 32 - 4 * F::RB;
  lo += (hi & ((1ll << S) - 1)) << (4 * F::RB);
  H = (hi >> S) + (lo >> 32);
  Lw = (unsigned)lo;
}
template <typename F> __device__ __forceinline__ void sl_level_add(long long &hi, long long &lo, int lv, int x) {
  if (lv < F::NL - 4)
    hi += (long long)x * (1 << (F::RB * (F::NL - 5 - lv)));
  else
    lo += (long long)x * (1 << (F::RB * (F::NL - 1 - lv)));
}

// (H 2^32 + Lw) 2^n rounded to FP64; integer arithmetic only (the FP64 pipe retires about 2 operations per clock and SM)
__device__ __forceinline__ double sl_to_double(long long H, unsigned Lw, int n) {
  const bool neg = H < 0;
  if (neg) {
    Lw = 0u - Lw;
    H = ~H + (Lw == 0u ? 1 : 0);
  }
  unsigned long long top;
  int ex;  // exponent of the top bit
  const int z = __clzll(H);
  if (z < 32) {
    top = ((unsigned long long)H << z) | (((unsigned long long)Lw << z) >> 32);
    ex = 95 - z;
  } else {
    top = ((unsigned long long)H << 32) | Lw;
    if (top == 0ull) return 0.0;
    const int z2 = __clzll((long long)top);
    top <<= z2;
    ex = 63 - z2;
  }
  const unsigned long long r = top + 1024ull;
  if (r < top) {
    top = 1ull << 63;
    ++ex;
  } else {
    top = r;
  }
  const int be = ex + n + 1023;
  if (be >= 1 && be <= 2046)
    return __longlong_as_double((long long)((top >> 11) & 0xfffffffffffffull) | ((long long)be << 52) |
                                (neg ? (long long)0x8000000000000000ull : 0ll));
  const double v = scalbn((double)(top >> 11), ex + n - 52);
  return neg ? -v : v;
}
// the pair sum_k L_k 2^-7k 2^n from level sums (integers of FP32), plus an FP32 addend
__device__ __forceinline__ df sl7_value(const float (&L)[8], int n, float z) {
  df s = two_sum(L[0], L[1] * 0x1p-7f);
  float e = s.lo;
  s = two_sum(s.hi, L[2] * 0x1p-14f);
  e += s.lo;
  s = two_sum(s.hi, L[3] * 0x1p-21f);
  e += s.lo;
  e += fmaf(fmaf(fmaf(L[7], 0x1p-7f, L[6]), 0x1p-7f, L[5]), 0x1p-7f, L[4]) * 0x1p-28f;
  if (n >= -60 && n <= 100) {  // both parts stay normal
    const float f = __int_as_float((n + 127) << 23);
    s.hi *= f;
    e *= f;
  } else {
    s.hi = ldexpf(s.hi, n);
    e = ldexpf(e, n);
  }
  return df_addf(quick_two_sum(s.hi, e), z);
}

// D (+)= A B^T, FP16 operands, FP32 accumulator
__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// instruction descriptor: D FP32 (bits 4-5 = 1), A and B FP16 (0), both K-major, N >> 3 at bits 17-22, M >> 4 at 24-28
__device__ __forceinline__ uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The MMAs of one K step (16 values) for all digit pairs of levels below NL. A: ND slices of 128 rows of 128 bytes;
// B: NL slices of nbp rows each, one after the other, so that one instruction multiplies slice i of A with several
// slices of B: slice j lands in the accumulator columns of level i + j (level k at column k nbp). The slices of B past ND
// are zero: the first instructions of a sum (i = 0) start the accumulators of all NL levels. An instruction's N is a
// multiple of 16; where nbp is 8 mod 16 (allowed for ND = NL even), odd counts take one slice more, into an unused
// level NL.
template <int ND, int NL>
__device__ __forceinline__ void sl_mma_step(uint32_t tmem, uint32_t a, uint32_t b, uint32_t ko_a, uint32_t ko_b, int nbp,
                                            bool first) {
  const int odd = (nbp >> 3) & 1;
  const int most = (256 / nbp) & ~odd;  // slices per instruction (N <= 256)
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    const uint64_t ad = sdesc(a + (uint32_t)i * 16384u + ko_a);
    const int count = NL - i;
    for (int j = 0; j < count; j += most) {
      int cnt = min(count - j, most);
      cnt += cnt & odd;
      mma_f16(tmem + (uint32_t)((i + j) * nbp), ad, sdesc(b + (uint32_t)(j * nbp) * 128u + ko_b), idesc_f16(128, cnt * nbp),
              (first && i == 0) ? 0u : 1u);
    }
  }
}

__device__ __forceinline__ void named_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// Gram products of FP64-accurate panels (gram_sl.cu), dtype PC_C128 or PC_DFS, one array part[bi][chunk][p][q] per
// product: SL_GENERAL A^H B; SL_PAIR A^H A, then A^H B, both upper triangles (q = p); SL_SELF the upper triangle of
// A^H A; each (PC_C128): every entry to the accuracy of its own terms, otherwise to that of the columns' norms
constexpr int SL_GENERAL = 0, SL_PAIR = 1, SL_SELF = 2;
int sl_gram_chunks(int nb, long L);
int launch_gram_sl(int nb, long L, int p, int q, int dtype, const void *A, long sa, const void *B, long sb, int mode,
                   double2 *part, int maxchunk, int *nchunk, cudaStream_t st, int *tmo, const int *act, bool each = false);

// Y = S C (+ Z, a complex64 addend, for pairs) for PC_C128 (1 <= p <= 64) or PC_DFS (1 <= p <= 32) blocks (update_sl.cu);
// each (PC_C128): every output to the accuracy of its own terms, otherwise to that of its row's largest
int launch_update_sl(int nb, long L, int p, int q, int dtype, const void *S, long ss, const void *C, long sc, void *Y,
                     long sy, const void *Z, long sz, cudaStream_t st, int *tmo, const int *act, bool each = false);

}  // namespace pc
