// Block updates Y = S C on the tensor cores (S: L x p, C: p x q complex), sliced exactly into FP16 digits (sliced.cuh):
// complex128 blocks, and blocks of double-float pairs with a complex64 addend, Y = S C + Z (the mixed solve's block X).
//
// One real product per tile of 128 rows: accumulator row = row of S, K = the 2 p real and imaginary parts of a row,
// accumulator columns 2 j + c = parts of up to 32 columns of Y, once per level. Row l is held against one exponent
// E_l = max_i (e(S_li) + a_i), where a_i is the exponent of the largest entry of row i of C; row i of C is scaled by
// 2^-a_i, and its columns have exponents of their own. So a small column of S with large coefficients (a preconditioned
// residual) is held as accurately as a large one with small coefficients: every term S_li C_ij is rounded relative to
// the largest term that its row and its column of C could form. That leaves an output few digits if all its own terms are
// far smaller (a small column of S that C picks out). The solves take it, since their errors count against the norm of a
// row; for other callers (EACH) the kernel finds such outputs and forms them in plain FP64: per output a bit is set where
// some term comes within a few bits of that largest one, from the exponents that the digits need anyway.
//
// One CTA (512 threads, one per SM) keeps the digits of C in shared memory and walks over row tiles of one k-point. A
// thread owns one row and a quarter of the columns (16-byte digit stores, no bank conflicts); it holds its elements in
// registers for the row's exponent, forms the digits in stages of 16 columns (two stages side by side in the 64-wide
// operand tile: digits of one stage while the MMAs of the stage before run) and loads the next tile's elements as soon
// as a stage's are used. The epilogue adds the levels as 64-bit integers and rounds once, in integer arithmetic (the
// FP64 pipe retires about 2 operations per clock and SM).
//
// A tile's first two stages are converted before the epilogue of the tile before it, so that the MMAs run meanwhile.
// Every wait is bounded. A warp whose wait runs out, or that finds the abort flag set, does nothing more; all leave
// together at the next tile, wait for the MMAs in flight and write NaN over the CTA's rows.
//
// Complex128 takes eight digits (smooth fields, 24 to 64 columns, against extended precision: off by 4.7e-17 of the
// result's norm, FP64 sums by 2.9e-16 to 4.7e-16; seven digits left 1.1e-15). Pairs take eight digits of base 128 (2.5e-15, the double-float sums 2.0e-14;
// seven left 5.4e-14 where C is near the identity).
//
// Bound: instructions of the digit extraction and the epilogue. Complex128, 8 k-points, 48 -> 16 columns at N = 32:
// 4.00 ms on the FP64 pipe (1.21 TFLOP/s, all of it), 0.48 ms here (EACH: 0.52 ms for smooth fields and dense C; 2.1 ms
// for C near the identity, where a fifth of the outputs takes FP64); 4 k-points, 57 -> 19 at N = 64: 27.5 and 2.7 ms; one
// k-point, 24 -> 8 at N = 16: 54.8 and 17.0 us; the smallest size tried (8 -> 4 columns of 1536 rows): 21.9 and 17.9 us.
// Pairs, 4 k-points, 19 -> 19 columns at N = 64: 2.03 ms in double-float arithmetic, 1.16 ms here (without the MMAs
// 0.25 ms less, without the digits 0.3 ms, without the epilogue 0.44 ms); 2 k-points, 12 -> 12 at N = 8: 16.9 and 12.9 us.
// (For complex64 the same scheme with four digits was slower than the FP32 pipe: 1.29 against 0.97 ms for 57 -> 19
// columns at N = 64.)
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>

#include "sliced.cuh"

namespace pc {

namespace {

constexpr int SU_THREADS = 512;
constexpr int SU_COLS = 16;  // columns per stage
constexpr int SU_BAD = 1 << 20;
constexpr int SU_SLACK = 5;  // most bits between an output's largest term and its row's (launch_update_sl)

struct SlUpdateArgs {
  const void *S;
  long ss;
  const double2 *C;
  long sc;
  void *Y;
  long sy;
  const float2 *Z;
  long sz;
  long L;
  int p, q, nbc, nbp, ntile;
  int slack;
  uint32_t tmem_cols;
  const int *act;
  int *tmo;
};

// four consecutive accumulator columns of this warp's lanes, without waiting
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait4(uint32_t (&r)[4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3])::"memory");
}

// words of shared memory past the exponents of C with EACH: sM and sNear of update_sl_kernel
constexpr int su_each_words(bool each) { return each ? 1536 + 2 * 65 * (SU_SLACK + 3) : 0; }

// T: element type of S and Y; NS: stages (p <= 16 NS); EACH: every output as accurate as its own terms, not as its row's
template <typename T, int NS, bool EACH>
__global__ void __launch_bounds__(SU_THREADS, 1) update_sl_kernel(const SlUpdateArgs a) {
  using F = SlFormShort<T>;
  constexpr int ND = F::ND, NL = F::NL;
  constexpr bool F64 = std::is_same<T, double2>::value;
  constexpr int NC = 4 * NS;          // columns per thread
  constexpr int NATOM = (NS + 1) / 2;  // 64-wide operand tiles of C
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_addr(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *const sm = smem_raw + (base - raw);
  const uint32_t off_b = ND * 16384u, atom = (uint32_t)(ND * a.nbp) * 128u, off_e = off_b + NATOM * atom;
  int *const sE = reinterpret_cast<int *>(sm + off_e);  // [3][4][128] row exponents (three tiles in turn, by column quarter)
  int *const sCA = sE + 1536, *const sCB = sCA + 64;    // exponents of the rows and columns of C
  // with EACH, bit j of a word for output j: sM [3][4][128] outputs of a row that the digits serve (laid out as sE), and
  // sNear [slack + 3][65], at k and i: outputs whose coefficient in row i of C is at most k - 2 (.x) and k - 1 (.y) bits
  // below the largest that its column allows
  unsigned *const sM = reinterpret_cast<unsigned *>(sCB + 64);
  uint2 *const sNear = reinterpret_cast<uint2 *>(sM + 1536);
  const uint32_t off_bar = off_e + (uint32_t)(1536 + 128 + su_each_words(EACH)) * 4u;
  const uint32_t bars = base + off_bar;
  const uint32_t ready = bars + 16u;  // bars: the MMAs of an operand buffer are done; ready: digits are there, in turn
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(sm + off_bar + 32);
  volatile int *abort = reinterpret_cast<volatile int *>(tmem_holder + 1);
  volatile int *badC = abort + 1;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = a.act ? a.act[blockIdx.z] : (int)blockIdx.z;
  const int j0 = blockIdx.y * a.nbc, nbc = min(a.nbc, a.q - j0);
  const long L = a.L;
  const T *const Sb = static_cast<const T *>(a.S) + (long)b * a.ss;
  const double2 *const Cb = a.C + (long)b * a.sc + j0;

  {
    float4 *z = reinterpret_cast<float4 *>(sm);
    const int nz = (int)(off_e / 16u);
    for (int i = tid; i < nz; i += SU_THREADS) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (tid == 0) {
    bar_init(bars, 1);
    bar_init(bars + 8u, 1);
    bar_init(ready, SU_THREADS / 32);
    bar_init(ready + 8u, SU_THREADS / 32);
    *abort = 0;
    *badC = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_holder)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  // the thread's row and columns: 4 g + c of every stage
  const int r = tid & 127, g = tid >> 7;
  T v[NC];
  auto load = [&](int s, long tile) {
    const long l = tile * 128 + r;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = s * SU_COLS + 4 * g + c;
      v[4 * s + c] = T{};
      if (i < a.p && l < L) v[4 * s + c] = Sb[(long)i * L + l];
    }
  };
#pragma unroll
  for (int s = 0; s < NS; ++s) load(s, blockIdx.x);

  // digits of C
  for (int i = warp; i < a.p; i += SU_THREADS / 32) {
    int mx = lane < nbc ? sl_key(Cb[(long)i * a.q + lane]) : 0;
    mx = sl_exp_of<double2>(__reduce_max_sync(0xffffffffu, mx));
    if (lane == 0) {
      sCA[i] = mx;
      if (mx >= SL_NONFINITE) *badC = 1;
    }
  }
  __syncthreads();
  for (int j = warp; j < nbc; j += SU_THREADS / 32) {
    int mx = -SU_BAD;
    for (int i = lane; i < a.p; i += 32) mx = max(mx, sl_exp_of<double2>(sl_key(Cb[(long)i * a.q + j])) - sCA[i]);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) sCB[j] = mx;
  }
  __syncthreads();
  const bool bad = *badC != 0;
  if constexpr (EACH) {
    for (int i = warp; i < a.p; i += SU_THREADS / 32) {
      const int d = lane < nbc ? sCB[lane] + sCA[i] - (sl_key(Cb[(long)i * a.q + lane]) >> 20) : SU_BAD;
      unsigned m = 0u;
      for (int k = 0; k < a.slack + 3; ++k) {
        const unsigned up = k ? __ballot_sync(0xffffffffu, d <= k - 1) : 0u;
        if (lane == 0) sNear[k * 65 + i] = make_uint2(m, up);
        m = up;
      }
    }
  }
  for (int t = tid; t < a.p * nbc && !bad; t += SU_THREADS) {
    const int i = t / nbc, j = t - i * nbc;
    const double2 c = Cb[(long)i * a.q + j];
    const int E = sCB[j] + sCA[i], ii = i & 31, kc = ii >> 2;  // four columns (8 values) per 16-byte chunk
    unsigned x0[ND], x1[ND];  // digits of (cr, -ci) and (ci, cr)
    if constexpr (F64) {
      const unsigned long long cr = sl_round<ND>(sl_raw<ND>(c.x, E)), ci = sl_round<ND>(sl_raw<ND>(c.y, E)),
                               cn = sl_round<ND>(sl_raw<ND>(-c.y, E));
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        x0[d] = sl_digits<ND>(cr, cn, ND - 1 - d);
        x1[d] = sl_digits<ND>(ci, cr, ND - 1 - d);
      }
    } else {
      // scaled in FP64 (|c| 2^(5 - (E - 1023)) < 64), then as pairs
      const double f = __longlong_as_double((long long)min(max(2051 - E, 1), 2046) << 52);
      const df re = df_from(c.x * f), im = df_from(c.y * f);
      unsigned tr[ND], ti[ND], tn[ND];
      sl7_digits(re.hi, re.lo, 1.0f, tr);
      sl7_digits(im.hi, im.lo, 1.0f, ti);
      sl7_digits(-im.hi, -im.lo, 1.0f, tn);
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        x0[d] = sl7_pack(tr[d], tn[d]);
        x1[d] = sl7_pack(ti[d], tr[d]);
      }
    }
    // (x + i y)(cr + i ci): row 2 j holds (cr, -ci), row 2 j + 1 holds (ci, cr)
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const int rr = d * a.nbp + 2 * j;
      unsigned char *o = sm + off_b + (i >> 5) * atom + (ii & 3) * 4;
      *reinterpret_cast<unsigned *>(o + rr * 128 + ((kc ^ (rr & 7)) << 4)) = x0[d];
      *reinterpret_cast<unsigned *>(o + (rr + 1) * 128 + ((kc ^ ((rr + 1) & 7)) << 4)) = x1[d];
    }
  }
  fence_proxy_async();

  const int quarter = warp & 3, slot = warp >> 2;
  const uint32_t tdrain = tmem + ((uint32_t)(quarter * 32) << 16);
  T *const Yb = static_cast<T *>(a.Y) + (long)b * a.sy + (long)j0 * L;
  const float2 *const Zb = a.Z ? a.Z + (long)b * a.sz + (long)j0 * L : nullptr;
  // Z of the epilogue's outputs, loaded before the digits of the next tile are formed
  constexpr int NZ = F64 ? 1 : 8;
  float2 z[NZ];
  auto load_z = [&](long tile) {
    if constexpr (!F64) {
      const long l = tile * 128 + quarter * 32 + lane;
#pragma unroll
      for (int u = 0; u < NZ; ++u) {
        const int j = 2 * slot + 8 * (u >> 1) + (u & 1);
        z[u] = Zb && j < nbc && l < L ? Zb[(long)j * L + l] : make_float2(0.f, 0.f);
      }
    }
  };
  bool live = true;  // no wait of this warp has run out; the steps below do nothing after that
  int nready = 0, issued = -1;  // arrivals on `ready`; the last stage whose MMAs this warp issued
  auto convert = [&](int s, int n, long tile, int ex) {
    const int buf = n & 1;
    if (live && n >= 2) live = warp_wait(bars + 8u * buf, ((n >> 1) & 1) ^ 1, abort);
    if (!live) return;
    unsigned char *o = sm + r * 128 + (((buf * 4 + g) ^ (r & 7)) << 4);
    if constexpr (F64) {
      unsigned long long m[8];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = min(s * SU_COLS + 4 * g + c, a.p - 1);  // (columns past p are zero)
        sl_split<ND>(v[4 * s + c], ex - sCA[i], m[2 * c], m[2 * c + 1]);
      }
      load(s, tile + gridDim.x);
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        uint4 x;
        x.x = sl_digits<ND>(m[0], m[1], ND - 1 - d);
        x.y = sl_digits<ND>(m[2], m[3], ND - 1 - d);
        x.z = sl_digits<ND>(m[4], m[5], ND - 1 - d);
        x.w = sl_digits<ND>(m[6], m[7], ND - 1 - d);
        *reinterpret_cast<uint4 *>(o + d * 16384) = x;
      }
    } else if (s * SU_COLS + 4 * g < a.p) {
      // (with at most two stages a quarter without columns keeps the zeros of the start)
      unsigned x[4][ND];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = min(s * SU_COLS + 4 * g + c, a.p - 1);
        const float f = sl7_scale(ex - sCA[i]);
        const float4 e = v[4 * s + c];
        unsigned tr[ND], ti[ND];
        sl7_digits(e.x, e.y, f, tr);
        sl7_digits(e.z, e.w, f, ti);
#pragma unroll
        for (int d = 0; d < ND; ++d) x[c][d] = sl7_pack(tr[d], ti[d]);
      }
      load(s, tile + gridDim.x);
#pragma unroll
      for (int d = 0; d < ND; ++d)
        *reinterpret_cast<uint4 *>(o + d * 16384) = make_uint4(x[0][d], x[1][d], x[2][d], x[3][d]);
    }
    fence_proxy_async();
  };
  // the MMAs of stages s0 .. s1 - 1 (converted by all threads), the first of them the n-th
  auto issue = [&](int s0, int s1, int n) {
    if (!live) return;
    tc_fence_before();
    __syncwarp();
    const uint32_t bar = ready + 8u * (nready & 1), phase = (nready >> 1) & 1;
    if (lane == 0) bar_arrive(bar);
    ++nready;
    if (warp == 0) {
      if (!(live = warp_wait(bar, phase, abort))) return;
      issued = n + s1 - s0 - 1;
      if (elect_one()) {
        tc_fence_after();
        for (int s = s0; s < s1; ++s) {
          const int buf = (n + s - s0) & 1, nks = a.p - s * SU_COLS > SU_COLS / 2 ? 2 : 1;  // K steps of 8 columns
          for (int ks = 0; ks < nks; ++ks)
            sl_mma_step<ND, NL>(tmem, base, base + off_b + (s >> 1) * atom, (uint32_t)(buf * 64 + ks * 32),
                                (uint32_t)((s & 1) * 64 + ks * 32), a.nbp, s == 0 && ks == 0);
          mma_commit(bars + 8u * buf);
        }
      }
      __syncwarp();
    }
  };
  // This warp's columns of Y: 2 slot + 8 it, and the next
  const unsigned own = (nbc < 32 ? (1u << nbc) - 1u : ~0u) & (0x03030303u << (2 * slot));
  // Output j of the rows row0 + r in plain FP64, for the lanes r of `todo`: a row with an infinity or a NaN (or C with
  // one), or an output that the digits do not serve. Up to half of the rows are taken eight at a time, the terms of a row
  // shared over four lanes; otherwise a lane takes its own row, past the terms of zero coefficients where the row is
  // finite. (An FP64 instruction takes the warp 64 cycles whatever the number of active lanes: p + 4 of them for eight rows
  // of the first form, 4 p for the second.)
  auto plain_fp64 = [&](unsigned todo, long row0, int j, bool finite) {
    double2 out = make_double2(0.0, 0.0);
    if (__popc(todo) <= 16) {
      const int at = __popc(todo & ((1u << lane) - 1u));  // this lane's place among the rows
      unsigned rest = todo;
      for (int first = 0; rest; first += 8) {
        unsigned t = rest;
        for (int k = 0; k < 8; ++k) {
          if (k < (lane >> 2)) t &= t - 1;
          rest &= rest - 1;
        }
        double2 v = make_double2(0.0, 0.0);
        if (t) {
          const double2 *x = Cb + j;
          const T *y = Sb + row0 + __ffs(t) - 1;
#pragma unroll 4
          for (int i = lane & 3; i < a.p; i += 4) {
            const double2 u = ld_c128(y + (long)i * L), c = x[(long)i * a.q];
            v.x = fma(u.x, c.x, fma(-u.y, c.y, v.x));
            v.y = fma(u.x, c.y, fma(u.y, c.x, v.y));
          }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
          v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        }
        const int from = 4 * ((at - first) & 7);
        const double2 w = make_double2(__shfl_sync(0xffffffffu, v.x, from), __shfl_sync(0xffffffffu, v.y, from));
        if (at >= first && at < first + 8) out = w;
      }
    } else if ((todo >> lane) & 1u) {
      for (int i = 0; i < a.p; ++i) {
        const double2 c = Cb[(long)i * a.q + j];
        if (finite && c.x == 0.0 && c.y == 0.0) continue;
        const double2 u = ld_c128(Sb + (long)i * L + row0 + lane);
        out.x = fma(u.x, c.x, fma(-u.y, c.y, out.x));
        out.y = fma(u.x, c.y, fma(u.y, c.x, out.y));
      }
    }
    if ((todo >> lane) & 1u) {
      const long o = (long)j * L + row0 + lane;
      if constexpr (F64) {
        Yb[o] = out;
      } else {
        if (Zb) {
          out.x += (double)Zb[o].x;
          out.y += (double)Zb[o].y;
        }
        const cdf d = cdf_from(out);
        Yb[o] = make_float4(d.re.hi, d.re.lo, d.im.hi, d.im.lo);
      }
    }
  };
  // the tile whose n-th stage was its last
  auto epilogue = [&](long tile, int n, int par) {
    if (live) live = warp_wait(bars + 8u * (n & 1), (n >> 1) & 1, abort);
    if (!live) return;
    tc_fence_after();
    // epilogue: lane = row, four accumulator columns (two columns of Y) at a time
    const int row = quarter * 32 + lane;
    const long l = tile * 128 + row;
    int E = 0;
    unsigned served = EACH ? 0u : ~0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      E = max(E, sE[par * 512 + k * 128 + row]);
      if constexpr (EACH) served |= sM[par * 512 + k * 128 + row];
    }
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int c0 = 4 * slot + 16 * it;
      if (c0 >= 2 * nbc) break;
      __syncwarp();
      uint32_t w[NL][4];
#pragma unroll
      for (int lv = 0; lv < NL; ++lv) tmem_ld4(tdrain + (uint32_t)(lv * a.nbp + c0), w[lv]);
#pragma unroll
      for (int lv = 0; lv < NL; ++lv) tmem_wait4(w[lv]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = (c0 >> 1) + h;
        if (j >= nbc || l >= L) continue;
        T out;
        if constexpr (F64) {
          const int sc = sl_weight<F>(E, sCB[j]);
          long long H[2];
          unsigned lo[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            long long hi = 0, s = 0;
#pragma unroll
            for (int lv = 0; lv < NL; ++lv) sl_level_add<F>(hi, s, lv, __float2int_rn(__uint_as_float(w[lv][2 * h + u])));
            sl_join<F>(hi, s, H[u], lo[u]);
          }
          out = make_double2(sl_to_double(H[0], lo[0], sc), sl_to_double(H[1], lo[1], sc));
        } else {
          const int sc = sl_weight<F>(E, sCB[j]) + F::RB * (NL - 1);
          float lr[NL], li[NL];
#pragma unroll
          for (int lv = 0; lv < NL; ++lv) {
            lr[lv] = __uint_as_float(w[lv][2 * h]);
            li[lv] = __uint_as_float(w[lv][2 * h + 1]);
          }
          const float2 zz = z[2 * it + h];
          const df re = sl7_value(lr, sc, zz.x), im = sl7_value(li, sc, zz.y);
          out = make_float4(re.hi, re.lo, im.hi, im.lo);
        }
        Yb[(long)j * L + l] = out;
      }
    }
    // the outputs that the digits do not serve, over what was stored
    const unsigned plain = l >= L ? 0u : (bad || E >= SU_BAD ? ~0u : ~served);
    if (__any_sync(0xffffffffu, plain & own)) {
#pragma unroll 1
      for (unsigned js = own; js; js &= js - 1) {
        const int j = __ffs(js) - 1;
        const unsigned todo = __ballot_sync(0xffffffffu, (plain >> j) & 1u);
        if (todo) plain_fp64(todo, tile * 128 + quarter * 32, j, E < SU_BAD);
      }
    }
  };
  // A tile's first two stages are converted before the epilogue of the tile before, whose MMAs run meanwhile
  constexpr int AHEAD = NS < 2 ? NS : 2;
  int n = 0, par = 0, ppar = 0;  // stages converted; exponent buffers of this tile and the one before
  long prev = -1;
  for (long tile = blockIdx.x; tile < a.ntile; tile += gridDim.x) {
    if (prev >= 0) load_z(prev);
    // exponent of the row
    int ex = 0;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int i = (k >> 2) * SU_COLS + 4 * g + (k & 3);
      if (i < a.p) {
        const int e = sl_exp_of<T>(sl_key(v[k]));
        ex = max(ex, e >= SL_NONFINITE ? SU_BAD : e + sCA[i]);
      }
    }
    sE[par * 512 + g * 128 + r] = ex;
    if (__syncthreads_or(!live)) break;  // all warps leave together
#pragma unroll
    for (int k = 0; k < 4; ++k) ex = max(ex, sE[par * 512 + k * 128 + r]);
    if constexpr (EACH) {
      // an output is served if one of its terms is within `slack` bits of the largest that its row and column allow, or
      // two of this thread's terms within slack + 1
      unsigned served = 0, seen = 0;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const int i = (k >> 2) * SU_COLS + 4 * g + (k & 3);
        if (i < a.p) {
          const uint2 m = sNear[max(a.slack + 2 - (ex - sCA[i] - (sl_key(v[k]) >> 20)), 0) * 65 + i];
          served |= m.x | (seen & m.y);
          seen |= m.y;
        }
      }
      sM[par * 512 + g * 128 + r] = served;
    }
#pragma unroll
    for (int s = 0; s < AHEAD; ++s) convert(s, n + s, tile, ex);
    if (prev >= 0) epilogue(prev, n - 1, ppar);
    issue(0, AHEAD, n);
    n += AHEAD;
#pragma unroll
    for (int s = AHEAD; s < NS; ++s) {
      convert(s, n, tile, ex);
      issue(s, s + 1, n);
      ++n;
    }
    prev = tile;
    ppar = par;
    par = par == 2 ? 0 : par + 1;
  }
  if (!__syncthreads_or(!live) && prev >= 0) {  // (and sM of the last tile)
    load_z(prev);
    epilogue(prev, n - 1, ppar);
  }
  __syncwarp();
  if (warp == 0 && *abort && issued >= 0) warp_wait(bars + 8u * (issued & 1), (issued >> 1) & 1, abort, false);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
  }
  if (*abort) {
    // nothing of this CTA can be trusted
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    for (long tile = blockIdx.x; tile < a.ntile; tile += gridDim.x) {
      const long l = tile * 128 + r;
      for (int j = g; j < nbc && l < L; j += 4) {
        if constexpr (F64)
          Yb[(long)j * L + l] = make_double2(nan, nan);
        else
          Yb[(long)j * L + l] = make_float4((float)nan, (float)nan, (float)nan, (float)nan);
      }
    }
    if (tid == 0) report_timeout(a.tmo);
  }
}

template <typename T, int NS, bool EACH = false>
int launch_su(SlUpdateArgs a, int nb, cudaStream_t st) {
  // columns of Y per block: all levels of 2 nbc columns in TMEM, the digits of C and of one tile in shared memory
  using F = SlFormShort<T>;
  constexpr int ND = F::ND, most_cols = NS > 2 ? 20 : 32;
  constexpr int NPAD = F::NL % 2 == 0 ? 8 : 16;  // (see sl_mma_step)
  const int nqb = (a.q + most_cols - 1) / most_cols;
  a.nbc = (a.q + nqb - 1) / nqb;
  a.nbp = (2 * a.nbc + NPAD - 1) / NPAD * NPAD;
  a.ntile = (int)((a.L + 127) / 128);
  a.tmem_cols = 32;
  while (a.tmem_cols < (uint32_t)((ND + ((a.nbp >> 3) & 1)) * a.nbp)) a.tmem_cols *= 2;
  auto smem_of = [](int nbp) {
    return (size_t)1024 + ND * 16384 + (size_t)((NS + 1) / 2) * ND * nbp * 128 + (1536 + 128 + su_each_words(EACH)) * 4 + 64;
  };
  // CTAs per k-point and column block: the least tiles (plus about one for the setup) in the longest sequence per SM
  const long per = (long)nb * nqb, nsm = sm_count();
  int gx = 1;
  double best = 0.0;
  for (int k = 1; k <= a.ntile && (k == 1 || (k - 1) * per < 4 * nsm); ++k) {
    const double cost = (double)((per * k + nsm - 1) / nsm) * ((a.ntile + k - 1) / k + 1.0);
    if (k == 1 || cost < best) {
      best = cost;
      gx = k;
    }
  }
  static bool configured[64] = {};
  int dev = 0;
  PC_CK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    PC_CK(cudaFuncSetAttribute(update_sl_kernel<T, NS, EACH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)smem_of(2 * most_cols)));
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  // a CTA's 512 threads of 128 registers take the SM: no second CTA waits for its TMEM columns there
  update_sl_kernel<T, NS, EACH><<<dim3(gx, nqb, nb), SU_THREADS, smem_of(a.nbp), st>>>(a);
  PC_CK_LAUNCH();
  return PC_OK;
}

}  // namespace

int launch_update_sl(int nb, long L, int p, int q, int dtype, const void *S, long ss, const void *C, long sc, void *Y,
                     long sy, const void *Z, long sz, cudaStream_t st, int *tmo, const int *act, bool each) {
  SlUpdateArgs a{};
  a.S = S;
  a.ss = ss;
  a.C = static_cast<const double2 *>(C);
  a.sc = sc;
  a.Y = Y;
  a.sy = sy;
  a.Z = static_cast<const float2 *>(Z);
  a.sz = sz;
  a.L = L;
  a.p = p;
  a.q = q;
  a.act = act;
  a.tmo = tmo;
  if (dtype == PC_DFS) return p <= SU_COLS ? launch_su<float4, 1>(a, nb, st) : launch_su<float4, 2>(a, nb, st);
  // EACH: the error of a digit product is 2^-60.2 sqrt(2 p) (rms) of the largest term that a row of S and a column of C
  // could form. An output with a term within 2^slack of that is off by 2^-54 of its own terms, no more than FP64 sums. The
  // others take FP64; where S and C are dense they are few (48 -> 16 columns: none of 10^5 outputs of random panels, 2 in
  // 10^4 of smooth fields).
  a.slack = std::min(SU_SLACK, (int)std::floor(6.2 - 0.5 * std::log2(2.0 * p)));
  switch ((p + SU_COLS - 1) / SU_COLS) {
    case 1: return each ? launch_su<double2, 1, true>(a, nb, st) : launch_su<double2, 1>(a, nb, st);
    case 2: return each ? launch_su<double2, 2, true>(a, nb, st) : launch_su<double2, 2>(a, nb, st);
    case 3: return each ? launch_su<double2, 3, true>(a, nb, st) : launch_su<double2, 3>(a, nb, st);
    default: return each ? launch_su<double2, 4, true>(a, nb, st) : launch_su<double2, 4>(a, nb, st);
  }
}

}  // namespace pc
