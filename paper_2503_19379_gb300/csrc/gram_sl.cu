// Gram products of FP64-accurate panels on the tensor cores: complex128 panels (the FP64 solve) and double-float pairs
// (the mixed solve's block X), sliced exactly into FP16 digits (sliced.cuh).
//
// D = A^H B over the L rows, as one real product of the columns' real and imaginary parts: accumulator row 2 i + c is
// part c of column i of A (M = 128, at most 64 columns), accumulator columns 2 j + c' the parts of a block of up to 32
// columns of B, once per level. Re = D[re,re] + D[im,im] and Im = D[re,im] - D[im,re] are added as integers.
//
// One CTA (17 warps, one CTA per SM) takes a chunk of rows and a block of columns. It works through the chunk in spans
// of SG_SUPER rows, which share one exponent per column (found by a scan of the span; the second read comes from the
// L2 cache), in stages of 32 rows: 16 warps turn the stage's elements into digits in the K-major tiles of the tensor
// core (128-byte swizzle; two stages side by side in the 64-wide tile, so that the digits of one stage are formed while
// the MMAs of the stage before run), the 17th issues the MMAs, and after every group of rows that FP32 holds
// exactly (SlForm::KMAX) the level sums are drained into 64-bit integer sums in registers. At the end of a span these are
// scaled and added to FP64 sums in shared memory.
//
// Digits are exact relative to the largest values of the two columns in the span, which need not meet: columns that are
// large in different rows have a product far below that of their largest values. The solves take that, since an entry's
// error counts against the norms of its columns there. For other callers (EACH) the rows of a span in which a column is
// within two bits of its largest are marked while the digits are formed, and an entry whose columns share too few of them
// is formed in plain FP64 for this span, as are, for all, those of a column with an infinity or a NaN (`unserved`).
//
// Every wait is bounded. A warp whose wait runs out, or that finds the abort flag set, leaves its stages; at the end of
// the span all roles leave together, the MMAs in flight are waited for, and the host is told (TimeoutWord).
//
// Complex128 panels take seven digits in eight levels, which leaves less error than the FP64 sums they replace on smooth
// and random panels (N = 8 to 32, against extended precision; 24 and 48 smooth columns: 1.2e-17 to 2.0e-17 of sum |a||b|,
// rms, FP64 sums 3e-17 to 1e-16; seven levels left up to 1.8 times more off the diagonal). Pairs take seven digits of base 128: 1e-15 of the diagonal, the double-float sums 3e-14.
//
// Bound: the latency of a stage (load, digits, hand-off to the tensor core, drain), then integer instructions of the digit
// extraction. 8 k-points x 48 complex128 columns at N = 32: 23.6 ms on the FP64 pipe, 2.06 ms here (without the scan
// 0.3 ms less, without the MMAs 0.4 ms, without the drains 0.2 ms, without the marks and their comparison 0.1 ms; with
// marks in the solves too, whose converged columns are far from dense, the FP64 solve at N = 64 took 16% longer); one k-point of 24 columns at N = 16: 1.77 ms and
// 64 us. X^H X of 4 k-points x 19 pair columns at N = 64: 1.61 ms in double-float arithmetic, 1.11 ms here; of one
// k-point x 13 at N = 16: 60 and 24 us. The pair A^H A, A^H B takes the block's columns of A and of B in one CTA, and the
// columns of A that the block shares with the left operand are extracted once and stored twice.

#include <cuda.h>
#include <cuda_runtime.h>

#include "sliced.cuh"

namespace pc {

namespace {

constexpr int SG_CONV = 512;                  // threads that form digits and drain
constexpr int SG_THREADS = SG_CONV + 32;      // and the warp that issues the MMAs
constexpr int SG_ROWS = 32;                   // rows per stage
constexpr int SG_SUPER = 1024;                // rows per common exponent, at most
constexpr int SG_WORDS = SG_SUPER / 32;       // words of a column's mask of large rows
constexpr int SG_WSTRIDE = SG_WORDS + 4;      // their distance from column to column (banks of 16-byte loads)
// a column's share of the common rows that an entry needs: ordinary, all zeros, with an infinity or a NaN
constexpr int SG_NEED = 8, SG_ZERO = -1000, SG_BAD = 1 << 20;

struct SlGramArgs {
  const void *A, *B;
  long sa, sb;
  long L;
  int p, q, mode;
  int nbc, nbp;  // columns per block; accumulator columns per level (2 per operand column, rounded up to 16)
  double2 *part0, *part1;
  const int *act;
  int *tmo;
};

// exponents, needs and masks of 96 columns
constexpr uint32_t sg_col_bytes(bool each) { return 96u * 4u * (each ? 2 + SG_WSTRIDE : 2); }

// TASKS: at most 32 TASKS columns to extract (each thread two rows of every 32nd column); DEPTH: stages loaded ahead; EACH:
// every entry to the accuracy of its own terms
template <typename T, int TASKS, int DEPTH, bool EACH>
__global__ void __launch_bounds__(SG_THREADS, 1) gram_sl_kernel(const SlGramArgs a) {
  using F = SlForm<T>;
  constexpr int ND = F::ND, NL = F::NL, GROUP = F::KMAX / SG_ROWS;  // stages per drain
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_addr(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *const sm = smem_raw + (base - raw);
  const uint32_t off_b = ND * 16384u, off_acc = off_b + (uint32_t)(NL * a.nbp) * 128u;
  const uint32_t off_e = off_acc + 8u * SG_CONV * 8u;  // FP64 sums, then exponents
  double *const acc = reinterpret_cast<double *>(sm + off_acc);
  int *const sE = reinterpret_cast<int *>(sm + off_e);
  int *const sNeed = sE + 96;                                        // SG_NEED, SG_ZERO or SG_BAD
  unsigned *const sMask = reinterpret_cast<unsigned *>(sNeed + 96);  // complex128: rows within 2 bits of the column's largest
  const uint32_t off_bar = off_e + sg_col_bytes(EACH);
  const uint32_t bars = base + off_bar;
  const uint32_t ready = bars + 16u;  // by operand buffer: bars, its MMAs are done; ready, its digits are there
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(sm + off_bar + 32);
  volatile int *abort = reinterpret_cast<volatile int *>(tmem_holder + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bi = blockIdx.z, b = a.act ? a.act[bi] : bi;
  const int j0 = blockIdx.y * a.nbc, nbc = min(a.nbc, a.q - j0);
  const int pa = a.mode == SL_GENERAL ? a.p : min(a.p, j0 + nbc);  // left columns (upper triangle: i <= j)
  // the right operand: [columns j0 .. of A (dup), columns j0 .. of B]; the first are extracted with the left operand
  const int ndup = a.mode == SL_GENERAL ? 0 : nbc, nown = a.mode == SL_SELF ? 0 : nbc;
  const int ncols = pa + nown;  // columns to extract
  const T *const Ab = static_cast<const T *>(a.A) + (long)b * a.sa;
  const T *const Bb = static_cast<const T *>(a.B) + (long)b * a.sb + (long)j0 * a.L;
  // the chunk's stages, in spans of nearly equal length (a short one would have few rows of normal size)
  const long L = a.L, nst = (L + SG_ROWS - 1) / SG_ROWS;
  const long st0 = blockIdx.x * nst / gridDim.x, cst = (blockIdx.x + 1) * nst / gridDim.x - st0;
  const int nspan = (int)((cst * SG_ROWS + SG_SUPER - 1) / SG_SUPER);

  {
    float4 *z = reinterpret_cast<float4 *>(sm);
    const int nz = (int)(off_e / 16u);
    for (int i = tid; i < nz; i += SG_THREADS) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    fence_proxy_async();
  }
  if (tid == 0) {
    bar_init(bars, 1);
    bar_init(bars + 8u, 1);
    bar_init(ready, SG_CONV / 32);
    bar_init(ready + 8u, SG_CONV / 32);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_holder)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  const bool issuer = warp == SG_CONV / 32;

  // digit tasks: rows 2 rp, 2 rp + 1 of the stage; the two columns of a warp are two apart, so that their digits fall
  // into different halves of the swizzled 128-byte rows (no bank conflict)
  const int rp = lane & 15, c0 = (warp >> 1) * 4 + (warp & 1) + 2 * (lane >> 4);
  // accumulator part of this warp: TMEM lane quarter, 16 columns of each level
  const int quarter = warp & 3, slot = warp >> 2;
  const int row = quarter * 32 + lane, ci = row >> 1;
  const bool odd = row & 1, drains = !issuer && slot * 16 < a.nbp;
  const uint32_t tdrain = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(slot * 16);
  // extracted column (index into sE) of operand column jj
  auto col_of = [&](int jj) { return jj < ndup ? j0 + jj : pa + jj - ndup; };
  // Whether a span's digits serve the product of two of its columns. They are exact to half a unit of 2^-53 of the largest
  // value of each, 2^(Ea + 1) and 2^(Eb + 1), so the product is off by at most 2 n 2^-52 2^(Ea + Eb) over n rows: twice
  // the bound of FP64 sums, if sum |a||b| is at least 2^(Ea + Eb). It is if a and b are within two bits of their largest in
  // 16 common rows. (Dense columns of random values: about a third of the rows.) Returns the entries k of this thread
  // (columns slot * 8 + k) that they do not serve.
  auto unserved = [&](int words) {
    // the threads of an entry's two parts take four columns each
    const int k0 = 4 * (lane & 1);
    int left[4], cb[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int jj = slot * 8 + k0 + h;
      const bool stored = jj < ndup + nown && ci < pa && (a.mode == SL_GENERAL || ci <= j0 + (jj < ndup ? jj : jj - ndup));
      cb[h] = stored ? col_of(jj) : 0;
      left[h] = stored ? sNeed[ci] + sNeed[cb[h]] : 0;
      if (left[h] < SG_BAD + SG_ZERO && (!EACH || cb[h] == ci)) left[h] = 0;  // (a column with itself; pairs: only SG_BAD)
    }
    if constexpr (EACH) {
      for (int w = 0; w < words; w += 4) {
        const uint4 ma = *reinterpret_cast<const uint4 *>(sMask + ci * SG_WSTRIDE + w);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const uint4 mb = *reinterpret_cast<const uint4 *>(sMask + cb[h] * SG_WSTRIDE + w);
          left[h] -= __popc(ma.x & mb.x) + __popc(ma.y & mb.y) + __popc(ma.z & mb.z) + __popc(ma.w & mb.w);
        }
        if (max(max(left[0], left[1]), max(left[2], left[3])) <= 0) break;
      }
    }
    unsigned plain = 0;
#pragma unroll
    for (int h = 0; h < 4; ++h) plain |= left[h] > 0 ? 1u << (k0 + h) : 0u;
    return plain | __shfl_xor_sync(0xffffffffu, plain, 1);
  };

  int n = 0;  // stages issued
  bool live = true;  // no wait of this warp has run out
  for (int sp = 0; sp < nspan; ++sp) {
    const long span0 = (st0 + sp * cst / nspan) * SG_ROWS, span1 = min(L, (st0 + (sp + 1) * cst / nspan) * SG_ROWS);
    for (int c = warp; c < ncols; c += SG_THREADS / 32) {
      const T *x = c < pa ? Ab + (long)c * L : Bb + (long)(c - pa) * L;
      int mx = 0;
      for (long l0 = span0; l0 < span1; l0 += 512) {  // 16 loads in flight (past the end: the last row again)
#pragma unroll
        for (int w = 0; w < 16; ++w) mx = max(mx, sl_key(x[min(l0 + 32 * w + lane, span1 - 1)]));
      }
      mx = __reduce_max_sync(0xffffffffu, mx);
      if constexpr (EACH) sMask[c * SG_WSTRIDE + lane] = 0u;
      const int E = sl_exp_of<T>(mx);
      if (lane == 0) {
        sE[c] = E;
        sNeed[c] = E >= SL_NONFINITE ? SG_BAD : (mx == 0 ? SG_ZERO : SG_NEED);
      }
    }
    __syncthreads();
    const int ns = (int)((span1 - span0 + SG_ROWS - 1) / SG_ROWS);
    if (issuer) {
      for (int s = 0; s < ns; ++s, ++n) {
        const int buf = n & 1;
        if (!warp_wait(ready + 8u * buf, (n >> 1) & 1, abort)) {
          live = false;
          break;
        }
        if (elect_one()) {
          tc_fence_after();
#pragma unroll
          for (int ks = 0; ks < SG_ROWS / 16; ++ks) {
            const uint32_t ko = (uint32_t)(buf * 64 + ks * 32);
            sl_mma_step<ND, NL>(tmem, base, base + off_b, ko, ko, a.nbp, (s & (GROUP - 1)) == 0 && ks == 0);
          }
          mma_commit(bars + 8u * buf);
        }
        __syncwarp();
      }
    } else {
      long long shi[8], slo[8];  // the levels before the last four, and the last four
#pragma unroll
      for (int k = 0; k < 8; ++k) shi[k] = slo[k] = 0;
      T ring[DEPTH][TASKS][2];
      auto load = [&](T(&v)[2], int k, int s) {
        const int c = c0 + 32 * k;
        const long l = span0 + (long)s * SG_ROWS + 2 * rp;
        v[0] = v[1] = T{};
        if (c < ncols) {
          const T *x = (c < pa ? Ab + (long)c * L : Bb + (long)(c - pa) * L) + l;
          if (l < span1) v[0] = x[0];
          if (l + 1 < span1) v[1] = x[1];
        }
      };
#pragma unroll
      for (int d = 0; d < DEPTH; ++d)
#pragma unroll
        for (int k = 0; k < TASKS; ++k) load(ring[d][k], k, d);
      for (int s0 = 0; s0 < ns && live; s0 += DEPTH)
#pragma unroll
      for (int dd = 0; dd < DEPTH; ++dd) {
        const int s = s0 + dd;
        if (s >= ns) break;
        const int buf = n & 1;
        if (n >= 2 && !warp_wait(bars + 8u * buf, ((n >> 1) & 1) ^ 1, abort)) {
          live = false;
          break;
        }
#pragma unroll
        for (int k = 0; k < TASKS; ++k) {
          const int c = c0 + 32 * k, E = c < ncols ? sE[c] : SL_NONFINITE;
          if constexpr (EACH) {
            // the rows within two bits of the column's largest: even rows in the low half of the stage's word
            const unsigned m0 = __ballot_sync(0xffffffffu, sl_key(ring[dd][k][0]) >= (E - 2) << 20);
            const unsigned m1 = __ballot_sync(0xffffffffu, sl_key(ring[dd][k][1]) >= (E - 2) << 20);
            if (rp == 0 && c < ncols) sMask[c * SG_WSTRIDE + s] = __byte_perm(m0, m1, lane ? 0x7632 : 0x5410);
          }
          if (c < ncols) {
            unsigned x[2][ND];  // the digits of rows 2 rp and 2 rp + 1, real and imaginary parts
            if constexpr (std::is_same<T, double2>::value) {
              unsigned long long m[2][2];
              sl_split<ND>(ring[dd][k][0], E, m[0][0], m[1][0]);
              sl_split<ND>(ring[dd][k][1], E, m[0][1], m[1][1]);
#pragma unroll
              for (int d = 0; d < ND; ++d) {
                x[0][d] = sl_digits<ND>(m[0][0], m[0][1], ND - 1 - d);
                x[1][d] = sl_digits<ND>(m[1][0], m[1][1], ND - 1 - d);
              }
            } else {
              const float f = sl7_scale(E);
              unsigned t0[ND], t1[ND];
              sl7_digits(ring[dd][k][0].x, ring[dd][k][0].y, f, t0);
              sl7_digits(ring[dd][k][1].x, ring[dd][k][1].y, f, t1);
#pragma unroll
              for (int d = 0; d < ND; ++d) x[0][d] = sl7_pack(t0[d], t1[d]);
              sl7_digits(ring[dd][k][0].z, ring[dd][k][0].w, f, t0);
              sl7_digits(ring[dd][k][1].z, ring[dd][k][1].w, f, t1);
#pragma unroll
              for (int d = 0; d < ND; ++d) x[1][d] = sl7_pack(t0[d], t1[d]);
            }
            load(ring[dd][k], k, s + DEPTH);  // in flight while the digits of the other columns are stored
            const bool left = c < pa, dup = left && c >= j0 && ndup > 0;
            const int jr = left ? c - j0 : ndup + c - pa;  // right operand column
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int ra = 2 * c + h, rb = 2 * jr + h;
              unsigned char *oa = sm + ra * 128 + (((buf * 4 + (rp >> 2)) ^ (ra & 7)) << 4) + (rp & 3) * 4;
              unsigned char *ob = sm + off_b + rb * 128 + (((buf * 4 + (rp >> 2)) ^ (rb & 7)) << 4) + (rp & 3) * 4;
#pragma unroll
              for (int d = 0; d < ND; ++d) {
                if (left) *reinterpret_cast<unsigned *>(oa + d * 16384) = x[h][d];
                if (!left || dup) *reinterpret_cast<unsigned *>(ob + d * (a.nbp * 128)) = x[h][d];
              }
            }
          }
        }
        fence_proxy_async();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(ready + 8u * buf);
        ++n;
        if ((s & (GROUP - 1)) == GROUP - 1 || s == ns - 1) {
          if (!warp_wait(bars + 8u * buf, ((n - 1) >> 1) & 1, abort)) {
            live = false;
            break;
          }
          tc_fence_after();
          if (drains) {
#pragma unroll
            for (int lv = 0; lv < NL; ++lv) {
              uint32_t r[16];
              tmem_ld16(tdrain + (uint32_t)(lv * a.nbp), r);
              // the re and im parts of a left column sit in adjacent lanes: even lanes form Re, odd lanes Im
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const int own = __float2int_rn(__uint_as_float(r[2 * k]));
                const int o = __shfl_xor_sync(0xffffffffu, __float2int_rn(__uint_as_float(r[2 * k + 1])), 1);
                const int d = odd ? o - own : own + o;
                sl_level_add<F>(shi[k], slo[k], lv, d);
              }
            }
          }
        }
      }
      // the span's sums, but for the entries that the digits do not serve
      unsigned plain = 0;
      if constexpr (EACH) named_sync(1, SG_CONV);  // (the masks)
      if (drains) plain = unserved(ns);
      if (drains && ci < pa) {
        const int EA = sE[ci];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int jj = slot * 8 + k;
          if (jj < ndup + nown && !((plain >> k) & 1u)) {
            long long H;
            unsigned Lw;
            sl_join<F>(shi[k], slo[k], H, Lw);
            acc[k * SG_CONV + tid] += sl_to_double(H, Lw, sl_weight<F>(EA, sE[col_of(jj)]));
          }
        }
      }
      // those in plain FP64, one after the other by the whole warp
      if (__any_sync(0xffffffffu, plain != 0)) {
#pragma unroll 1
        for (int k = 0; k < 8; ++k) {
          unsigned todo = __ballot_sync(0xffffffffu, (plain >> k) & 1u) & 0x55555555u;
          for (; todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1, jj = slot * 8 + k;
            const T *x = Ab + (long)(quarter * 16 + (src >> 1)) * L;
            const T *y = jj < ndup ? Ab + (long)(j0 + jj) * L : Bb + (long)(jj - ndup) * L;
            double re = 0.0, im = 0.0;
#pragma unroll 4
            for (long l = span0 + lane; l < span1; l += 32) {
              const double2 u = ld_c128(x + l), v = ld_c128(y + l);
              re = fma(u.x, v.x, fma(u.y, v.y, re));
              im = fma(u.x, v.y, fma(-u.y, v.x, im));
            }
            // the lower half-warp sums re and the upper half im, one FP64 instruction a level
            const bool up = lane & 16;
            double t = (up ? im : re) + __shfl_xor_sync(0xffffffffu, up ? re : im, 16);
#pragma unroll
            for (int o = 8; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            t = __shfl_sync(0xffffffffu, t, lane & 1 ? 16 : 0);
            if ((lane & ~1) == src) acc[k * SG_CONV + tid] += t;
          }
        }
      }
    }
    if (__syncthreads_or(!live)) break;  // all roles leave together
  }
  if (drains && ci < pa) {
    const long o = ((long)bi * gridDim.x + blockIdx.x) * a.p * a.q;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int jj = slot * 8 + k;
      if (jj >= ndup + nown) break;
      const bool dup = jj < ndup;
      const int j = j0 + (dup ? jj : jj - ndup);
      double2 *const part = dup || a.mode == SL_GENERAL ? a.part0 : a.part1;
      if (a.mode == SL_GENERAL || ci <= j)
        reinterpret_cast<double *>(part + o + (long)ci * a.q + j)[odd] = acc[k * SG_CONV + tid];
    }
  }
  // on abort: the MMAs in flight (the issuer counts those that it issued)
  if (issuer && *abort && n > 0) warp_wait(bars + 8u * ((n - 1) & 1), ((n - 1) >> 1) & 1, abort, false);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
  if (tid == 0 && *abort) report_timeout(a.tmo);
}

template <typename T> size_t sg_smem(int nbp, bool each) {
  return 1024 + SlForm<T>::ND * 16384 + (size_t)SlForm<T>::NL * nbp * 128 + 8 * SG_CONV * 8 + sg_col_bytes(each) + 64;
}

}  // namespace

// most chunks per k-point that launch_gram_sl takes (partial-sum scratch sizing)
int sl_gram_chunks(int nb, long L) {
  const long want = (4L * sm_count() + nb - 1) / std::max(nb, 1);
  return (int)std::max<long>(1, std::min<long>({want, L / 128, 256}));
}

int launch_gram_sl(int nb, long L, int p, int q, int dtype, const void *A, long sa, const void *B, long sb, int mode,
                   double2 *part, int maxchunk, int *nchunk, cudaStream_t st, int *tmo, const int *act, bool each) {
  SlGramArgs a{};
  a.A = A;
  a.B = B;
  a.sa = sa;
  a.sb = sb;
  a.L = L;
  a.p = p;
  a.q = q;
  a.mode = mode;
  a.act = act;
  a.tmo = tmo;
  // blocks of up to 32 operand columns (8 levels of 64 accumulator columns fill TMEM); a pair's block has two per column
  const int most_cols = mode == SL_PAIR ? 16 : 32, nblk = (q + most_cols - 1) / most_cols;
  a.nbc = (q + nblk - 1) / nblk;
  a.nbp = (2 * a.nbc * (mode == SL_PAIR ? 2 : 1) + 15) / 16 * 16;
  // the chunk count with the least rows (plus a CTA's fixed cost, about 100 rows) in the longest sequence of CTAs per SM
  const long per = (long)nb * nblk, nsm = sm_count();
  const int most = (int)std::max<long>(1, std::min<long>(maxchunk, sl_gram_chunks(nb, L)));
  double best = 0.0;
  int c = 1;
  for (int k = 1; k <= most; ++k) {
    const long rows = ((L + k - 1) / k + SG_ROWS - 1) / SG_ROWS * SG_ROWS;
    const double cost = (double)((per * k + nsm - 1) / nsm) * (double)(rows + 100);
    if (k == 1 || cost < best) {
      best = cost;
      c = k;
    }
  }
  *nchunk = c;
  a.part0 = part;
  a.part1 = part + (size_t)nb * c * p * q;
  const size_t smem = dtype == PC_DFS ? sg_smem<float4>(a.nbp, false) : sg_smem<double2>(a.nbp, each);
  const dim3 grid(c, nblk, nb);
  // columns that a block extracts: its left columns, up to all p, and its own of B
  const int ncols = p + (mode == SL_SELF ? 0 : a.nbc);
  const int kind = dtype == PC_DFS ? 0 : (ncols <= 32 ? 1 : (ncols <= 64 ? 2 : 3)) + (each ? 3 : 0);
  if (kind == 0 && ncols > 32) {
    set_error("gram_sl: at most 32 columns of double-float pairs");
    return PC_EINVAL;
  }
  using Kernel = void (*)(SlGramArgs);
  static constexpr Kernel kernels[7] = {gram_sl_kernel<float4, 1, 3, false>,  gram_sl_kernel<double2, 1, 3, false>,
                                        gram_sl_kernel<double2, 2, 1, false>, gram_sl_kernel<double2, 3, 1, false>,
                                        gram_sl_kernel<double2, 1, 3, true>,  gram_sl_kernel<double2, 2, 1, true>,
                                        gram_sl_kernel<double2, 3, 1, true>};
  const Kernel kernel = kernels[kind];
  static bool configured[64][7] = {};  // per device
  int dev = 0;
  PC_CK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !configured[dev][kind]) {
    PC_CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(kind ? sg_smem<double2>(64, each) : sg_smem<float4>(64, false))));
    if (dev >= 0 && dev < 64) configured[dev][kind] = true;
  }
  kernel<<<grid, SG_THREADS, smem, st>>>(a);
  PC_CK_LAUNCH();
  return PC_OK;
}

}  // namespace pc
