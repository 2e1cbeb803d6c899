// Block updates Y = S C of complex128 blocks on the tensor cores (S: L x p, C: p x q complex), sliced exactly into
// FP16 digits (sliced.cuh).
//
// One real product per tile of 128 rows: accumulator row = row of S, K = the 2 p real and imaginary parts of a row,
// accumulator columns 2 j + c = parts of up to 32 columns of Y, once per level. Row l is held against one exponent
// E_l = max_i (e(S_li) + a_i), where a_i is the exponent of the largest entry of row i of C; row i of C is scaled by
// 2^-a_i, and its columns have exponents of their own. So a small column of S with large coefficients (a preconditioned
// residual) is held as accurately as a large one with small coefficients: every term S_li C_ij is rounded relative to
// the largest term of its row.
//
// One CTA (512 threads, one per SM) keeps the digits of C in shared memory and walks over row tiles of one k-point. A
// thread owns one row and a quarter of the columns (16-byte digit stores, no bank conflicts); it holds its elements in
// registers for the row's exponent, forms the digits in stages of 16 columns (two stages side by side in the 64-wide
// operand tile: digits of one stage while the MMAs of the stage before run) and loads the next tile's elements as soon
// as a stage's are used. The epilogue adds the levels as 64-bit integers and rounds once, in integer arithmetic (the
// FP64 pipe retires about 2 operations per clock and SM).
//
// Bound: integer instructions of the digit extraction and the epilogue. 8 k-points, 48 -> 16 columns at N = 32:
// 4.00 ms on the FP64 pipe (1.21 TFLOP/s, all of it), 0.53 ms here; 4 k-points, 57 -> 19 at N = 64: 27.5 and 2.67 ms;
// one k-point, 24 -> 8 at N = 16: 54.8 and 17.0 us; the smallest size tried (8 -> 4 columns of 1536 rows): 21.9 and
// 17.9 us. (For complex64 the same scheme with four digits was slower than the FP32 pipe: 1.29 against 0.97 ms for
// 57 -> 19 columns at N = 64.)
#include <cuda.h>
#include <cuda_runtime.h>

#include "sliced.cuh"

namespace pc {

namespace {

constexpr int SU_THREADS = 512;
constexpr int SU_COLS = 16;  // columns per stage
constexpr int SU_BAD = 1 << 20;
constexpr int SU_ND = 8;

__device__ int g_update_sl_error = 0;

struct SlUpdateArgs {
  const void *S;
  long ss;
  const double2 *C;
  long sc;
  void *Y;
  long sy;
  long L;
  int p, q, nbc, nbp, ntile;
  uint32_t tmem_cols;
  const int *act;
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

// NS: stages (p <= 16 NS)
template <int NS>
__global__ void __launch_bounds__(SU_THREADS, 1) update_sl_kernel(const SlUpdateArgs a) {
  using T = double2;
  constexpr int ND = SU_ND;
  constexpr int NC = 4 * NS;          // columns per thread
  constexpr int NATOM = (NS + 1) / 2;  // 64-wide operand tiles of C
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_addr(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *const sm = smem_raw + (base - raw);
  const uint32_t off_b = ND * 16384u, atom = (uint32_t)(ND * a.nbp) * 128u, off_e = off_b + NATOM * atom;
  int *const sE = reinterpret_cast<int *>(sm + off_e);  // [2][4][128] row exponents (per tile parity and column quarter)
  int *const sCA = sE + 1024, *const sCB = sCA + 64;    // exponents of the rows and columns of C
  const uint32_t off_bar = off_e + (1024u + 128u) * 4u;
  const uint32_t bars = base + off_bar;
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(sm + off_bar + 16);
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
  for (int t = tid; t < a.p * nbc && !bad; t += SU_THREADS) {
    const int i = t / nbc, j = t - i * nbc;
    const double2 c = Cb[(long)i * a.q + j];
    const int E = sCB[j] + sCA[i], ii = i & 31, kc = ii >> 2;  // four columns (8 values) per 16-byte chunk
    const unsigned long long cr = sl_round<ND>(sl_raw<ND>(c.x, E)), ci = sl_round<ND>(sl_raw<ND>(c.y, E)),
                             cn = sl_round<ND>(sl_raw<ND>(-c.y, E));
    // (x + i y)(cr + i ci): row 2 j holds (cr, -ci), row 2 j + 1 holds (ci, cr)
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const int rr = d * a.nbp + 2 * j;
      unsigned char *o = sm + off_b + (i >> 5) * atom + (ii & 3) * 4;
      *reinterpret_cast<unsigned *>(o + rr * 128 + ((kc ^ (rr & 7)) << 4)) = sl_digits<ND>(cr, cn, ND - 1 - d);
      *reinterpret_cast<unsigned *>(o + (rr + 1) * 128 + ((kc ^ ((rr + 1) & 7)) << 4)) = sl_digits<ND>(ci, cr, ND - 1 - d);
    }
  }
  fence_proxy_async();

  const int quarter = warp & 3, slot = warp >> 2;
  const uint32_t tdrain = tmem + ((uint32_t)(quarter * 32) << 16);
  T *const Yb = static_cast<T *>(a.Y) + (long)b * a.sy + (long)j0 * L;
  int n = 0, par = 0;
  for (long tile = blockIdx.x; tile < a.ntile; tile += gridDim.x, par ^= 1) {
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
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) ex = max(ex, sE[par * 512 + k * 128 + r]);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int buf = n & 1;
      if (n >= 2) bar_wait(bars + 8u * buf, ((n >> 1) & 1) ^ 1, abort);
      unsigned long long m[8];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = min(s * SU_COLS + 4 * g + c, a.p - 1);  // (columns past p are zero)
        sl_split<ND>(v[4 * s + c], ex - sCA[i], m[2 * c], m[2 * c + 1]);
      }
      load(s, tile + gridDim.x);
      unsigned char *o = sm + r * 128 + (((buf * 4 + g) ^ (r & 7)) << 4);
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        uint4 x;
        x.x = sl_digits<ND>(m[0], m[1], ND - 1 - d);
        x.y = sl_digits<ND>(m[2], m[3], ND - 1 - d);
        x.z = sl_digits<ND>(m[4], m[5], ND - 1 - d);
        x.w = sl_digits<ND>(m[6], m[7], ND - 1 - d);
        *reinterpret_cast<uint4 *>(o + d * 16384) = x;
      }
      fence_proxy_async();
      tc_fence_before();
      if (warp == 0) {
        named_sync(1 + buf, SU_THREADS);
        if (lane == 0) {
          tc_fence_after();
          const int nks = a.p - s * SU_COLS > SU_COLS / 2 ? 2 : 1;  // K steps of 8 columns
          for (int ks = 0; ks < nks; ++ks)
            sl_mma_step<ND, ND>(tmem, base, base + off_b + (s >> 1) * atom, (uint32_t)(buf * 64 + ks * 32),
                            (uint32_t)((s & 1) * 64 + ks * 32), a.nbp, s == 0 && ks == 0);
          mma_commit(bars + 8u * buf);
        }
        __syncwarp();
      } else {
        named_arrive(1 + buf, SU_THREADS);
      }
      ++n;
    }
    bar_wait(bars + 8u * ((n - 1) & 1), ((n - 1) >> 1) & 1, abort);
    tc_fence_after();
    // epilogue: lane = row, four accumulator columns (two columns of Y) at a time
    const int row = quarter * 32 + lane;
    const long l = tile * 128 + row;
    int E = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) E = max(E, sE[par * 512 + k * 128 + row]);
    for (int c0 = 4 * slot; c0 < 2 * nbc; c0 += 16) {
      __syncwarp();
      uint32_t w[ND][4];
#pragma unroll
      for (int lv = 0; lv < ND; ++lv) tmem_ld4(tdrain + (uint32_t)(lv * a.nbp + c0), w[lv]);
#pragma unroll
      for (int lv = 0; lv < ND; ++lv) tmem_wait4(w[lv]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = (c0 >> 1) + h;
        if (j >= nbc || l >= L) continue;
        T out;
        if (bad || E >= SU_BAD) {
          // an infinity or a NaN in the row or in C: plain FP64
          double re = 0.0, im = 0.0;
          for (int i = 0; i < a.p; ++i) {
            const double2 x = ld_c128(Sb + (long)i * L + l), c = Cb[(long)i * a.q + j];
            re = fma(x.x, c.x, fma(-x.y, c.y, re));
            im = fma(x.x, c.y, fma(x.y, c.x, im));
          }
          out = make_double2(re, im);
        } else {
          const int sc = E + sCB[j] - 2046 - 2 * (sl_bits<ND>() - 1) + 8 * (ND - 1);
          long long H[2];
          unsigned lo[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            long long hi = 0, s = 0;
#pragma unroll
            for (int lv = 0; lv < ND; ++lv) {
              const int x = __float2int_rn(__uint_as_float(w[lv][2 * h + u]));
              if (lv < ND - 4)
                hi += (long long)x * (1 << (8 * (ND - 5 - lv)));
              else
                s += (long long)x * (1 << (8 * (ND - 1 - lv)));
            }
            H[u] = hi + (s >> 32);
            lo[u] = (unsigned)s;
          }
          out = make_double2(sl_to_double(H[0], lo[0], sc), sl_to_double(H[1], lo[1], sc));
        }
        Yb[(long)j * L + l] = out;
      }
    }
  }
  __syncwarp();
  if (tid == 0 && *abort && n > 0) bar_wait(bars + 8u * ((n - 1) & 1), ((n - 1) >> 1) & 1, abort, false);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
  }
  if (tid == 0 && *abort) atomicExch(&g_update_sl_error, 1);
}

template <int NS>
int launch_su(SlUpdateArgs a, int nb, cudaStream_t st) {
  // columns of Y per block: all levels of 2 nbc columns in TMEM, the digits of C and of one tile in shared memory
  constexpr int ND = SU_ND, most_cols = NS > 2 ? 20 : 32;
  const int nqb = (a.q + most_cols - 1) / most_cols;
  a.nbc = (a.q + nqb - 1) / nqb;
  a.nbp = (2 * a.nbc + 7) / 8 * 8;
  a.ntile = (int)((a.L + 127) / 128);
  a.tmem_cols = 32;
  while (a.tmem_cols < (uint32_t)((ND + ((a.nbp >> 3) & 1)) * a.nbp)) a.tmem_cols *= 2;
  auto smem_of = [](int nbp) {
    return (size_t)1024 + ND * 16384 + (size_t)((NS + 1) / 2) * ND * nbp * 128 + (1024 + 128) * 4 + 64;
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
    PC_CK(cudaFuncSetAttribute(update_sl_kernel<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)smem_of(2 * most_cols)));
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  // a CTA's 512 threads of 128 registers take the SM: no second CTA waits for its TMEM columns there
  update_sl_kernel<NS><<<dim3(gx, nqb, nb), SU_THREADS, smem_of(a.nbp), st>>>(a);
  PC_CK_LAUNCH();
  return PC_OK;
}

}  // namespace

int launch_update_sl(int nb, long L, int p, int q, const void *S, long ss, const void *C, long sc, void *Y,
                     long sy, cudaStream_t st, const int *act) {
  SlUpdateArgs a{};
  a.S = S;
  a.ss = ss;
  a.C = static_cast<const double2 *>(C);
  a.sc = sc;
  a.Y = Y;
  a.sy = sy;
  a.L = L;
  a.p = p;
  a.q = q;
  a.act = act;
  switch ((p + SU_COLS - 1) / SU_COLS) {
    case 1: return launch_su<1>(a, nb, st);
    case 2: return launch_su<2>(a, nb, st);
    case 3: return launch_su<3>(a, nb, st);
    default: return launch_su<4>(a, nb, st);
  }
}

int update_sl_check() {
  int v = 0;
  PC_CK(cudaMemcpyFromSymbol(&v, g_update_sl_error, sizeof(int)));
  if (v) {
    const int zero = 0;
    PC_CK(cudaMemcpyToSymbol(g_update_sl_error, &zero, sizeof(int)));
    set_error("sliced update kernel: a pipeline wait ran out of time");
    return PC_ECUDA;
  }
  return PC_OK;
}

}  // namespace pc
