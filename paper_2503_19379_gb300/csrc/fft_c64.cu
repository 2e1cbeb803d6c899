// Complex64 FFT preconditioner W = P^{-1} R (Section 5.2, Algorithm 5.1, with the 3x3 mode symbol of
// eq. penalised_marix) for N = 8 .. 128: three passes over the block, each one HBM read and one HBM write.
//   1. forward transforms along x and y of one (component, z) plane held in shared memory;
//   2. along z, all three components of U consecutive (x, y) columns: forward transform, the exact inverse of the
//      mode's 3x3 symbol sigma I + (gamma - 1) conj(d) d^T times 1/N^3, inverse transform;
//   3. inverse transforms along y and x of each plane.
// A line transform of length N = N1 N2 (N2 = N up to 16, 8 at N = 32, 16 above) is a DFT of length N2 and one of length N1 (Cooley-Tukey) with
// the twiddles W_N between them; a thread holds N2 elements in registers. The small DFTs are radix-2 decimation in time on
// registers with the constant roots of unity of order 16. Inputs and outputs are in natural order, so the symbol is
// applied at the natural mode indices.
//
// What bounds the passes besides HBM is the trips through shared memory and the barriers around them, so the steps are
// ordered for few of both. Plane pass: the first axis' length-N2 DFTs; the length-N1 DFTs of both axes on an N1 x N1 block
// of a thread (N = 128: one axis after the other); the second axis' length-N2 DFTs, two exchanges in all. z pass: the
// length-N2 DFTs; then a thread takes the N1 modes of one residue and all three components through the length-N1 DFTs,
// the symbol and the inverse DFTs back; the inverse length-N2 DFTs. The middle steps write where they read, so
// one buffer serves and a step needs one barrier. 76 fields of N = 64: 0.71 ms with the axes one after the other, an
// exchange and a transposition each, N1 <= N2 split nearly even and the modes gathered once more for the symbol; 0.54 ms
// so (5.2 TB/s over the three passes). 256 fields of N = 32: 315 and 250 us; 20 of N = 128: 1.72 and 1.54 ms. Passes over
// blocks of fields that would stay in L2 were slower at every block size (0.61 to 0.95 ms): the launches get too small.
//
// Shared-memory layouts: every half warp touches each bank pair once. In a plane, the N1 pieces of a row are N2 + 1 apart,
// which makes the row stride N1 (mod N2); loads and stores of rows are N1 consecutive elements per thread group (32 bytes
// at N = 64), those of columns are consecutive threads on consecutive columns, as in the z pass.
#include <cmath>

#include "pc_internal.cuh"

namespace pc {

namespace {

constexpr int clog2(int n) { return n <= 1 ? 0 : 1 + clog2(n / 2); }
constexpr int cbrev(int i, int bits) {
  int r = 0;
  for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
  return r;
}
// cos(2 pi e / 16) for e = 0 .. 15
__host__ __device__ constexpr float cos16(int e) {
  switch (e & 15) {
    case 0: return 1.0f;
    case 1: case 15: return 0.92387953251128676f;
    case 2: case 14: return 0.70710678118654752f;
    case 3: case 13: return 0.38268343236508977f;
    case 4: case 12: return 0.0f;
    case 5: case 11: return -0.38268343236508977f;
    case 6: case 10: return -0.70710678118654752f;
    case 7: case 9: return -0.92387953251128676f;
    default: return -1.0f;
  }
}

// x * exp(-2 pi i e / 16) (forward) or x * exp(+2 pi i e / 16) (inverse); e is a compile-time constant after unrolling
template <bool INV> __device__ __forceinline__ float2 rot16(float2 x, int e) {
  e &= 15;
  if (e == 0) return x;
  if (e == 8) return make_float2(-x.x, -x.y);
  if (e == 4) return INV ? make_float2(-x.y, x.x) : make_float2(x.y, -x.x);
  if (e == 12) return INV ? make_float2(x.y, -x.x) : make_float2(-x.y, x.x);
  const float c = cos16(e), s = cos16(e - 4);  // sin(t) = cos(t - pi / 2)
  return INV ? make_float2(x.x * c - x.y * s, x.x * s + x.y * c) : make_float2(x.x * c + x.y * s, x.y * c - x.x * s);
}

// In-register DFT of length R <= 16 (natural order in and out): radix-2 decimation in time after the bit-reversal
// permutation (a renaming of registers).
template <int R, bool INV> __device__ __forceinline__ void dft(float2 *v) {
  if constexpr (R > 1) {
    constexpr int LOG = clog2(R);
    float2 t[R];
#pragma unroll
    for (int i = 0; i < R; ++i) t[i] = v[cbrev(i, LOG)];
#pragma unroll
    for (int len = 2; len <= R; len <<= 1) {
#pragma unroll
      for (int blk = 0; blk < R; blk += len) {
#pragma unroll
        for (int j = 0; j < len / 2; ++j) {
          const float2 a = t[blk + j];
          const float2 b = rot16<INV>(t[blk + j + len / 2], j * (16 / len));
          t[blk + j] = make_float2(a.x + b.x, a.y + b.y);
          t[blk + j + len / 2] = make_float2(a.x - b.x, a.y - b.y);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = t[i];
  }
}

// x * w (forward) or x * conj(w) (inverse)
template <bool INV> __device__ __forceinline__ float2 twmul(float2 x, float2 w) {
  return INV ? make_float2(x.x * w.x + x.y * w.y, x.y * w.x - x.x * w.y)
             : make_float2(x.x * w.x - x.y * w.y, x.x * w.y + x.y * w.x);
}

// Split of a length-N transform.
template <int N> struct Split {
  static constexpr int N2 = N < 16 ? N : (N == 32 ? 8 : 16);  // (32 = 2 x 16: 262 us for 256 fields; 4 x 8: 250)
  static constexpr int N1 = N / N2;
  static_assert(N1 * N2 == N && N1 <= 8, "unsupported length");
};

// planes per CTA (at least 128 threads where the planes of a component allow it; P divides the 3 N planes of a field)
template <int N> struct PlaneCfg {
  static constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2;
  static constexpr int P0 = (N * N1 >= 128) ? 1 : 128 / (N * N1);
  static constexpr int P = P0 < N ? P0 : N;
  static constexpr int PN = N2 + 1;   // stride of the N1 pieces of a row
  static constexpr int LD = N1 * PN;  // row stride of the plane
  static constexpr int THREADS = P * N * N1;
  static constexpr size_t smem() { return sizeof(float2) * ((size_t)P * N * LD + N); }
};

// twiddle table W_N^t = exp(-2 pi i t / N), t < N, from the context's table of the first N / 2
__device__ __forceinline__ void load_twiddles(float2 *s_tw, const float2 *tw, int N) {
  for (int t = threadIdx.x; t < N / 2; t += blockDim.x) {
    const float2 w = tw[t];
    s_tw[t] = w;
    s_tw[t + N / 2] = make_float2(-w.x, -w.y);
  }
}

// Forward (x then y) or inverse (y then x) transforms of P planes (component, z) per CTA. grid (3N / P, m, nb).
template <int N, bool FWD>
__global__ void __launch_bounds__(PlaneCfg<N>::THREADS) fft_plane_kernel(const float2 *__restrict__ in, long si,
                                                                         float2 *__restrict__ out, long so,
                                                                         const float2 *__restrict__ tw,
                                                                         const int *__restrict__ act) {
  using CF = PlaneCfg<N>;
  constexpr int N1 = CF::N1, N2 = CF::N2, P = CF::P, LD = CF::LD, PN = CF::PN, T = CF::THREADS;
  constexpr bool INV = !FWD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *s_tw = reinterpret_cast<float2 *>(smem_raw);
  float2 *A = s_tw + N;  // planes [P N rows][N1 pieces, PN apart][N2]
  const long n = (long)N * N * N;
  const int b = act ? act[blockIdx.z] : (int)blockIdx.z;
  const long off = (long)blockIdx.y * 3 * n + (long)blockIdx.x * P * N * N;
  const float2 *src = in + (long)b * si + off;
  float2 *dst = out + (long)b * so + off;
  load_twiddles(s_tw, tw, N);
  const int tid = threadIdx.x;
  // a thread's share of the outer steps: of a row (plane, y) the elements n1 + N1 j, or of a column the rows m1 + N1 j
  const int n1 = tid % N1, row = tid / N1;
  const int x = tid % N, m1 = tid / N % N1, pl = tid / (N * N1);
  const int xs = x / N2 * PN + x % N2;  // the column's place in a row
  float2 v[N2];

  // ---- the first axis' DFTs of length N2 over its elements n1 + N1 j; result k2 of piece n1 to n1 N2 + k2
#pragma unroll
  for (int j = 0; j < N2; ++j) v[j] = FWD ? src[row * N + n1 + N1 * j] : src[(pl * N + m1 + N1 * j) * N + x];
  __syncthreads();  // twiddle table
  dft<N2, INV>(v);
#pragma unroll
  for (int j = 1; j < N2; ++j)
    if (N1 > 1) v[j] = twmul<INV>(v[j], s_tw[(FWD ? n1 : m1) * j]);
#pragma unroll
  for (int j = 0; j < N2; ++j) A[FWD ? row * LD + n1 * PN + j : (pl * N + m1 * N2 + j) * LD + xs] = v[j];
  __syncthreads();

  // ---- DFTs of length N1 of both axes, in place. Stride N2 on both: the second axis' elements r + N2 i, result k1 of
  // residue r times W_N^(r k1)
  if constexpr (N1 > 1 && N1 <= 4) {
    for (int i = tid; i < P * N2 * N2; i += T) {
      const int ix = i % N2, iy = i / N2 % N2, rr = FWD ? iy : ix;
      float2 *B = A + (i / (N2 * N2) * N + iy) * LD + ix;
      float2 w[N1][N1];  // [y][x]
#pragma unroll
      for (int e = 0; e < N1; ++e)
#pragma unroll
        for (int c = 0; c < N1; ++c) w[e][c] = B[e * N2 * LD + c * PN];
#pragma unroll
      for (int axis = 0; axis < 2; ++axis) {  // the first axis, then the second
        if ((axis == 0) == FWD) {
#pragma unroll
          for (int e = 0; e < N1; ++e) dft<N1, INV>(w[e]);
        } else {
#pragma unroll
          for (int c = 0; c < N1; ++c) {
            float2 q[N1];
#pragma unroll
            for (int e = 0; e < N1; ++e) q[e] = w[e][c];
            dft<N1, INV>(q);
#pragma unroll
            for (int e = 0; e < N1; ++e) w[e][c] = q[e];
          }
        }
      }
#pragma unroll
      for (int k = 1; k < N1; ++k) {
        const float2 t = s_tw[rr * k];
#pragma unroll
        for (int c = 0; c < N1; ++c) {
          float2 &z = FWD ? w[k][c] : w[c][k];
          z = twmul<INV>(z, t);
        }
      }
#pragma unroll
      for (int e = 0; e < N1; ++e)
#pragma unroll
        for (int c = 0; c < N1; ++c) B[e * N2 * LD + c * PN] = w[e][c];
    }
    __syncthreads();
  } else if constexpr (N1 > 4) {
    // one axis after the other: rows then columns (forward), columns then rows (inverse)
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const bool rows = FWD == (s == 0);
      for (int i = tid; i < P * N * N2; i += T) {
        // rows: (row, ix) of the row's pieces; columns: (plane, iy, x)
        const int r = rows ? i % N2 : i / N % N2;
        float2 *B = rows ? A + i / N2 * LD + r
                         : A + (i / (N * N2) * N + r) * LD + i % N / N2 * PN + i % N % N2;
        const int st = rows ? PN : N2 * LD;
        float2 w[N1];
#pragma unroll
        for (int e = 0; e < N1; ++e) w[e] = B[e * st];
        dft<N1, INV>(w);
        if (s == 1) {
#pragma unroll
          for (int k = 1; k < N1; ++k) w[k] = twmul<INV>(w[k], s_tw[r * k]);
        }
#pragma unroll
        for (int e = 0; e < N1; ++e) B[e * st] = w[e];
      }
      __syncthreads();
    }
  }

  // ---- the second axis' DFTs of length N2 over the residues of k1 = n1 (m1): outputs k1 + N1 k2
#pragma unroll
  for (int j = 0; j < N2; ++j) v[j] = A[FWD ? (pl * N + m1 * N2 + j) * LD + xs : row * LD + n1 * PN + j];
  dft<N2, INV>(v);
#pragma unroll
  for (int j = 0; j < N2; ++j) {
    if (FWD)
      dst[(pl * N + m1 + N1 * j) * N + x] = v[j];
    else
      dst[row * N + n1 + N1 * j] = v[j];
  }
}

// columns per CTA of the z pass, and threads: one per task of the outer steps (3 N1 U), or a third of that where the
// middle step's N2 U tasks would leave more of them idle (N = 32, 128). The other choice: 271 against 250 us for 256
// fields of N = 32, 585 against 545 us for 76 of N = 64, 1.60 against 1.53 ms for 20 of N = 128
template <int N> struct ZCfg {
  static constexpr int N1 = Split<N>::N1;
  static constexpr int U = N == 64 ? 16 : 32;
  static constexpr int THREADS = U * N1 * (3 * N1 <= Split<N>::N2 ? 3 : 1);
  static constexpr size_t smem() {
    // elements [3][N][U], twiddles N, symbols: x/y parts [3][U] and z part [3][N]
    return sizeof(float2) * ((size_t)3 * N * U + N + 3 * (size_t)U + 3 * (size_t)N);
  }
};

// Along z with the symbol, for U consecutive (x, y) columns (flattened index xy = y N + x) and all 3 components.
// grid (N^2 / U, m, nb). LAT: general lattice (Section 4.2.2), d_i = sum_j (part of axis j)(m_j) from the tables
// [b][i][j][N]; otherwise d_i from the per-axis tables [b][i][N].
template <int N, bool LAT>
__global__ void __launch_bounds__(ZCfg<N>::THREADS) fft_zsym_kernel(const float2 *__restrict__ in, long si,
                                                                    float2 *__restrict__ out, long so,
                                                                    const float2 *__restrict__ tw,
                                                                    const double2 *__restrict__ sym,
                                                                    const KParam *__restrict__ kp,
                                                                    const int *__restrict__ act, int laplacian) {
  using CF = ZCfg<N>;
  constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2, U = CF::U, T = CF::THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *E = reinterpret_cast<float2 *>(smem_raw);  // [3][N][U]
  float2 *s_tw = E + 3 * N * U;                      // [N]
  float2 *dxy = s_tw + N;                            // [3][U]: x and y parts of d_i at each column
  float2 *dz = dxy + 3 * U;                          // [3][N]: z part of d_i (on the cube: d_3 itself)
  const long n = (long)N * N * N;
  const int b = act ? act[blockIdx.z] : (int)blockIdx.z;
  const int xy0 = blockIdx.x * U;
  const long base_i = (long)b * si + (long)blockIdx.y * 3 * n + xy0;
  const long base_o = (long)b * so + (long)blockIdx.y * 3 * n + xy0;
  load_twiddles(s_tw, tw, N);
  {
    const double2 *symb = sym + (long)b * (LAT ? 9 : 3) * N;
    for (int i = threadIdx.x; i < 3 * U; i += blockDim.x) {
      const int u = i / 3, c = i % 3;
      const int xx = (xy0 + u) % N, yy = (xy0 + u) / N;
      double re, im;
      if (LAT) {
        const double2 px = symb[(c * 3 + 0) * N + xx], py = symb[(c * 3 + 1) * N + yy];
        re = px.x + py.x;
        im = px.y + py.y;
      } else {
        // cube: d_1 depends on x, d_2 on y, d_3 on z only
        const double2 d = c == 0 ? symb[xx] : (c == 1 ? symb[N + yy] : make_double2(0.0, 0.0));
        re = d.x;
        im = d.y;
      }
      dxy[c * U + u] = make_float2((float)re, (float)im);
    }
    for (int i = threadIdx.x; i < 3 * N; i += blockDim.x) {
      const int c = i / N, zz = i % N;
      const double2 d = LAT ? symb[(c * 3 + 2) * N + zz] : (c == 2 ? symb[2 * N + zz] : make_double2(0.0, 0.0));
      dz[i] = make_float2((float)d.x, (float)d.y);
    }
  }
  const int tid = threadIdx.x, u = tid % U;  // (U divides T: a thread stays on its column)
  // forward along z, the DFTs of length N2 over z = n1 + N1 j: result k2 to n1 N2 + k2
  constexpr int R1 = 3 * N1 * U / T;
#pragma unroll
  for (int it = 0; it < R1; ++it) {
    const int r = (tid + it * T) / U, n1 = r % N1, c = r / N1;
    float2 v[N2];
#pragma unroll
    for (int j = 0; j < N2; ++j) v[j] = in[base_i + (long)c * n + (n1 + N1 * j) * N * N + u];
    if (it == 0) __syncthreads();  // twiddles and symbols
    dft<N2, false>(v);
#pragma unroll
    for (int j = 1; j < N2; ++j)
      if (N1 > 1) v[j] = twmul<false>(v[j], s_tw[n1 * j]);
#pragma unroll
    for (int j = 0; j < N2; ++j) E[(c * N + n1 * N2 + j) * U + u] = v[j];
  }
  __syncthreads();
  // the modes kz = k2 + N2 k1 of residue k2: DFTs of length N1, the symbol's inverse on all three components, the DFTs back
  // and their twiddles
  {
    const float fac = kp[b].pfacf;  // (gamma - 1) / gamma
    const float scale = 1.0f / (float)n;
    const float2 e1 = dxy[u], e2 = dxy[U + u], e3 = dxy[2 * U + u];
    for (int k2 = tid / U; k2 < N2; k2 += T / U) {
      float2 *B = E + k2 * U + u;
      float2 w[3][N1];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int a = 0; a < N1; ++a) w[c][a] = B[(c * N + a * N2) * U];
        dft<N1, false>(w[c]);
      }
#pragma unroll
      for (int a = 0; a < N1; ++a) {
        const int kz = k2 + N2 * a;
        const float2 d1 = LAT ? cadd(e1, dz[kz]) : e1, d2 = LAT ? cadd(e2, dz[N + kz]) : e2;
        const float2 d3 = LAT ? cadd(e3, dz[2 * N + kz]) : dz[2 * N + kz];
        const float sigma = d1.x * d1.x + d1.y * d1.y + d2.x * d2.x + d2.y * d2.y + d3.x * d3.x + d3.y * d3.y;
        float2 &r1 = w[0][a], &r2 = w[1][a], &r3 = w[2][a];
        if (!(sigma > 0.f)) {
          r1 = r2 = r3 = make_float2(0.f, 0.f);
        } else {
          const float rs = __frcp_rn(sigma);
          if (!laplacian) {
            // r_c - (gamma - 1) / (gamma sigma) conj(d_c) (d^T r)
            const float2 sd = cscale(cadd(cadd(cmul(d1, r1), cmul(d2, r2)), cmul(d3, r3)), fac * rs);
            r1 = csub(r1, cmulc(d1, sd));
            r2 = csub(r2, cmulc(d2, sd));
            r3 = csub(r3, cmulc(d3, sd));
          }
          const float f = scale * rs;
          r1 = cscale(r1, f);
          r2 = cscale(r2, f);
          r3 = cscale(r3, f);
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dft<N1, true>(w[c]);
#pragma unroll
        for (int a = 0; a < N1; ++a)
          B[(c * N + a * N2) * U] = a == 0 ? w[c][a] : twmul<true>(w[c][a], s_tw[a * k2]);
      }
    }
  }
  __syncthreads();
  // inverse along z: the DFTs of length N2 over k2, outputs z = n1 + N1 j
#pragma unroll
  for (int it = 0; it < R1; ++it) {
    const int r = (tid + it * T) / U, n1 = r % N1, c = r / N1;
    float2 v[N2];
#pragma unroll
    for (int j = 0; j < N2; ++j) v[j] = E[(c * N + n1 * N2 + j) * U + u];
    dft<N2, true>(v);
#pragma unroll
    for (int j = 0; j < N2; ++j) out[base_o + (long)c * n + (n1 + N1 * j) * N * N + u] = v[j];
  }
}

template <int N>
int launch_precond_c64_n(pc_ctx *ctx, int nb, int m, const float2 *R, long sr, float2 *W, long sw, const int *act) {
  using PC = PlaneCfg<N>;
  using ZC = ZCfg<N>;
  static bool configured = false;
  if (!configured) {
    PC_CK(cudaFuncSetAttribute(fft_plane_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)PC::smem()));
    PC_CK(cudaFuncSetAttribute(fft_plane_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)PC::smem()));
    PC_CK(cudaFuncSetAttribute(fft_zsym_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)ZC::smem()));
    PC_CK(cudaFuncSetAttribute(fft_zsym_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)ZC::smem()));
    configured = true;
  }
  const float2 *tw = ctx->twf.as<float2>();
  const int lap = ctx->opts.precond == PC_PRECOND_LAPLACIAN;
  fft_plane_kernel<N, true><<<dim3(3 * N / PC::P, m, nb), PC::THREADS, PC::smem(), ctx->stream>>>(R, sr, W, sw, tw,
                                                                                                  act);
  PC_CK_LAUNCH();
  if (ctx->lat)
    fft_zsym_kernel<N, true><<<dim3(N * N / ZC::U, m, nb), ZC::THREADS, ZC::smem(), ctx->stream>>>(
        W, sw, W, sw, tw, ctx->symd.as<double2>(), ctx->kparam.as<KParam>(), act, lap);
  else
    fft_zsym_kernel<N, false><<<dim3(N * N / ZC::U, m, nb), ZC::THREADS, ZC::smem(), ctx->stream>>>(
        W, sw, W, sw, tw, ctx->symd.as<double2>(), ctx->kparam.as<KParam>(), act, lap);
  PC_CK_LAUNCH();
  fft_plane_kernel<N, false><<<dim3(3 * N / PC::P, m, nb), PC::THREADS, PC::smem(), ctx->stream>>>(W, sw, W, sw, tw,
                                                                                                   act);
  PC_CK_LAUNCH();
  return PC_OK;
}

}  // namespace

// complex64 path for 8 <= N <= 128 (cube and general lattice); PC_EUNSUPPORTED for other sizes
int launch_precond_c64(pc_ctx *ctx, int nb, int m, const void *R, long sr, void *W, long sw, const int *act) {
  const float2 *Rf = static_cast<const float2 *>(R);
  float2 *Wf = static_cast<float2 *>(W);
  switch (ctx->N) {
    case 8: return launch_precond_c64_n<8>(ctx, nb, m, Rf, sr, Wf, sw, act);
    case 16: return launch_precond_c64_n<16>(ctx, nb, m, Rf, sr, Wf, sw, act);
    case 32: return launch_precond_c64_n<32>(ctx, nb, m, Rf, sr, Wf, sw, act);
    case 64: return launch_precond_c64_n<64>(ctx, nb, m, Rf, sr, Wf, sw, act);
    case 128: return launch_precond_c64_n<128>(ctx, nb, m, Rf, sr, Wf, sw, act);
    default: return PC_EUNSUPPORTED;
  }
}

}  // namespace pc
