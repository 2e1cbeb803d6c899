// The FP64-accurate kernels of the mixed-precision solve, in double-float arithmetic (dfloat.cuh) on the FP32 pipe
// (GB300: 75 TFLOP/s FP32 against 1.2 TFLOP/s FP64). The solver's block X is stored as double-float pairs (PC_DFS,
// one float4 per complex element), so the stencils do no FP64 arithmetic on it; the public entry point takes complex128
// and converts on load and store.
//   op_df_kernel / opz_df_kernel  AX = Op X (the stencil of stencil.cu; differences, shifts, M0, gamma in
//                     double-float), or, in the solver, the residual epilogue: R = AX - X Theta and complex64 copies
//                     of R, X and AX, plus column norms (AX itself is not stored)
//   launch_update_df  X' = X C + Z  (Z: the complex64 correction [W P] coef_{W,P}; on the tensor cores, update_sl.cu)
//   launch_gram_df    G = X^H X  (on the tensor cores, gram_sl.cu)
#include <cmath>
#include <type_traits>

#include "dfloat.cuh"
#include "pc_internal.cuh"
#include "sliced.cuh"

namespace pc {

// ---------------------------------------------------------------- packed complex double-float
// A complex double-float as two packed FP32 pairs, hi = (re.hi, im.hi) and lo = (re.lo, im.lo): every operation runs on
// both parts with one instruction (add, mul, fma .f32x2). Their rate in results is that of the scalar ones (measured: 124
// and 119 per clock and SM), in half the issue slots, and the stencils below are bound by issue in the solver's pair
// storage (71% of the cycles with scalar operations, the FMA pipe 60% busy). On complex128 blocks the FP64 pipe bounds
// them, 76% busy with the conversions to pairs and back, of halo points too (issue 37%, FMA 22%): 15 k-points x 16
// fields at N = 32 take 1.10 ms with scalar operations and 1.00 ms with these. The operations and their order are those
// of dfloat.cuh: the same bits.
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, 0xbf800000bf800000ull, a); }  // b (-1, -1) + a
__device__ __forceinline__ f32x2 swap2(f32x2 v) {
  const float2 t = unpack2(v);
  return pack2(t.y, t.x);
}

struct zdf {
  f32x2 hi, lo;
};
__device__ __forceinline__ zdf zdf_quick(f32x2 a, f32x2 b) {  // quick_two_sum
  zdf r;
  r.hi = add2(a, b);
  r.lo = sub2(b, sub2(r.hi, a));
  return r;
}
__device__ __forceinline__ zdf cdf_add(zdf x, zdf y) {
  const f32x2 s = add2(x.hi, y.hi), bb = sub2(s, x.hi);
  const f32x2 e = add2(sub2(x.hi, sub2(s, bb)), sub2(y.hi, bb));
  return zdf_quick(s, add2(e, add2(x.lo, y.lo)));
}
__device__ __forceinline__ zdf cdf_sub(zdf x, zdf y) {
  const f32x2 s = sub2(x.hi, y.hi), bb = sub2(s, x.hi);
  const f32x2 e = sub2(sub2(x.hi, sub2(s, bb)), add2(y.hi, bb));
  return zdf_quick(s, add2(e, sub2(x.lo, y.lo)));
}
// a s for a real double-float s (df_mul(a, s) for both parts)
__device__ __forceinline__ zdf cdf_scale(zdf a, df s) {
  const f32x2 sh = pack2(s.hi, s.hi), sl = pack2(s.lo, s.lo);
  const f32x2 p = mul2(a.hi, sh);
  f32x2 e = fma2(a.hi, sh, mul2(p, 0xbf800000bf800000ull));
  e = fma2(a.hi, sl, e);
  e = fma2(a.lo, sh, e);
  return zdf_quick(p, e);
}
// i k s for a real double-float k as the pairs (-k, k) in kp and (k, -k) in km: df_mul(k, .) of the exchanged parts
struct kdf {
  f32x2 hp, lp, hm, lm;
};
__device__ __forceinline__ kdf kdf_of(float hi, float lo) {
  return kdf{pack2(-hi, hi), pack2(-lo, lo), pack2(hi, -hi), pack2(lo, -lo)};
}
__device__ __forceinline__ zdf imul(zdf s, f32x2 kh, f32x2 kl, f32x2 nkh, f32x2 nkl) {
  const f32x2 sh = swap2(s.hi), sl = swap2(s.lo);
  const f32x2 p = mul2(kh, sh);
  f32x2 e = fma2(nkh, sh, p);  // minus the rounding error of p
  e = fma2(nkh, sl, e);
  e = fma2(nkl, sh, e);
  zdf r;
  r.hi = sub2(p, e);
  r.lo = sub2(sub2(p, r.hi), e);
  return r;
}

__device__ __forceinline__ zdf ld_zdf(const double2 *p) {
  const double2 v = *p;
  const df re = df_from(v.x), im = df_from(v.y);
  return zdf{pack2(re.hi, im.hi), pack2(re.lo, im.lo)};
}
__device__ __forceinline__ zdf ld_zdf(const float4 *p) {
  const float4 v = *p;
  return zdf{pack2(v.x, v.z), pack2(v.y, v.w)};
}
__device__ __forceinline__ cdf to_cdf(zdf z) {
  const float2 h = unpack2(z.hi), l = unpack2(z.lo);
  return cdf{df{h.x, l.x}, df{h.y, l.y}};
}
__device__ __forceinline__ void st_cdf(double2 *p, zdf z) { st_cdf(p, to_cdf(z)); }
__device__ __forceinline__ void st_cdf(float4 *p, zdf z) { st_cdf(p, to_cdf(z)); }

// ---------------------------------------------------------------- stencil
// (D f)_r = ih (f_{r+1} - f_r) + i kh (f_r + f_{r+1});  (D' g)_r = ih (g_{r-1} - g_r) - i kh (g_{r-1} + g_r)
__device__ __forceinline__ zdf dfwd_df(zdf f0, zdf f1, f32x2 ih, const kdf &k) {
  const zdf a = cdf_sub(f1, f0), s = cdf_add(f0, f1);
  return cdf_add(zdf{mul2(a.hi, ih), mul2(a.lo, ih)}, imul(s, k.hp, k.lp, k.hm, k.lm));
}
__device__ __forceinline__ zdf dbwd_df(zdf gm, zdf g0, f32x2 ih, const kdf &k) {
  const zdf a = cdf_sub(gm, g0), s = cdf_add(gm, g0);
  return cdf_add(zdf{mul2(a.hi, ih), mul2(a.lo, ih)}, imul(s, k.hm, k.lm, k.hp, k.lp));
}

// Residual epilogue of the stencil (the mixed solve's phase 2): instead of AX the kernel writes, per point,
// r = AX - theta_j X rounded to complex64 (twice: the preconditioner's input slot and the persistent copy used by
// the Rayleigh-Ritz coupling), complex64 copies of X and AX for the complex64 Gram products, and per-block partial
// sums of |r|^2 and |x|^2 (FP32 per thread, FP64 per block), reduced per column by residual_reduce.
struct ResidArgs {
  const double *theta;  // [nb][m]
  int m;
  float2 *R1, *R2, *X32, *AX32;
  long sr1, sr2, sx32, sax32;
  double *part;  // [nb][m][blocks per field][2]
};

__device__ __forceinline__ float2 cdf_round(zdf a) { return unpack2(add2(a.hi, a.lo)); }
__device__ __forceinline__ float2 cdf_high(zdf a) { return unpack2(a.hi); }
__device__ __forceinline__ float2 cdf_high(cdf a) { return make_float2(a.re.hi, a.im.hi); }
__device__ __forceinline__ float2 cdf_round(cdf a) { return make_float2(a.re.hi + a.re.lo, a.im.hi + a.im.lo); }
__device__ __forceinline__ df ld_m0(const float2 *p) {
  const float2 v = *p;
  return df{v.x, v.y};
}

// writes the three components of one point; returns |r|^2 and |x|^2 contributions
template <typename Z>
__device__ __forceinline__ void resid_point(const ResidArgs &ra, int b, int j, long n, long gi, df th, const Z (&y)[3],
                                            const Z (&x)[3], float &sr, float &sxx) {
  const long L = 3 * n;
  float2 *r1 = ra.R1 + (long)b * ra.sr1 + (long)j * L, *r2 = ra.R2 + (long)b * ra.sr2 + (long)j * L;
  float2 *x32 = ra.X32 + (long)b * ra.sx32 + (long)j * L, *ax32 = ra.AX32 + (long)b * ra.sax32 + (long)j * L;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Z r = cdf_sub(y[c], cdf_scale(x[c], th));
    const float2 rf = cdf_round(r), xf = cdf_high(x[c]);
    const long o = c * n + gi;
    r1[o] = rf;
    r2[o] = rf;
    x32[o] = xf;
    ax32[o] = cdf_round(y[c]);
    sr += rf.x * rf.x + rf.y * rf.y;
    sxx += xf.x * xf.x + xf.y * xf.y;
  }
}

// block sum of (sr, sxx) into the partial-sum slot of this block
__device__ __forceinline__ void resid_block_sum(const ResidArgs &ra, float sr, float sxx) {
  __shared__ double red[2][32];
  double a = sr, c = sxx;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[0][w] = a;
    red[1][w] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0, s1 = 0;
    for (int i = 0; i < nw; ++i) {
      s0 += red[0][i];
      s1 += red[1][i];
    }
    double *o = ra.part + (((long)blockIdx.z * ra.m + blockIdx.y) * gridDim.x + blockIdx.x) * 2;
    o[0] = s0;
    o[1] = s1;
  }
}

template <int TX, int TY, int TZ> constexpr size_t op_df_smem_bytes() {
  return sizeof(zdf) * (size_t)(3 * (TZ + 2) * (TY + 2) * (TX + 2) + 3 * (TZ + 1) * (TY + 1) * (TX + 1) +
                                (TZ + 1) * (TY + 1) * (TX + 1));
}

// Same tiling as op_kernel (stencil.cu): a face tile with a one-point halo, e = M0 A' v on the tile grown upward,
// c = B v on the tile grown downward, then y = A e + gamma B' c. The grid spacing factor ih = N is a power of two,
// so scaling by it is exact in double-float.
// The block is complex128 (converted on load and store) for the public entry point, double-float pairs (PC_DFS) for
// the solver's fused residual version.
template <bool RES> using df_store_t = typename std::conditional<RES, float4, double2>::type;

__device__ __forceinline__ df kp_df(float hi, float lo) { return df{hi, lo}; }

template <int TX, int TY, int TZ, bool RES>
__global__ void __launch_bounds__(256) op_df_kernel(const df_store_t<RES> *__restrict__ X, long sx,
                                                    df_store_t<RES> *__restrict__ Y, long sy,
                                                    const float2 *__restrict__ m0, const KParam *__restrict__ kp,
                                                    const int *__restrict__ act, int logN, const ResidArgs ra) {
  using XS = df_store_t<RES>;
  constexpr int VX = TX + 2, VY = TY + 2, VZ = TZ + 2;
  constexpr int EX = TX + 1, EY = TY + 1, EZ = TZ + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  zdf *v = reinterpret_cast<zdf *>(smem_raw);
  zdf *e = v + 3 * VZ * VY * VX;
  zdf *c = e + 3 * EZ * EY * EX;
  const int N = 1 << logN, mask = N - 1;
  const long n = 1L << (3 * logN);
  const int b = act ? act[blockIdx.z] : (int)blockIdx.z;
  const int j = blockIdx.y;
  const int tilesX = N / TX, tilesY = N / TY;
  int t = blockIdx.x;
  const int x0 = (t % tilesX) * TX;
  t /= tilesX;
  const int y0 = (t % tilesY) * TY;
  const int z0 = (t / tilesY) * TZ;
  const XS *Xb = X + (long)b * sx + (long)j * 3 * n;
  XS *Yb = Y + (long)b * sy + (long)j * 3 * n;
  const KParam p = kp[b];
  const kdf kh0 = kdf_of(p.khf[0], p.khl[0]), kh1 = kdf_of(p.khf[1], p.khl[1]), kh2 = kdf_of(p.khf[2], p.khl[2]);
  const df gam = kp_df(p.gammaf, p.gammal);
  const f32x2 ih = pack2((float)N, (float)N);

  for (int i = threadIdx.x; i < 3 * VZ * VY * VX; i += blockDim.x) {
    int lx = i % VX, r = i / VX;
    int ly = r % VY;
    r /= VY;
    int lz = r % VZ, comp = r / VZ;
    int gx = (x0 + lx - 1) & mask, gy = (y0 + ly - 1) & mask, gz = (z0 + lz - 1) & mask;
    v[i] = ld_zdf(Xb + comp * n + ((long)gz << (2 * logN)) + ((long)gy << logN) + gx);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < EZ * EY * EX; i += blockDim.x) {
    const int ex = i % EX, ey = (i / EX) % EY, ez = i / (EX * EY);
#define VV(comp, dz, dy, dx) v[(((comp) * VZ + ez + 1 + (dz)) * VY + ey + 1 + (dy)) * VX + ex + 1 + (dx)]
    const zdf v1 = VV(0, 0, 0, 0), v2 = VV(1, 0, 0, 0), v3 = VV(2, 0, 0, 0);
    const zdf d3v2 = dbwd_df(VV(1, -1, 0, 0), v2, ih, kh2);
    const zdf d2v3 = dbwd_df(VV(2, 0, -1, 0), v3, ih, kh1);
    const zdf d3v1 = dbwd_df(VV(0, -1, 0, 0), v1, ih, kh2);
    const zdf d1v3 = dbwd_df(VV(2, 0, 0, -1), v3, ih, kh0);
    const zdf d2v1 = dbwd_df(VV(0, 0, -1, 0), v1, ih, kh1);
    const zdf d1v2 = dbwd_df(VV(1, 0, 0, -1), v2, ih, kh0);
#undef VV
    const int gx = (x0 + ex) & mask, gy = (y0 + ey) & mask, gz = (z0 + ez) & mask;
    const long gi = ((long)gz << (2 * logN)) + ((long)gy << logN) + gx;
    const int eo = (ez * EY + ey) * EX + ex;
    e[eo] = cdf_scale(cdf_sub(d3v2, d2v3), ld_m0(m0 + gi));
    e[EZ * EY * EX + eo] = cdf_scale(cdf_sub(d1v3, d3v1), ld_m0(m0 + n + gi));
    e[2 * EZ * EY * EX + eo] = cdf_scale(cdf_sub(d2v1, d1v2), ld_m0(m0 + 2 * n + gi));
#define WW(comp, dz, dy, dx) v[(((comp) * VZ + ez + (dz)) * VY + ey + (dy)) * VX + ex + (dx)]
    zdf cc = dfwd_df(WW(0, 0, 0, 0), WW(0, 0, 0, 1), ih, kh0);
    cc = cdf_add(cc, dfwd_df(WW(1, 0, 0, 0), WW(1, 0, 1, 0), ih, kh1));
    cc = cdf_add(cc, dfwd_df(WW(2, 0, 0, 0), WW(2, 1, 0, 0), ih, kh2));
#undef WW
    c[eo] = cc;
  }
  __syncthreads();
  float sr = 0.f, sxx = 0.f;
  for (int i = threadIdx.x; i < TZ * TY * TX; i += blockDim.x) {
    const int lx = i % TX, ly = (i / TX) % TY, lz = i / (TX * TY);
#define EE(comp, dz, dy, dx) e[(((comp) * EZ + lz + (dz)) * EY + ly + (dy)) * EX + lx + (dx)]
#define CC(dz, dy, dx) c[((lz + 1 + (dz)) * EY + ly + 1 + (dy)) * EX + lx + 1 + (dx)]
    const zdf c0 = CC(0, 0, 0);
    const zdf e1 = EE(0, 0, 0, 0), e2 = EE(1, 0, 0, 0), e3 = EE(2, 0, 0, 0);
    zdf y1 = cdf_sub(dfwd_df(e3, EE(2, 0, 1, 0), ih, kh1), dfwd_df(e2, EE(1, 1, 0, 0), ih, kh2));
    y1 = cdf_add(y1, cdf_scale(dbwd_df(CC(0, 0, -1), c0, ih, kh0), gam));
    zdf y2 = cdf_sub(dfwd_df(e1, EE(0, 1, 0, 0), ih, kh2), dfwd_df(e3, EE(2, 0, 0, 1), ih, kh0));
    y2 = cdf_add(y2, cdf_scale(dbwd_df(CC(0, -1, 0), c0, ih, kh1), gam));
    zdf y3 = cdf_sub(dfwd_df(e2, EE(1, 0, 0, 1), ih, kh0), dfwd_df(e1, EE(0, 0, 1, 0), ih, kh1));
    y3 = cdf_add(y3, cdf_scale(dbwd_df(CC(-1, 0, 0), c0, ih, kh2), gam));
#undef EE
#undef CC
    const long gi = ((long)(z0 + lz) << (2 * logN)) + ((long)(y0 + ly) << logN) + x0 + lx;
    if constexpr (RES) {
#define XV(comp) v[(((comp) * VZ + lz + 1) * VY + ly + 1) * VX + lx + 1]
      const zdf yv[3] = {y1, y2, y3}, xv[3] = {XV(0), XV(1), XV(2)};
#undef XV
      resid_point(ra, b, j, n, gi, df_from(ra.theta[(long)b * ra.m + j]), yv, xv, sr, sxx);
    } else {
      st_cdf(Yb + gi, y1);
      st_cdf(Yb + n + gi, y2);
      st_cdf(Yb + 2 * n + gi, y3);
    }
  }
  if constexpr (RES) resid_block_sum(ra, sr, sxx);
}

template <int TX, int TY, int TZ, bool RES>
static int launch_op_df_t(pc_ctx *ctx, int nb, int m, const void *X, long sx, void *Y, long sy, const int *act,
                          const ResidArgs &ra, int *nchunk) {
  constexpr size_t smem = op_df_smem_bytes<TX, TY, TZ>();
  static bool configured = false;
  if (!configured) {
    PC_CK(cudaFuncSetAttribute(op_df_kernel<TX, TY, TZ, RES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)smem));
    configured = true;
  }
  const int N = ctx->N;
  dim3 grid((N / TX) * (N / TY) * (N / TZ), m, nb);
  *nchunk = (int)grid.x;
  if (RES && ra.part == nullptr) return PC_OK;  // sizing call
  op_df_kernel<TX, TY, TZ, RES><<<grid, 256, smem, ctx->stream>>>(
      static_cast<const df_store_t<RES> *>(X), sx, static_cast<df_store_t<RES> *>(Y), sy, ctx->m0p.as<float2>(),
      ctx->kparam.as<KParam>(), act, ctx->logN, ra);
  PC_CK_LAUNCH();
  return PC_OK;
}

// z-marching version (the blocking of opz_kernel in stencil.cu): a TX x TY column tile walks ZC planes with ring
// buffers of v (2 planes), e = M0 A' v (2 planes) and c = B v (2 planes).
template <int TX, int TY> constexpr size_t opz_df_smem_bytes() {
  return sizeof(zdf) * (size_t)(2 * 3 * (TY + 2) * (TX + 2) + 2 * 3 * (TY + 1) * (TX + 1) + 2 * (TY + 1) * (TX + 1));
}

template <int TX, int TY, bool RES>
__global__ void __launch_bounds__(TX * TY) opz_df_kernel(const df_store_t<RES> *__restrict__ X, long sx,
                                                         df_store_t<RES> *__restrict__ Y, long sy,
                                                         const float2 *__restrict__ m0,
                                                         const KParam *__restrict__ kp, const int *__restrict__ act,
                                                         int logN, int ZC, const ResidArgs ra) {
  using XS = df_store_t<RES>;
  constexpr int VX = TX + 2, VY = TY + 2, VP = VX * VY;
  constexpr int EX = TX + 1, EY = TY + 1, EP = EX * EY;
  constexpr int NT = TX * TY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  zdf *vbuf = reinterpret_cast<zdf *>(smem_raw);
  zdf *ebuf = vbuf + 2 * 3 * VP;
  zdf *cbuf = ebuf + 2 * 3 * EP;
  const int N = 1 << logN, mask = N - 1;
  const long n = 1L << (3 * logN), plane = 1L << (2 * logN);
  const int b = act ? act[blockIdx.z] : (int)blockIdx.z;
  const int j = blockIdx.y;
  const int tilesX = N / TX, tilesY = N / TY;
  int t = blockIdx.x;
  const int x0 = (t % tilesX) * TX;
  t /= tilesX;
  const int y0 = (t % tilesY) * TY;
  const int zb = (t / tilesY) * ZC;
  const XS *Xb = X + (long)b * sx + (long)j * 3 * n;
  XS *Yb = Y + (long)b * sy + (long)j * 3 * n;
  const KParam &p = kp[b];
  const kdf kh0 = kdf_of(p.khf[0], p.khl[0]), kh1 = kdf_of(p.khf[1], p.khl[1]), kh2 = kdf_of(p.khf[2], p.khl[2]);
  const df gam = kp_df(p.gammaf, p.gammal);
  const f32x2 ih = pack2((float)N, (float)N);
  const int tid = threadIdx.x;
  auto load_v = [&](int slot, int z) {
    const int gz = z & mask;
    zdf *vs = vbuf + slot * 3 * VP;
    for (int i = tid; i < 3 * VP; i += NT) {
      const int comp = i / VP, r = i - comp * VP, ly = r / VX, lx = r - ly * VX;
      const int gx = (x0 + lx - 1) & mask, gy = (y0 + ly - 1) & mask;
      vs[i] = ld_zdf(Xb + comp * n + gz * plane + ((long)gy << logN) + gx);
    }
  };
  auto make_e = [&](int eslot, int z, int sz, int szm) {
    const zdf *v0 = vbuf + sz * 3 * VP, *vm = vbuf + szm * 3 * VP;
    zdf *es = ebuf + eslot * 3 * EP;
    const int gz = z & mask;
    for (int i = tid; i < EP; i += NT) {
      const int ey = i / EX, ex = i - ey * EX;
      const int o = (ey + 1) * VX + ex + 1;
      const zdf v1 = v0[o], v2 = v0[VP + o], v3 = v0[2 * VP + o];
      const zdf d3v2 = dbwd_df(vm[VP + o], v2, ih, kh2);
      const zdf d2v3 = dbwd_df(v0[2 * VP + o - VX], v3, ih, kh1);
      const zdf d3v1 = dbwd_df(vm[o], v1, ih, kh2);
      const zdf d1v3 = dbwd_df(v0[2 * VP + o - 1], v3, ih, kh0);
      const zdf d2v1 = dbwd_df(v0[o - VX], v1, ih, kh1);
      const zdf d1v2 = dbwd_df(v0[VP + o - 1], v2, ih, kh0);
      const long gi = gz * plane + ((long)((y0 + ey) & mask) << logN) + ((x0 + ex) & mask);
      es[i] = cdf_scale(cdf_sub(d3v2, d2v3), ld_m0(m0 + gi));
      es[EP + i] = cdf_scale(cdf_sub(d1v3, d3v1), ld_m0(m0 + n + gi));
      es[2 * EP + i] = cdf_scale(cdf_sub(d2v1, d1v2), ld_m0(m0 + 2 * n + gi));
    }
  };
  auto make_c = [&](int cslot, int sz, int szp) {
    const zdf *v0 = vbuf + sz * 3 * VP, *vp = vbuf + szp * 3 * VP;
    zdf *cs = cbuf + cslot * EP;
    for (int i = tid; i < EP; i += NT) {
      const int cy = i / EX, cx = i - cy * EX;
      const int o = cy * VX + cx;
      zdf cc = dfwd_df(v0[o], v0[o + 1], ih, kh0);
      cc = cdf_add(cc, dfwd_df(v0[VP + o], v0[VP + o + VX], ih, kh1));
      cc = cdf_add(cc, dfwd_df(v0[2 * VP + o], vp[2 * VP + o], ih, kh2));
      cs[i] = cc;
    }
  };
  load_v(0, zb - 1);
  load_v(1, zb);
  __syncthreads();
  make_e(0, zb, 1, 0);
  make_c(0, 0, 1);
  int sv = 1, se = 0, sc = 0;
  float sr = 0.f, sxx = 0.f;
  const df th = RES ? df_from(ra.theta[(long)b * ra.m + j]) : df{0.f, 0.f};
  for (int z = zb; z < zb + ZC; ++z) {
    __syncthreads();
    load_v(1 - sv, z + 1);
    __syncthreads();
    make_e(1 - se, z + 1, 1 - sv, sv);
    make_c(1 - sc, sv, 1 - sv);
    __syncthreads();
    {
      const zdf *e0 = ebuf + se * 3 * EP, *e1p = ebuf + (1 - se) * 3 * EP;
      const zdf *cm = cbuf + sc * EP, *c0p = cbuf + (1 - sc) * EP;
      const int ly = tid / TX, lx = tid - ly * TX;
      const int eo = ly * EX + lx;
      const int co = (ly + 1) * EX + lx + 1;
      const zdf c0 = c0p[co];
      const zdf e1 = e0[eo], e2 = e0[EP + eo], e3 = e0[2 * EP + eo];
      zdf y1 = cdf_sub(dfwd_df(e3, e0[2 * EP + eo + EX], ih, kh1), dfwd_df(e2, e1p[EP + eo], ih, kh2));
      y1 = cdf_add(y1, cdf_scale(dbwd_df(c0p[co - 1], c0, ih, kh0), gam));
      zdf y2 = cdf_sub(dfwd_df(e1, e1p[eo], ih, kh2), dfwd_df(e3, e0[2 * EP + eo + 1], ih, kh0));
      y2 = cdf_add(y2, cdf_scale(dbwd_df(c0p[co - EX], c0, ih, kh1), gam));
      zdf y3 = cdf_sub(dfwd_df(e2, e0[EP + eo + 1], ih, kh0), dfwd_df(e1, e0[eo + EX], ih, kh1));
      y3 = cdf_add(y3, cdf_scale(dbwd_df(cm[co], c0, ih, kh2), gam));
      const long gi = (long)z * plane + ((long)(y0 + ly) << logN) + x0 + lx;
      if constexpr (RES) {
        const zdf *v0 = vbuf + sv * 3 * VP;  // plane z
        const int o = (ly + 1) * VX + lx + 1;
        const zdf yv[3] = {y1, y2, y3}, xv[3] = {v0[o], v0[VP + o], v0[2 * VP + o]};
        resid_point(ra, b, j, n, gi, th, yv, xv, sr, sxx);
      } else {
        st_cdf(Yb + gi, y1);
        st_cdf(Yb + n + gi, y2);
        st_cdf(Yb + 2 * n + gi, y3);
      }
    }
    sv = 1 - sv;
    se = 1 - se;
    sc = 1 - sc;
  }
  if constexpr (RES) resid_block_sum(ra, sr, sxx);
}

template <int TX, int TY, bool RES>
static int launch_opz_df_t(pc_ctx *ctx, int nb, int m, const void *X, long sx, void *Y, long sy, const int *act,
                           const ResidArgs &ra, int *nchunk) {
  constexpr size_t smem = opz_df_smem_bytes<TX, TY>();
  static bool configured = false;
  if (!configured) {
    PC_CK(cudaFuncSetAttribute(opz_df_kernel<TX, TY, RES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    configured = true;
  }
  const int N = ctx->N;
  const long tiles = (long)(N / TX) * (N / TY) * m * nb;
  int ZC = N;
  while (ZC > 4 && tiles * (N / ZC) < 16L * sm_count()) ZC >>= 1;
  dim3 grid((N / TX) * (N / TY) * (N / ZC), m, nb);
  *nchunk = (int)grid.x;
  if (RES && ra.part == nullptr) return PC_OK;  // sizing call
  opz_df_kernel<TX, TY, RES><<<grid, TX * TY, smem, ctx->stream>>>(
      static_cast<const df_store_t<RES> *>(X), sx, static_cast<df_store_t<RES> *>(Y), sy, ctx->m0p.as<float2>(),
      ctx->kparam.as<KParam>(), act, ctx->logN, ZC, ra);
  PC_CK_LAUNCH();
  return PC_OK;
}

// ---------------------------------------------------------------- general lattice (Section 4.2.2)
// D_hat_a f = sum_j (b_ja / h)(f_{r+e_j} - f_r) + i kh_a (f_r + f_{r+e_a}) and its adjoint
// D_hat_a' g = sum_j (b_ja / h)(g_{r-e_j} - g_r) - i kh_a (g_{r-e_a} + g_r), second order, in double-float; the
// weights b_ja / h are double-float pairs. Two passes through a per-stream scratch block (e = M0 A' v, c = B v as
// double-float pairs, then y = A e + gamma B' c), the second with the residual epilogue of the cubic kernels.
struct LatDF {
  df bh[9];  // bh[3 j + a] = b_ja N
};

__device__ __forceinline__ long lat_nb(long i, int axis, int off, int logN) {
  const int N = 1 << logN, mask = N - 1;
  int x = (int)(i & mask), y = (int)((i >> logN) & mask), z = (int)(i >> (2 * logN));
  if (axis == 0) x = (x + off) & mask;
  else if (axis == 1) y = (y + off) & mask;
  else z = (z + off) & mask;
  return ((long)z << (2 * logN)) + ((long)y << logN) + x;
}

// D_hat_a (adj = false) or D_hat_a' (adj = true) of field f at point i; f[...] read through ld_cdf
template <typename S>
__device__ __forceinline__ cdf dlat_df(const S *__restrict__ f, long i, int a, bool adj, int logN, const LatDF &lt,
                                       df kh) {
  const cdf f0 = ld_cdf(f + i);
  cdf acc = cdf{df{0.f, 0.f}, df{0.f, 0.f}}, sm = acc;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const cdf fj = ld_cdf(f + lat_nb(i, j, adj ? -1 : 1, logN));
    acc = cdf_add(acc, cdf_scale(cdf_sub(fj, f0), lt.bh[3 * j + a]));
    if (j == a) sm = cdf_add(fj, f0);
  }
  // acc + i kh sm (forward) or acc - i kh sm (adjoint)
  const df sr = df_mul(kh, sm.re), si = df_mul(kh, sm.im);
  return adj ? cdf{df_add(acc.re, si), df_sub(acc.im, sr)} : cdf{df_sub(acc.re, si), df_add(acc.im, sr)};
}

// pass 1: E (3 fields) and Cc (1 field) of column j of k-point act[bz], double-float pairs. grid (n / 256, m, nb)
template <typename XS>
__global__ void __launch_bounds__(256) lat_df_half_kernel(const XS *__restrict__ X, long sx, float4 *__restrict__ E,
                                                          const float2 *__restrict__ m0, const KParam *__restrict__ kp,
                                                          const int *__restrict__ act, int logN, const LatDF lt) {
  const long n = 1L << (3 * logN);
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int bz = blockIdx.z, j = blockIdx.y, m = gridDim.y;
  const int b = act ? act[bz] : bz;
  const KParam &p = kp[b];
  const df kh0 = kp_df(p.khf[0], p.khl[0]), kh1 = kp_df(p.khf[1], p.khl[1]), kh2 = kp_df(p.khf[2], p.khl[2]);
  const XS *v1 = X + (long)b * sx + (long)j * 3 * n, *v2 = v1 + n, *v3 = v2 + n;
  const cdf e1 = cdf_scale(cdf_sub(dlat_df(v2, i, 2, true, logN, lt, kh2), dlat_df(v3, i, 1, true, logN, lt, kh1)),
                           ld_m0(m0 + i));
  const cdf e2 = cdf_scale(cdf_sub(dlat_df(v3, i, 0, true, logN, lt, kh0), dlat_df(v1, i, 2, true, logN, lt, kh2)),
                           ld_m0(m0 + n + i));
  const cdf e3 = cdf_scale(cdf_sub(dlat_df(v1, i, 1, true, logN, lt, kh1), dlat_df(v2, i, 0, true, logN, lt, kh0)),
                           ld_m0(m0 + 2 * n + i));
  const cdf c = cdf_add(cdf_add(dlat_df(v1, i, 0, false, logN, lt, kh0), dlat_df(v2, i, 1, false, logN, lt, kh1)),
                        dlat_df(v3, i, 2, false, logN, lt, kh2));
  float4 *eb = E + ((long)bz * m + j) * 4 * n;
  st_cdf(eb + i, e1);
  st_cdf(eb + n + i, e2);
  st_cdf(eb + 2 * n + i, e3);
  st_cdf(eb + 3 * n + i, c);
}

// pass 2: y = A e + gamma B' c, stored (RES = false) or reduced to the residual epilogue (RES = true; every thread
// of the block takes part in its block sum). grid (n / 256, m, nb), 256 threads
template <bool RES>
__global__ void __launch_bounds__(256) lat_df_full_kernel(const float4 *__restrict__ E, const df_store_t<RES> *__restrict__ X,
                                                          long sx, df_store_t<RES> *__restrict__ Y, long sy,
                                                          const KParam *__restrict__ kp, const int *__restrict__ act,
                                                          int logN, const LatDF lt, const ResidArgs ra) {
  const long n = 1L << (3 * logN);
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const int bz = blockIdx.z, j = blockIdx.y, m = gridDim.y;
  const int b = act ? act[bz] : bz;
  const KParam &p = kp[b];
  float sr = 0.f, sxx = 0.f;
  if (i < n) {
    const df kh0 = kp_df(p.khf[0], p.khl[0]), kh1 = kp_df(p.khf[1], p.khl[1]), kh2 = kp_df(p.khf[2], p.khl[2]);
    const df gam = kp_df(p.gammaf, p.gammal);
    const float4 *e1 = E + ((long)bz * m + j) * 4 * n, *e2 = e1 + n, *e3 = e2 + n, *c = e3 + n;
    cdf y1 = cdf_sub(dlat_df(e3, i, 1, false, logN, lt, kh1), dlat_df(e2, i, 2, false, logN, lt, kh2));
    y1 = cdf_add(y1, cdf_scale(dlat_df(c, i, 0, true, logN, lt, kh0), gam));
    cdf y2 = cdf_sub(dlat_df(e1, i, 2, false, logN, lt, kh2), dlat_df(e3, i, 0, false, logN, lt, kh0));
    y2 = cdf_add(y2, cdf_scale(dlat_df(c, i, 1, true, logN, lt, kh1), gam));
    cdf y3 = cdf_sub(dlat_df(e2, i, 0, false, logN, lt, kh0), dlat_df(e1, i, 1, false, logN, lt, kh1));
    y3 = cdf_add(y3, cdf_scale(dlat_df(c, i, 2, true, logN, lt, kh2), gam));
    if constexpr (RES) {
      const df_store_t<RES> *xb = X + (long)b * sx + (long)j * 3 * n;
      const cdf yv[3] = {y1, y2, y3}, xv[3] = {ld_cdf(xb + i), ld_cdf(xb + n + i), ld_cdf(xb + 2 * n + i)};
      const df th = df_from(ra.theta[(long)b * ra.m + j]);
      resid_point(ra, b, j, n, i, th, yv, xv, sr, sxx);
    } else {
      df_store_t<RES> *yb = Y + (long)b * sy + (long)j * 3 * n;
      st_cdf(yb + i, y1);
      st_cdf(yb + n + i, y2);
      st_cdf(yb + 2 * n + i, y3);
    }
  }
  if constexpr (RES) resid_block_sum(ra, sr, sxx);
}

template <bool RES>
int launch_op_df_lat(pc_ctx *ctx, int nb, int m, const void *X, long sx, void *Y, long sy, const int *act,
                     const ResidArgs &ra, int *nchunk) {
  const long n = ctx->n;
  const dim3 grid((unsigned)((n + 255) / 256), m, nb);
  *nchunk = (int)grid.x;
  if (RES && ra.part == nullptr) return PC_OK;  // sizing call
  LatDF lt;
  for (int q = 0; q < 9; ++q) {
    const double v = ctx->binv[q] * (double)ctx->N;
    lt.bh[q].hi = (float)v;
    lt.bh[q].lo = (float)(v - (double)lt.bh[q].hi);
  }
  DevBuf &ks = kscratch_for(ctx);
  PC_CK(ks.reserve(sizeof(float4) * 4 * (size_t)n * m * nb));
  float4 *E = ks.as<float4>();
  using XS = df_store_t<RES>;
  lat_df_half_kernel<XS><<<grid, 256, 0, ctx->stream>>>(static_cast<const XS *>(X), sx, E, ctx->m0p.as<float2>(),
                                                         ctx->kparam.as<KParam>(), act, ctx->logN, lt);
  PC_CK_LAUNCH();
  lat_df_full_kernel<RES><<<grid, 256, 0, ctx->stream>>>(E, static_cast<const XS *>(X), sx, static_cast<XS *>(Y), sy,
                                                          ctx->kparam.as<KParam>(), act, ctx->logN, lt, ra);
  PC_CK_LAUNCH();
  return PC_OK;
}

template <bool RES>
static int op_df_dispatch(pc_ctx *ctx, int nb, int m, const void *X, long sx, void *Y, long sy, const int *act,
                          const ResidArgs &ra, int *nchunk) {
  if (ctx->lat) return launch_op_df_lat<RES>(ctx, nb, m, X, sx, Y, sy, act, ra, nchunk);
  const int N = ctx->N;
  if (N >= 32) return launch_opz_df_t<32, 8, RES>(ctx, nb, m, X, sx, Y, sy, act, ra, nchunk);
  if (N == 16) return launch_op_df_t<16, 4, 4, RES>(ctx, nb, m, X, sx, Y, sy, act, ra, nchunk);
  return launch_op_df_t<8, 4, 4, RES>(ctx, nb, m, X, sx, Y, sy, act, ra, nchunk);
}

int launch_apply_op_df(pc_ctx *ctx, int nb, int m, const void *X, long sx, void *Y, long sy, const int *act) {
  if (nb == 0 || m == 0) return PC_OK;
  if (ctx->opts.order != 1) {
    set_error("double-float stencil: second order (order 1) only");
    return PC_EUNSUPPORTED;
  }
  int nchunk = 0;
  return op_df_dispatch<false>(ctx, nb, m, X, sx, Y, sy, act, ResidArgs{}, &nchunk);
}

size_t op_df_resid_scratch_bytes(pc_ctx *ctx, int nb, int m) {
  int nchunk = 0;
  op_df_dispatch<true>(ctx, nb, m, nullptr, 0, nullptr, 0, nullptr, ResidArgs{}, &nchunk);
  return sizeof(double) * 2 * (size_t)nb * m * nchunk;
}

int launch_op_df_resid(pc_ctx *ctx, int nb, int m, const void *X, long sx, const double *theta, void *R1, long sr1,
                       void *R2, long sr2, void *X32, long sx32, void *AX32, long sax32, double *norms, void *scratch,
                       size_t scratch_bytes, const int *act) {
  if (nb == 0 || m == 0) return PC_OK;
  if (op_df_resid_scratch_bytes(ctx, nb, m) > scratch_bytes) {
    set_error("op_df_resid: scratch too small");
    return PC_EINVAL;
  }
  ResidArgs ra{theta, m, static_cast<float2 *>(R1), static_cast<float2 *>(R2), static_cast<float2 *>(X32),
               static_cast<float2 *>(AX32), sr1, sr2, sx32, sax32, static_cast<double *>(scratch)};
  int nchunk = 0;
  int rc = op_df_dispatch<true>(ctx, nb, m, X, sx, nullptr, 0, act, ra, &nchunk);
  if (rc) return rc;
  launch_residual_reduce(nb, nchunk, m, static_cast<const double *>(scratch), act, norms, ctx->stream);
  PC_CK_LAUNCH();
  return PC_OK;
}

// ---------------------------------------------------------------- block update Y = X C + Z
// On the tensor cores (update_sl.cu).
int launch_update_df(int nb, long L, int p, int q, const void *X, long sx, const void *C, long sc, void *Y, long sy,
                     const void *Z, long sz, cudaStream_t st, int *tmo, const int *act) {
  if (nb == 0 || q == 0) return PC_OK;
  if (p < 1 || p > 32) {
    set_error("update_df: 1 to 32 input columns");
    return PC_EINVAL;
  }
  return launch_update_sl(nb, L, p, q, PC_DFS, X, sx, C, sc, Y, sy, Z, sz, st, tmo, act);
}

// ---------------------------------------------------------------- Gram G = X^H X of the FP64 block
// (X^H AX is not formed here: the mixed solve takes it as Theta X^H X + R^H X, R = AX - X Theta.)
// On the tensor cores (gram_sl.cu).
size_t gram_df_scratch_bytes(int nb, long L, int p) {
  return sizeof(double2) * (size_t)nb * sl_gram_chunks(nb, L) * p * p;
}

int launch_gram_df(int nb, long L, int p, const void *X, long sx, void *G, void *scratch, size_t scratch_bytes,
                   cudaStream_t st, int *tmo, const int *act) {
  if (nb == 0 || p == 0) return PC_OK;
  if (p > 32 || gram_df_scratch_bytes(nb, L, p) > scratch_bytes) {
    set_error("gram_df: at most 32 columns and enough scratch");
    return PC_EINVAL;
  }
  double2 *part = static_cast<double2 *>(scratch);
  int nchunk = 0;
  const int rc = launch_gram_sl(nb, L, p, p, PC_DFS, X, sx, X, sx, SL_SELF, part, sl_gram_chunks(nb, L), &nchunk, st,
                                tmo, act);
  if (rc) return rc;
  launch_gram_self_reduce(nb, nchunk, p, part, act, G, st);
  PC_CK_LAUNCH();
  return PC_OK;
}

}  // namespace pc
