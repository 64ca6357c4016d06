// Kernels of the nonlinear compressed-sensing path (Sec. 2.2.5 with an
// L1-wavelet FISTA reconstruction): periodised orthonormal 2-D DWT passes,
// the element-wise FISTA steps, the complex soft threshold and its R-linear
// tangent, the reverse-sweep updates of the VJP, and the 2-D-mask helpers of
// the forward / adjoint encoding operator.
#include "common.cuh"
#include "kernels.cuh"

namespace pico {

namespace {

inline unsigned blocks(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// ---- DWT passes on the top-left nyl x nxl region of n-strided images ----
// analysis along rows: a[k] = sum_m h[m] x[(2k+m) mod nxl], d[k] = sum_m g[m] x[...]; [a | d]
__global__ void k_dwt_rows_fwd(const float2* __restrict__ in, float2* __restrict__ out, int n, int nyl, int nxl,
                               int64_t img, Wavelet w) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int half = nxl / 2;
  if (t >= (int64_t)nyl * half) return;
  const int y = (int)(t / half), k = (int)(t % half);
  const float2* row = in + (size_t)blockIdx.y * img + (size_t)y * n;
  float2 a = make_float2(0.f, 0.f), d = a;
  for (int m = 0; m < w.L; ++m) {
    int j = 2 * k + m;
    while (j >= nxl) j -= nxl;   // sides shorter than the filter wrap more than once
    const float2 v = row[j];
    a.x = fmaf(w.h[m], v.x, a.x);
    a.y = fmaf(w.h[m], v.y, a.y);
    d.x = fmaf(w.g[m], v.x, d.x);
    d.y = fmaf(w.g[m], v.y, d.y);
  }
  float2* o = out + (size_t)blockIdx.y * img + (size_t)y * n;
  o[k] = a;
  o[half + k] = d;
}

__global__ void k_dwt_cols_fwd(const float2* __restrict__ in, float2* __restrict__ out, int n, int nyl, int nxl,
                               int64_t img, Wavelet w) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int half = nyl / 2;
  if (t >= (int64_t)half * nxl) return;
  const int k = (int)(t / nxl), x = (int)(t % nxl);
  const float2* base = in + (size_t)blockIdx.y * img + x;
  float2 a = make_float2(0.f, 0.f), d = a;
  for (int m = 0; m < w.L; ++m) {
    int j = 2 * k + m;
    while (j >= nyl) j -= nyl;
    const float2 v = base[(size_t)j * n];
    a.x = fmaf(w.h[m], v.x, a.x);
    a.y = fmaf(w.h[m], v.y, a.y);
    d.x = fmaf(w.g[m], v.x, d.x);
    d.y = fmaf(w.g[m], v.y, d.y);
  }
  float2* o = out + (size_t)blockIdx.y * img + x;
  o[(size_t)k * n] = a;
  o[(size_t)(half + k) * n] = d;
}

// synthesis (transpose of the analysis): x[i] = sum over taps m with (i - m) even of
// h[m] a[k] + g[m] d[k], k = ((i - m) mod len) / 2  (gather form, no atomics)
__global__ void k_dwt_rows_inv(const float2* __restrict__ in, float2* __restrict__ out, int n, int nyl, int nxl,
                               int64_t img, Wavelet w) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)nyl * nxl) return;
  const int y = (int)(t / nxl), i = (int)(t % nxl);
  const int half = nxl / 2;
  const float2* row = in + (size_t)blockIdx.y * img + (size_t)y * n;
  float2 acc = make_float2(0.f, 0.f);
  for (int m = (i & 1); m < w.L; m += 2) {
    int j = i - m;
    while (j < 0) j += nxl;
    const int k = j / 2;
    const float2 a = row[k], d = row[half + k];
    acc.x = fmaf(w.h[m], a.x, fmaf(w.g[m], d.x, acc.x));
    acc.y = fmaf(w.h[m], a.y, fmaf(w.g[m], d.y, acc.y));
  }
  out[(size_t)blockIdx.y * img + (size_t)y * n + i] = acc;
}

__global__ void k_dwt_cols_inv(const float2* __restrict__ in, float2* __restrict__ out, int n, int nyl, int nxl,
                               int64_t img, Wavelet w) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)nyl * nxl) return;
  const int i = (int)(t / nxl), x = (int)(t % nxl);
  const int half = nyl / 2;
  const float2* base = in + (size_t)blockIdx.y * img + x;
  float2 acc = make_float2(0.f, 0.f);
  for (int m = (i & 1); m < w.L; m += 2) {
    int j = i - m;
    while (j < 0) j += nyl;
    const int k = j / 2;
    const float2 a = base[(size_t)k * n], d = base[(size_t)(half + k) * n];
    acc.x = fmaf(w.h[m], a.x, fmaf(w.g[m], d.x, acc.x));
    acc.y = fmaf(w.h[m], a.y, fmaf(w.g[m], d.y, acc.y));
  }
  out[(size_t)blockIdx.y * img + (size_t)i * n + x] = acc;
}

__global__ void k_copy_region(const float2* __restrict__ in, float2* __restrict__ out, int n, int nyl, int nxl,
                              int64_t img) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)nyl * nxl) return;
  const int y = (int)(t / nxl), x = (int)(t % nxl);
  const size_t o = (size_t)blockIdx.y * img + (size_t)y * n + x;
  out[o] = in[o];
}

// ---- element-wise FISTA / Jacobian steps (image index i, batch b = blockIdx.y) ----
// |c|, the one rounding order written out so that every kernel that inlines it agrees
__device__ __forceinline__ float cs_abs(float2 c) { return sqrtf(fmaf(c.x, c.x, __fmul_rn(c.y, c.y))); }
__device__ __forceinline__ float2 soft1(float2 c, float tau) {
  const float a = cs_abs(c);
  if (!(a > tau)) return make_float2(0.f, 0.f);
  return cscale(c, 1.f - tau / a);
}
__device__ __forceinline__ float2 soft_tan1(float2 c, float tau, float2 dc) {
  const float a = cs_abs(c);
  if (!(a > tau)) return make_float2(0.f, 0.f);
  const float2 u = cscale(c, 1.f / a);
  const float re = cdot_re(u, dc);  // Re(conj(u) dc)
  const float s = 1.f - tau / a, q = (tau / a) * re;
  return make_float2(fmaf(s, dc.x, q * u.x), fmaf(s, dc.y, q * u.y));
}

// The element-wise steps as passes of their own: for transforms whose last
// levels are shorter than the filter (cs_fused_supported).
// y = z - (Mz - rhs) / Lc ; rhs broadcast when rhs_stride == 0
__global__ void k_cs_gradstep(const float2* __restrict__ z, const float2* __restrict__ Mz,
                              const float2* __restrict__ rhs, int64_t rhs_stride, float inv_lc, float2* __restrict__ y,
                              int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  const float2 r = rhs ? rhs[(size_t)blockIdx.y * rhs_stride + i] : make_float2(0.f, 0.f);
  const float2 zz = z[o], mz = Mz[o];
  y[o] = make_float2(fmaf(-inv_lc, mz.x - r.x, zz.x), fmaf(-inv_lc, mz.y - r.y, zz.y));
}

// primal: threshold the coefficients (batch b = blockIdx.y); `keep` (one image) stores them
// as the linearisation point of the Jacobian
__global__ void k_cs_soft(const float2* c, float2* __restrict__ keep, float2* out, float tau, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  const float2 v = c[o];
  if (keep) keep[i] = v;
  out[o] = soft1(v, tau);
}

// tangent of the soft threshold at the stored coefficients (broadcast over the batch), in place
__global__ void k_cs_soft_tan(const float2* __restrict__ at, float2* __restrict__ dc, float tau, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  dc[o] = soft_tan1(at[i], tau, dc[o]);
}

// z = xn + c (xn - x); x = xn
__global__ void k_cs_momentum(const float2* __restrict__ xn, float2* __restrict__ x, float2* __restrict__ z, float c,
                              int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  const float2 a = xn[o], b = x[o];
  z[o] = make_float2(fmaf(c, a.x - b.x, a.x), fmaf(c, a.y - b.y, a.y));
  x[o] = a;
}

// reverse sweep, first half: xk1 = xbn + (1 + c) zb ; xbn = -c zb
__global__ void k_vjp_a(float2* __restrict__ xbn, const float2* __restrict__ zb, float2* __restrict__ xk1, float c,
                        int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  const float2 z = zb[o], xb = xbn[o];
  xk1[o] = make_float2(fmaf(1.f + c, z.x, xb.x), fmaf(1.f + c, z.y, xb.y));
  xbn[o] = make_float2(-c * z.x, -c * z.y);
}

// reverse sweep, second half: zb = yb - M yb / Lc ; ysum += yb
__global__ void k_vjp_b(const float2* __restrict__ yb, const float2* __restrict__ Myb, float inv_lc,
                        float2* __restrict__ zb, float2* __restrict__ ysum, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  const float2 y = yb[o], m = Myb[o];
  zb[o] = make_float2(fmaf(-inv_lc, m.x, y.x), fmaf(-inv_lc, m.y, y.y));
  const float2 s = ysum[o];
  ysum[o] = make_float2(s.x + y.x, s.y + y.y);
}

// x[b] += alpha y (y one image, broadcast over the batch)
__global__ void k_axpy_bcast(float2* __restrict__ x, const float2* __restrict__ y, float alpha, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  const float2 a = x[o], b = y[i];
  x[o] = make_float2(fmaf(alpha, b.x, a.x), fmaf(alpha, b.y, a.y));
}

// ---------------------------------------------------------------------------
// One FISTA / tangent / adjoint iteration around the normal operator, fused:
//   cs_fwd    (level 0)  iteration step on load, 2-D analysis, threshold of the finished coefficients
//   cs_fwd    (level l)  2-D analysis of the approximation band, threshold
//   cs_core              the remaining levels of one image in shared memory: analysis, threshold, synthesis
//   cs_inv    (level l)  2-D synthesis
//   cs_inv    (level 0)  2-D synthesis, iteration step on store
// instead of one launch per direction and level and one per element-wise step:
// 5 launches per iteration of a 4-level transform at 320 x 320 in place of
// 19-20, the images cross memory once per level and direction instead of twice,
// and the element-wise steps take no pass of their own (320 x 320, an iteration
// without its normal operator: 48 images 367 us as single passes, 164 us fused; one
// image 84 and 42 us).  The arithmetic of every value is that of the single passes
// (rows before columns in the analysis, columns before rows in the synthesis, taps
// in the same order).  Bound by shared memory, local memory (the synthesis taps
// below) and the loads of the level-0 kernels for many images, by the latency of
// each launch for one.
// ---------------------------------------------------------------------------
constexpr int kTapMax = 8;
// Coefficients per tile and band.  8 rows (halo 1.5x, 24 KB of shared memory per
// block) rather than 16 (1.3x, 41 KB): more and smaller blocks per SM outweigh the
// halo for every size and batch tried (wavelet kernels of one iteration, 320 x 320:
// 96 images 254 against 286 us, 4 images 41 against 50 us; 64 x 64, 512 images 68
// against 73 us).
constexpr int kFuseTX = 32, kFuseTY = 8;
constexpr int kFuseThreads = 256;
constexpr int kLoadAhead = 6;      // global loads in flight per thread and operand

struct FwdArgs {
  int n, m;                        // image side, side of this level's input region
  const float2 *a, *b, *c;         // load operands (see cs_load)
  int64_t c_stride;                // image stride of c (0: one image for the whole batch)
  float s0, s1, s2;
  float2* zout;                    // kLoadVjp: the new z, stored by the tile that owns the pixel
  float2* dst;
  const float2* at;                // threshold tangent: stored coefficients (one image)
  float2* keep;                    // primal: raw coefficients kept (one image), or nullptr
  float tau;
  int last;                        // the approximation band is finished too
};
enum { kLoadGrad, kLoadVjp, kLoadPlain };

// kLoadGrad:  a - (b - c) s0            (y = z - (M z - rhs) / Lc)
// kLoadVjp:   z = a - b s0 (0 if !a);  c' = a ? -s2 c : c;  c' + s1 z
//             (reverse sweep: zb = yb - M yb / Lc, xk = xb + (1 + c_k) zb with xb = -c_{k+1} zb_prev)
template <int LOAD>
__device__ __forceinline__ float2 cs_load(const FwdArgs& f, size_t o, size_t i, int b, float2& z) {
  if (LOAD == kLoadPlain) return f.a[o];
  if (LOAD == kLoadGrad) {
    const float2 zz = f.a[o], mz = f.b[o], r = f.c[(size_t)b * f.c_stride + i];
    return make_float2(fmaf(-f.s0, mz.x - r.x, zz.x), fmaf(-f.s0, mz.y - r.y, zz.y));
  }
  float2 xb = f.c[o];
  z = make_float2(0.f, 0.f);
  if (f.a) {
    const float2 y = f.a[o], my = f.b[o];
    z = make_float2(fmaf(-f.s0, my.x, y.x), fmaf(-f.s0, my.y, y.y));
    xb = make_float2(-f.s2 * xb.x, -f.s2 * xb.y);
  }
  return make_float2(fmaf(f.s1, z.x, xb.x), fmaf(f.s1, z.y, xb.y));
}

template <bool TAN>
__device__ __forceinline__ float2 cs_threshold(float2 v, size_t i, const float2* at, float2* keep, float tau) {
  if (TAN) return soft_tan1(at[i], tau, v);
  if (keep) keep[i] = v;
  return soft1(v, tau);
}

// One analysis level on tiles of kFuseTY x kFuseTX coefficients per band.
template <int LOAD, bool TAN>
__global__ void __launch_bounds__(kFuseThreads) k_cs_fwd(FwdArgs f, Wavelet w) {
  constexpr int TX = kFuseTX, TY = kFuseTY, IY = 2 * TY + kTapMax - 2, IX = 2 * TX + kTapMax - 2;
  __shared__ __align__(16) float2 in[IY][IX];
  __shared__ float2 mid[IY][2 * TX];   // row analysis: [approximation | detail]
  const int t = threadIdx.x, b = blockIdx.z, n = f.n, m = f.m, half = m / 2;
  const int kx0 = blockIdx.x * TX, ky0 = blockIdx.y * TY;
  const size_t img = (size_t)b * n * n;
  // kLoadAhead values per thread are requested before the first is used: the
  // loads, not the transforms, are the time of a launch of few tiles
  for (int e0 = t; e0 < IY * IX; e0 += kLoadAhead * kFuseThreads) {
    float2 v[kLoadAhead], z[kLoadAhead];
#pragma unroll
    for (int u = 0; u < kLoadAhead; ++u) {
      const int e = min(e0 + u * kFuseThreads, IY * IX - 1), r = e / IX, q = e - r * IX;
      // the last tile's overhang beyond the periodic halo is loaded from a valid place and not used
      int y = 2 * ky0 + r, x = 2 * kx0 + q;
      if (y >= m) y -= m;
      if (x >= m) x -= m;
      const size_t i = (size_t)min(y, m - 1) * n + min(x, m - 1);
      v[u] = cs_load<LOAD>(f, img + i, i, b, z[u]);
    }
#pragma unroll
    for (int u = 0; u < kLoadAhead; ++u) {
      const int e = e0 + u * kFuseThreads, r = e / IX, q = e - r * IX;
      if (e >= IY * IX) break;
      in[r][q] = v[u];
      if (LOAD == kLoadVjp) {
        const int y = 2 * ky0 + r, x = 2 * kx0 + q;
        if (r < 2 * TY && q < 2 * TX && y < m && x < m) f.zout[img + (size_t)y * n + x] = z[u];
      }
    }
  }
  __syncthreads();
  for (int e = t; e < IY * TX; e += kFuseThreads) {
    const int r = e / TX, k = e - r * TX;
    float2 a = make_float2(0.f, 0.f), d = a;
#pragma unroll
    for (int q = 0; q < kTapMax; q += 2) {   // two values per access: no bank conflicts
      const float4 v = *reinterpret_cast<const float4*>(&in[r][2 * k + q]);
      a.x = fmaf(w.h[q], v.x, a.x);
      a.y = fmaf(w.h[q], v.y, a.y);
      d.x = fmaf(w.g[q], v.x, d.x);
      d.y = fmaf(w.g[q], v.y, d.y);
      a.x = fmaf(w.h[q + 1], v.z, a.x);
      a.y = fmaf(w.h[q + 1], v.w, a.y);
      d.x = fmaf(w.g[q + 1], v.z, d.x);
      d.y = fmaf(w.g[q + 1], v.w, d.y);
    }
    mid[r][k] = a;
    mid[r][TX + k] = d;
  }
  __syncthreads();
  for (int e = t; e < TY * 2 * TX; e += kFuseThreads) {
    const int k = e / (2 * TX), q0 = e - k * (2 * TX);
    const int ky = ky0 + k, kx = kx0 + (q0 & (TX - 1)), band = q0 >= TX;
    if (ky >= half || kx >= half) continue;
    float2 a = make_float2(0.f, 0.f), d = a;
#pragma unroll
    for (int q = 0; q < kTapMax; ++q) {
      const float2 v = mid[2 * k + q][q0];
      a.x = fmaf(w.h[q], v.x, a.x);
      a.y = fmaf(w.h[q], v.y, a.y);
      d.x = fmaf(w.g[q], v.x, d.x);
      d.y = fmaf(w.g[q], v.y, d.y);
    }
    const size_t ia = (size_t)ky * n + kx + band * half, id = ia + (size_t)half * n;
    f.dst[img + ia] = (band || f.last) ? cs_threshold<TAN>(a, ia, f.at, f.keep, f.tau) : a;
    f.dst[img + id] = cs_threshold<TAN>(d, id, f.at, f.keep, f.tau);
  }
}

struct InvArgs {
  int n, m;
  const float2* src;   // all bands of the level, [m][m] of an n-strided image
  float2 *o0, *o1;     // plain: o0 (n-strided); step: see cs_store
  float c;
};
enum { kStorePlain, kStoreMomentum, kStoreVjp };

// kStoreMomentum: z = v + c (v - x); x = v       (o0 = x, o1 = z)
// kStoreVjp:      yb = v; ysum += v              (o0 = yb, o1 = ysum)
template <int STORE>
__device__ __forceinline__ void cs_store(const InvArgs& f, size_t o, float2 v) {
  if (STORE == kStoreMomentum) {
    const float2 x = f.o0[o];
    f.o1[o] = make_float2(fmaf(f.c, v.x - x.x, v.x), fmaf(f.c, v.y - x.y, v.y));
  } else if (STORE == kStoreVjp) {
    const float2 s = f.o1[o];
    f.o1[o] = make_float2(s.x + v.x, s.y + v.y);
  }
  f.o0[o] = v;
}

// One synthesis level on tiles of 2 kFuseTY x 2 kFuseTX outputs.  The tap of an output
// depends on its parity, so the filters are indexed at run time: the compiler keeps
// a copy of them in local memory (72 bytes of stack) and each tap is a load from there.
template <int STORE>
__global__ void __launch_bounds__(kFuseThreads) k_cs_inv(InvArgs f, Wavelet w) {
  constexpr int TX = kFuseTX, TY = kFuseTY, HB = kTapMax / 2 - 1, CY = TY + HB, CX = TX + HB;
  __shared__ float2 in[2][CY][2 * CX];     // [rows: approximation | detail][k][columns: approximation | detail]
  __shared__ float2 mid[2 * TY][2 * CX];   // column synthesis
  const int t = threadIdx.x, b = blockIdx.z, n = f.n, m = f.m, half = m / 2;
  const int kx0 = blockIdx.x * TX, ky0 = blockIdx.y * TY;   // first own coefficient of the tile
  const size_t img = (size_t)b * n * n;
  for (int e0 = t; e0 < 2 * CY * 2 * CX; e0 += kLoadAhead * kFuseThreads) {
    float2 v[kLoadAhead];
#pragma unroll
    for (int u = 0; u < kLoadAhead; ++u) {
      const int e = min(e0 + u * kFuseThreads, 2 * CY * 2 * CX - 1);
      const int hy = e / (CY * 2 * CX), r = (e / (2 * CX)) % CY, q = e % (2 * CX), hx = q >= CX;
      int ky = ky0 + r - HB, kx = kx0 + (q - hx * CX) - HB;
      if (ky < 0) ky += half;
      if (kx < 0) kx += half;
      v[u] = f.src[img + (size_t)(min(ky, half - 1) + hy * half) * n + min(kx, half - 1) + hx * half];
    }
#pragma unroll
    for (int u = 0; u < kLoadAhead; ++u) {
      const int e = e0 + u * kFuseThreads;
      if (e < 2 * CY * 2 * CX) (&in[0][0][0])[e] = v[u];
    }
  }
  __syncthreads();
  for (int e = t; e < 2 * TY * 2 * CX; e += kFuseThreads) {
    const int i = e / (2 * CX), q = e - i * (2 * CX);
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kTapMax / 2; ++u) {   // tap q0 = 2 u + (i & 1), coefficient (i - q0) / 2
      const int tap = 2 * u + (i & 1), k = (i >> 1) - u + HB;
      const float2 a = in[0][k][q], d = in[1][k][q];
      acc.x = fmaf(w.h[tap], a.x, fmaf(w.g[tap], d.x, acc.x));
      acc.y = fmaf(w.h[tap], a.y, fmaf(w.g[tap], d.y, acc.y));
    }
    mid[i][q] = acc;
  }
  __syncthreads();
  for (int e = t; e < 2 * TY * 2 * TX; e += kFuseThreads) {
    const int r = e / (2 * TX), i = e - r * (2 * TX);
    const int y = 2 * ky0 + r, x = 2 * kx0 + i;
    if (y >= m || x >= m) continue;
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kTapMax / 2; ++u) {
      const int tap = 2 * u + (i & 1), k = (i >> 1) - u + HB;
      const float2 a = mid[r][k], d = mid[r][CX + k];
      acc.x = fmaf(w.h[tap], a.x, fmaf(w.g[tap], d.x, acc.x));
      acc.y = fmaf(w.h[tap], a.y, fmaf(w.g[tap], d.y, acc.y));
    }
    cs_store<STORE>(f, img + (size_t)y * n + x, acc);
  }
}

// The last levels of one image (side m at the first of them, at most kCoreSide)
// in shared memory: each pass reads one buffer and writes the other, rows with
// consecutive lanes along the row, columns with consecutive lanes across them.
// A latency-bound chain of 4 passes per level: 1024 threads, one (approximation,
// detail) pair or one sample each and a barrier per pass.
// kCoreSide 96 against 48 (one more level as tiled launches, the core 19 -> 7 us for
// one 320 x 320 image): kernel time of an iteration 37 -> 33 us for one image, equal
// for 48, 4 % more for 64 of 128 x 128 -- but two more launches, and whole calls are slower:
// reconstruction of one 320 x 320 image 7.84 against 8.04 ms, Jacobian map of 48
// probes 160.5 against 161.4 ms, 40 replicas at 256 x 256 equal within 0.4 %.
constexpr int kCoreSide = 96;
constexpr int kCoreThreads = 1024;

// taps along a line of `len` values (value x at p[x * st]): coefficient pair k
__device__ __forceinline__ void core_pair(const float2* p, int st, int k, int len, const Wavelet& w, float2& oa,
                                          float2& od) {
  float2 a = make_float2(0.f, 0.f), d = a;
#pragma unroll
  for (int q = 0; q < kTapMax; ++q) {
    int x = 2 * k + q;
    if (x >= len) x -= len;
    const float2 v = p[x * st];
    a.x = fmaf(w.h[q], v.x, a.x);
    a.y = fmaf(w.h[q], v.y, a.y);
    d.x = fmaf(w.g[q], v.x, d.x);
    d.y = fmaf(w.g[q], v.y, d.y);
  }
  oa = a;
  od = d;
}
// samples 2 j and 2 j + 1 of a line from its [approximation | detail]
__device__ __forceinline__ void core_samples(const float2* p, int st, int j, int half, const Wavelet& w, float2& oe,
                                             float2& oo) {
  float2 e = make_float2(0.f, 0.f), o = e;
#pragma unroll
  for (int u = 0; u < kTapMax / 2; ++u) {
    int k = j - u;
    if (k < 0) k += half;
    const float2 a = p[k * st], d = p[(half + k) * st];
    e.x = fmaf(w.h[2 * u], a.x, fmaf(w.g[2 * u], d.x, e.x));
    e.y = fmaf(w.h[2 * u], a.y, fmaf(w.g[2 * u], d.y, e.y));
    o.x = fmaf(w.h[2 * u + 1], a.x, fmaf(w.g[2 * u + 1], d.x, o.x));
    o.y = fmaf(w.h[2 * u + 1], a.y, fmaf(w.g[2 * u + 1], d.y, o.y));
  }
  oe = e;
  oo = o;
}

template <bool TAN>
__global__ void __launch_bounds__(kCoreThreads) k_cs_core(float2* data, int n, int m, int levels, const float2* at,
                                                          float2* keep, float tau, Wavelet w) {
  extern __shared__ float2 core[];
  float2 *A = core, *B = core + m * m;
  float2* img = data + (size_t)blockIdx.x * n * n;
  const int t = threadIdx.x;
  constexpr int U = kCoreSide * kCoreSide / kCoreThreads;   // values per thread
  {
    float2 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = min(t + u * kCoreThreads, m * m - 1);
      v[u] = img[(size_t)(e / m) * n + e % m];
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (t + u * kCoreThreads < m * m) A[t + u * kCoreThreads] = v[u];
  }
  __syncthreads();
  for (int l = 0; l < levels; ++l) {
    const int s = m >> l, half = s / 2;
    for (int e = t; e < s * half; e += kCoreThreads) {
      const int y = e / half, k = e - y * half;
      core_pair(A + y * m, 1, k, s, w, B[y * m + k], B[y * m + half + k]);
    }
    __syncthreads();
    for (int e = t; e < s * half; e += kCoreThreads) {
      const int k = e / s, x = e - k * s;
      core_pair(B + x, m, k, s, w, A[k * m + x], A[(half + k) * m + x]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int e = t + u * kCoreThreads;
    if (e < m * m) A[e] = cs_threshold<TAN>(A[e], (size_t)(e / m) * n + e % m, at, keep, tau);
  }
  __syncthreads();
  for (int l = levels - 1; l >= 0; --l) {
    const int s = m >> l, half = s / 2;
    for (int e = t; e < s * half; e += kCoreThreads) {
      const int j = e / s, x = e - j * s;
      core_samples(A + x, m, j, half, w, B[2 * j * m + x], B[(2 * j + 1) * m + x]);
    }
    __syncthreads();
    for (int e = t; e < s * half; e += kCoreThreads) {
      const int y = e / half, j = e - y * half;
      core_samples(B + y * m, 1, j, half, w, A[y * m + 2 * j], A[y * m + 2 * j + 1]);
    }
    __syncthreads();
  }
  for (int e = t; e < m * m; e += kCoreThreads) img[(size_t)(e / m) * n + e % m] = A[e];
}

inline dim3 level_tiles(int m, int nb) {
  return dim3((m / 2 + kFuseTX - 1) / kFuseTX, (m / 2 + kFuseTY - 1) / kFuseTY, nb);
}

// Coefficients of y (from cs_load<LOAD>) thresholded and transformed back:
// analysis level 0 from the load operands into b0, further levels alternating
// between b1 and b0, the small levels in place, synthesis up to level 1.
// The thresholded level-0 bands end in b0.
template <int LOAD, bool TAN>
void cs_shrink(FwdArgs f, float2* b0, float2* b1, int levels, int nb, const Wavelet& w, cudaStream_t s) {
  const int n = f.n;
  float2* buf[2] = {b0, b1};
  int l0 = 1;   // first level of the in-memory core
  while (l0 < levels && (n >> l0) > kCoreSide) ++l0;
  f.m = n;
  f.dst = b0;
  f.last = levels == 1;
  k_cs_fwd<LOAD, TAN><<<level_tiles(f.m, nb), kFuseThreads, 0, s>>>(f, w);
  for (int l = 1; l < l0; ++l) {
    f.a = buf[(l - 1) & 1];
    f.dst = buf[l & 1];
    f.m = n >> l;
    f.last = l == levels - 1;
    k_cs_fwd<kLoadPlain, TAN><<<level_tiles(f.m, nb), kFuseThreads, 0, s>>>(f, w);
  }
  if (l0 < levels) {
    const int m = n >> l0;
    const size_t sm = (size_t)2 * m * m * sizeof(float2);
    auto k = k_cs_core<TAN>;
    // always the limit of the largest core: it belongs to the function, and a context
    // of another size in another thread must not lower it under this launch
    constexpr int most = 2 * kCoreSide * kCoreSide * (int)sizeof(float2);
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    k<<<nb, kCoreThreads, sm, s>>>(buf[(l0 - 1) & 1], n, m, levels - l0, f.at, f.keep, f.tau, w);
  }
  for (int l = l0 - 1; l >= 1; --l)
    k_cs_inv<kStorePlain><<<level_tiles(n >> l, nb), kFuseThreads, 0, s>>>(
        InvArgs{n, n >> l, buf[l & 1], buf[(l - 1) & 1], nullptr, 0.f}, w);
}

__global__ void k_scale(float2* __restrict__ x, float s, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  x[o] = cscale(x[o], s);
}

// 2-D mask: out = mask2d . in . scale (k-space planes)
__global__ void k_mask2d(const float2* __restrict__ in, float2* __restrict__ out, const uint8_t* __restrict__ mask,
                         float scale, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t o = (size_t)blockIdx.y * n + i;
  out[o] = mask[i] ? cscale(in[o], scale) : make_float2(0.f, 0.f);
}

// x[b] = sum_c conj(S_c) . G[b][c]
__global__ void k_coil_combine(const float2* __restrict__ G, const float2* __restrict__ S, int nc,
                               float2* __restrict__ x, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int b = blockIdx.y;
  float2 acc = make_float2(0.f, 0.f);
  for (int c = 0; c < nc; ++c) acc = cfma_c(acc, S[(size_t)c * n + i], G[((size_t)b * nc + c) * n + i]);
  x[(size_t)b * n + i] = acc;
}

// CN(0, sigma^2) noise on the sampled positions of a 2-D mask, element index (c * ny + ky) * nx + kx
__global__ void k_noise_kspace2d(float2* __restrict__ G, const uint8_t* __restrict__ mask, int nc, int64_t n,
                                 uint64_t seed, int64_t rep_begin, float sigma) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int bc = blockIdx.y, b = bc / nc, c = bc % nc;
  float2 v = make_float2(0.f, 0.f);
  if (mask[i]) {
    const uint64_t key = splitmix64(seed, (uint64_t)(rep_begin + b));
    v = draw_cnoise(key, (uint64_t)c * (uint64_t)n + (uint64_t)i, sigma);
  }
  G[(size_t)bc * n + i] = v;
}

}  // namespace

// The first analysis level covers the whole image, so it reads x directly (x may equal coef).
void launch_dwt(const float2* x, float2* coef, float2* tmp, int n, int levels, int nb, const Wavelet& w,
                cudaStream_t s) {
  const int64_t img = (int64_t)n * n;
  for (int l = 0; l < levels; ++l) {
    const int m = n >> l;
    k_dwt_rows_fwd<<<dim3(blocks((int64_t)m * (m / 2)), nb), 256, 0, s>>>(l == 0 ? x : coef, tmp, n, m, m, img, w);
    k_dwt_cols_fwd<<<dim3(blocks((int64_t)(m / 2) * m), nb), 256, 0, s>>>(tmp, coef, n, m, m, img, w);
  }
}

// Synthesis runs in place on x; with x == coef no copy is needed.
void launch_idwt(const float2* coef, float2* x, float2* tmp, int n, int levels, int nb, const Wavelet& w,
                 cudaStream_t s) {
  const int64_t img = (int64_t)n * n;
  if (coef != x) k_copy_region<<<dim3(blocks(img), nb), 256, 0, s>>>(coef, x, n, n, n, img);
  for (int l = levels - 1; l >= 0; --l) {
    const int m = n >> l;
    k_dwt_cols_inv<<<dim3(blocks((int64_t)m * m), nb), 256, 0, s>>>(x, tmp, n, m, m, img, w);
    k_dwt_rows_inv<<<dim3(blocks((int64_t)m * m), nb), 256, 0, s>>>(tmp, x, n, m, m, img, w);
  }
}

int dwt_kernels(int levels) { return 2 * levels; }
int idwt_kernels(int levels, bool in_place) { return 2 * levels + (in_place ? 0 : 1); }

void launch_axpy_bcast(float2* x, const float2* y, float alpha, int64_t n, int nb, cudaStream_t s) {
  k_axpy_bcast<<<dim3(blocks(n), nb), 256, 0, s>>>(x, y, alpha, n);
}
void launch_cs_gradstep(const float2* z, const float2* Mz, const float2* rhs, int64_t rhs_stride, float inv_lc,
                        float2* y, int64_t n, int nb, cudaStream_t s) {
  k_cs_gradstep<<<dim3(blocks(n), nb), 256, 0, s>>>(z, Mz, rhs, rhs_stride, inv_lc, y, n);
}
void launch_cs_soft(const float2* c, float2* keep, float2* out, float tau, int64_t n, int nb, cudaStream_t s) {
  k_cs_soft<<<dim3(blocks(n), nb), 256, 0, s>>>(c, keep, out, tau, n);
}
void launch_cs_soft_tan(const float2* at, float2* dc, float tau, int64_t n, int nb, cudaStream_t s) {
  k_cs_soft_tan<<<dim3(blocks(n), nb), 256, 0, s>>>(at, dc, tau, n);
}
void launch_cs_momentum(const float2* xn, float2* x, float2* z, float c, int64_t n, int nb, cudaStream_t s) {
  k_cs_momentum<<<dim3(blocks(n), nb), 256, 0, s>>>(xn, x, z, c, n);
}
void launch_vjp_a(float2* xbn, const float2* zb, float2* xk1, float c, int64_t n, int nb, cudaStream_t s) {
  k_vjp_a<<<dim3(blocks(n), nb), 256, 0, s>>>(xbn, zb, xk1, c, n);
}
void launch_vjp_b(const float2* yb, const float2* Myb, float inv_lc, float2* zb, float2* ysum, int64_t n, int nb,
                  cudaStream_t s) {
  k_vjp_b<<<dim3(blocks(n), nb), 256, 0, s>>>(yb, Myb, inv_lc, zb, ysum, n);
}
bool cs_fused_supported(int n, int levels) { return levels >= 1 && (n >> (levels - 1)) >= kTapMax - 2; }
int cs_fused_kernels(int n, int levels) {
  int l0 = 1;
  while (l0 < levels && (n >> l0) > kCoreSide) ++l0;
  return 2 * l0 + (l0 < levels ? 1 : 0);
}

void launch_cs_iter(const float2* z, const float2* Mz, const float2* rhs, int64_t rhs_stride, float inv_lc,
                    const float2* at, float2* keep, float tau, float2* b0, float2* b1, float2* x, float2* zout,
                    float c, int n, int levels, int nb, const Wavelet& w, cudaStream_t s) {
  FwdArgs f{n, n, z, Mz, rhs, rhs_stride, inv_lc, 0.f, 0.f, nullptr, b0, at, keep, tau, 0};
  if (at)
    cs_shrink<kLoadGrad, true>(f, b0, b1, levels, nb, w, s);
  else
    cs_shrink<kLoadGrad, false>(f, b0, b1, levels, nb, w, s);
  k_cs_inv<kStoreMomentum><<<level_tiles(n, nb), kFuseThreads, 0, s>>>(InvArgs{n, n, b0, x, zout, c}, w);
}

void launch_vjp_iter(const float2* yb, const float2* Myb, float inv_lc, const float2* xb, float c_prev, float c,
                     float2* znew, const float2* at, float tau, float2* b0, float2* b1, float2* yout, float2* ysum,
                     int n, int levels, int nb, const Wavelet& w, cudaStream_t s) {
  FwdArgs f{n, n, yb, Myb, xb, 0, inv_lc, 1.f + c, c_prev, znew, b0, at, nullptr, tau, 0};
  cs_shrink<kLoadVjp, true>(f, b0, b1, levels, nb, w, s);
  k_cs_inv<kStoreVjp><<<level_tiles(n, nb), kFuseThreads, 0, s>>>(InvArgs{n, n, b0, yout, ysum, 0.f}, w);
}
void launch_scale(float2* x, float sc, int64_t n, int nb, cudaStream_t s) {
  k_scale<<<dim3(blocks(n), nb), 256, 0, s>>>(x, sc, n);
}
void launch_mask2d(const float2* in, float2* out, const uint8_t* mask, float scale, int64_t n, int planes,
                   cudaStream_t s) {
  k_mask2d<<<dim3(blocks(n), planes), 256, 0, s>>>(in, out, mask, scale, n);
}
void launch_coil_combine(const float2* G, const float2* S, int nc, float2* x, int64_t n, int nb, cudaStream_t s) {
  k_coil_combine<<<dim3(blocks(n), nb), 256, 0, s>>>(G, S, nc, x, n);
}
void launch_noise_kspace2d(float2* G, const uint8_t* mask, int nc, int64_t n, int nb, uint64_t seed,
                           int64_t rep_begin, float sigma, cudaStream_t s) {
  k_noise_kspace2d<<<dim3(blocks(n), nb * nc), 256, 0, s>>>(G, mask, nc, n, seed, rep_begin, sigma);
}

}  // namespace pico
