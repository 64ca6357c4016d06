// Non-Cartesian (spiral) operators on the GPU (kernel templates).
//
// Normal operator by Toeplitz embedding (Sec. 3.2.2 / Sec. 3.3, Fessler 2005):
// for an N x N image and the exact NUDFT A_c = E diag(S_c),
//     A^H A x = sum_c conj(S_c) . crop_N IDFT_2N( T^ . DFT_2N( pad_2N(S_c . x) ) )
// where T^ = DFT_2N of the point-spread kernel h(d) = (1/N^2) sum_m e^{+2 pi i k_m.d/N},
// d in (-N, N)^2, placed circularly on the 2N grid (its DFT is real because h
// is Hermitian).  Three passes per normal operator, all on the 2N grid:
//   rows_fwd : per image row and coil, S_c . p zero-padded to 2N, row FFT  -> G[b][c][N][2N]
//   cols     : per grid column and coil, column FFT (rows >= N are zero), x T^,
//              inverse column FFT, rows < N written back in place
//   rows_inv : per image row, inverse row FFT of every coil, first N samples,
//              conj(S_c) coil combine, + lam p, p^H q partial
// The CG direction update p = r + beta p is fused into rows_fwd.
//
// PMR adjoint A^H n (Sec. 1; Kaiser-Bessel gridding, width W, oversampling 2):
//   grid     : gather-form gridding of CN(0, sigma^2) k-space noise drawn per
//              (replica, coil, sample) onto the 2N grid, no atomics
//   fft rows : inverse row FFT of the grid
//   cols_adj : inverse column FFT, centred crop, deapodisation, conj(S_c)
//              coil combine
#pragma once
#include "common.cuh"
#include "fft_blocks.cuh"
#include "kernels.cuh"
#include "row_pass.cuh"
#include "tc_util.cuh"

namespace pico {


__device__ __forceinline__ const double* sp_rr(const CgArgs& a, int b, int it) {
  return a.rr_part + ((size_t)b * (a.itmax + 1) + it) * a.PB;
}
__device__ __forceinline__ double* sp_pq(const CgArgs& a, int b, int it) {
  return a.pq_part + ((size_t)b * a.itmax + it) * a.PA;
}

// CG scalars of iteration it (computed by warp 0): returns done flag and beta
__device__ __forceinline__ void cg_scalars(const CgArgs& a, int b, int it, int* sh_done, float* sh_beta) {
  if (threadIdx.x < 32) {
    const double rr = warp_sum_parts(sp_rr(a, b, it), a.PB);
    const double rr0 = warp_sum_parts(sp_rr(a, b, 0), a.PB);
    const double rrp = it > 0 ? warp_sum_parts(sp_rr(a, b, it - 1), a.PB) : 1.0;
    if (threadIdx.x == 0) {
      *sh_done = !(rr > a.rtol2 * rr0);
      *sh_beta = it > 0 ? (float)(rr / rrp) : 0.f;
    }
  }
}

// ---------------------------------------------------------------------------
// Pass 1: rows of the image, forward transform of S_c . p padded to L = 2N
// ---------------------------------------------------------------------------
// PAD: the grid is 2N (Toeplitz embedding, image in the first half of each
// line); otherwise L = N (2-D Cartesian masks: plain 2-D DFT, no padding).
// The next step's sensitivity rows (contiguous) arrive by bulk copies while the
// b-jobs of the current step run.
template <int P1, int P2, bool CG, bool PAD, int NT>
__global__ void __launch_bounds__(NT, 512 / NT)
    k_toep_rows_fwd(SpiralOp op, const float2* __restrict__ xin, float2* __restrict__ G, CgArgs a, int it) {
  using Rp = RowPass<P1, P2, NT>;
  constexpr int RL = Rp::RL, CS = Rp::CS, GA = Rp::GA, CA = Rp::CA;
  constexpr int NIN = PAD ? P2 / 2 : P2;  // samples n1 + P1 n2 inside the image: n2 < NIN
  constexpr int L = P1 * P2;
  constexpr int N = PAD ? L / 2 : L;
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* ex = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
  float2* sst = reinterpret_cast<float2*>(ex + CS * Rp::slot);  // [CS][RL][N]
  float2* twt = sst + CS * RL * N;                              // [P2][P1]
  uint64_t* bar = reinterpret_cast<uint64_t*>(twt + L);
  __shared__ float sh_beta;
  __shared__ int sh_done;
  const int t = threadIdx.x, b = blockIdx.y, y0 = blockIdx.x * RL;
  if (t == 0) {
    tc::mbar_init(bar, 1);
    tc::fence_mbar_init();
  }
  for (int i = t; i < L; i += NT) twt[i] = op.tw2[(i / P1) * (i % P1)];
  if (CG) cg_scalars(a, b, it, &sh_done, &sh_beta);
  __syncthreads();
  if (CG && blockIdx.x == 0 && t == 0 && a.done) a.done[b] = sh_done;  // for the column pass
  if (CG && sh_done) return;
  auto issue = [&](int c0) {  // sensitivity rows of a step
    const int cn = min(CS, op.nc - c0);
    tc::mbar_expect_tx(bar, (uint32_t)(cn * RL * N * 8));
    for (int c = 0; c < cn; ++c)
      tc::bulk_load(sst + c * RL * N, op.smaps + ((size_t)(c0 + c) * N + y0) * N, RL * N * 8, bar);
  };
  if (t == 0) issue(0);

  const int g = t / (RL * P1), mm = t - g * (RL * P1), ra = mm / P1, n1 = mm - ra * P1;
  const bool ajob = t < Rp::AT;
  const int cb = t / (RL * P2), rb = (t / P2) % RL, k2 = t % P2;
  float2 p[NIN];
  if (ajob) {
    const float beta = CG ? sh_beta : 0.f;
    const size_t row = ((size_t)b * N + y0 + ra) * N + n1;
#pragma unroll
    for (int n2 = 0; n2 < NIN; ++n2) {
      const size_t idx = row + P1 * n2;
      if (CG) {
        float2 v = a.R[idx];
        if (it > 0) {
          const float2 po = a.P[idx];
          v = make_float2(fmaf(beta, po.x, v.x), fmaf(beta, po.y, v.y));
        }
        p[n2] = v;
      } else {
        p[n2] = xin[idx];
      }
    }
    if (CG && GA == 1)
#pragma unroll
      for (int n2 = 0; n2 < NIN; ++n2) a.P[row + P1 * n2] = p[n2];
  }
  if (CG && GA > 1) {  // every subgroup has read the old direction before one writes the new
    __syncthreads();
    if (t < RL * P1)
#pragma unroll
      for (int n2 = 0; n2 < NIN; ++n2) a.P[((size_t)b * N + y0 + ra) * N + n1 + P1 * n2] = p[n2];
  }
  bool ok = true;
  int phase = 0;
  for (int c0 = 0; c0 < op.nc; c0 += CS, phase ^= 1) {
    if (ok && !tc::mbar_wait(bar, phase)) {  // reported by pico_sync; the block runs on so that its barriers pair up
      ok = false;
      if (op.err) atomicCAS(op.err, 0, kWaitToepRowsFwd);
    }
    if (ajob) {
#pragma unroll
      for (int j = 0; j < CA; ++j) {
        const int cs = j * GA + g;
        if (c0 + cs < op.nc) {
          float2 z[P2];
          const float2* S = sst + (cs * RL + ra) * N + n1;
#pragma unroll
          for (int n2 = 0; n2 < P2; ++n2) z[n2] = n2 < NIN ? cmul(S[P1 * n2], p[n2]) : make_float2(0.f, 0.f);
          dft_nz<P2, -1, NIN>(z);
          unsigned char* e = ex + cs * Rp::slot + ra * Rp::line;
#pragma unroll
          for (int k = 0; k < P2; k += 2) {
            const float2 u = k == 0 ? z[0] : cmul(z[k], twt[k * P1 + n1]), v = cmul(z[k + 1], twt[(k + 1) * P1 + n1]);
            *reinterpret_cast<float4*>(e + Rp::at(n1, k)) = make_float4(u.x, u.y, v.x, v.y);
          }
        }
      }
    }
    __syncthreads();  // exchange slots full, sensitivities read
    if (t == 0 && ok && c0 + CS < op.nc) issue(c0 + CS);
    if (c0 + cb < op.nc) {
      float2 y[P1];
      const unsigned char* e = ex + cb * Rp::slot + rb * Rp::line;
#pragma unroll
      for (int m = 0; m < P1; ++m) y[m] = *reinterpret_cast<const float2*>(e + Rp::at(m, k2));
      DFT<P1, -1>::run(y);
      float2* __restrict__ gr = G + (((size_t)b * op.nc + c0 + cb) * N + y0 + rb) * L + k2;
#pragma unroll
      for (int k1 = 0; k1 < P1; ++k1) gr[P2 * k1] = y[k1];
    }
    __syncthreads();  // the slots are rewritten by the next step
  }
  if (t == 0 && !ok)  // nothing more was requested: wait (bounded) for what was
    for (int i = 0; i < 2; ++i) tc::mbar_wait(bar, i, 200000000ull);
}

// ---------------------------------------------------------------------------
// Pass 2: columns of the grid: FFT (rows >= N zero), x T^, inverse FFT, rows < N
// ---------------------------------------------------------------------------
// Persistent: each block walks work items (plane, group of CL grid columns) and
// one thread brings the next item's N x CL input values into a staging buffer
// with TMA tensor loads while the block transforms the current item, so the
// global-load latency of a plane does not stall every thread at its start.
// done: per-image stop flags of the CG iteration (nullptr outside CG); planes of
// converged images are skipped.
//
// CL = 16 columns: a half-warp's 16 columns fill a 128-byte shared-memory
// wavefront and a full 128-byte line of the grid, and blocks of P2 x 16 threads
// (one b-job each) run two or three to an SM, so one block's barriers and loads
// overlap another's arithmetic.  96 images, 240 x 240, 20 coils (L = 480), whole
// normal operator: groups of 30 columns (one 480-thread block per SM) 2397 us,
// 16 columns 2287 us, 8 columns 2403 us (64-byte global accesses), 4 columns
// 2824 us.  The twiddles are read two at a time, [n1][k] with padded rows, by
// the a-jobs in both directions (single look-ups W^(n1 k) by a- and b-jobs:
// 2084 us against 2045 us, with the row passes below in place).
// Bound by shared-memory wavefronts and the FP32 pipes at about half each (ncu,
// 32 images: 59 % and 47 %): every value crosses shared memory five times, and
// two blocks of 8 warps overlap the two pipes only partly.
template <int P1, int P2>
struct ColsW {
  static constexpr int CL = 16;                    // grid columns per item
  static constexpr int NT = P2 * CL;               // one b-job per thread
  static constexpr int KS = P1 * CL;               // k2 stride of the exchange buffer
  static constexpr int TS = P2 + 2;                // twiddle row, padded against bank conflicts
  static constexpr size_t smem(int n) {
    return 1024 + ((size_t)n * CL + (size_t)P2 * KS + P1 * TS) * sizeof(float2) + 16;
  }
  // blocks per SM to compile for: three of 256 threads (six of 128) where the
  // shorter DFT and the shared memory allow, otherwise two (four)
  static constexpr int blocks(int n) {
    const int want = (P1 <= 20 ? 768 : 512) / NT, fit = (int)((size_t)227 * 1024 / (smem(n) + 1024));
    return fit < 1 ? 1 : fit < want ? fit : want;
  }
};
template <int P1, int P2, bool PAD>
__global__ void __launch_bounds__(ColsW<P1, P2>::NT, (ColsW<P1, P2>::blocks(PAD ? P1 * P2 / 2 : P1 * P2)))
    k_toep_cols_w(SpiralOp op, const __grid_constant__ CUtensorMap mG, float2* __restrict__ G,
                  const int* __restrict__ done, int nplanes, int box_rows) {
  constexpr int NIN = PAD ? P2 / 2 : P2;
  constexpr int L = P1 * P2;
  constexpr int NT = ColsW<P1, P2>::NT;
  constexpr int CL = ColsW<P1, P2>::CL;
  constexpr int NG = L / CL;
  constexpr int KS = ColsW<P1, P2>::KS, TS = ColsW<P1, P2>::TS;
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
  const int t = threadIdx.x, N = op.n;          // N input rows per plane
  float2* stage = reinterpret_cast<float2*>(sm);  // [N][CL] input rows of the item
  float2* buf = stage + (size_t)N * CL;           // [k2][n1][CL]
  float2* tws = buf + (size_t)P2 * KS;            // [n1][k]: W^(n1 k)
  uint64_t* bar = reinterpret_cast<uint64_t*>(tws + P1 * TS);
  int* arrived = reinterpret_cast<int*>(bar + 1);
  const int items = NG * nplanes;
  const uint32_t bytes = (uint32_t)N * CL * sizeof(float2);
  if (t == 0) {
    tc::mbar_init(bar, 1);
    tc::fence_mbar_init();
  }
  for (int i = t; i < L; i += NT) tws[(i / P2) * TS + i % P2] = op.tw2[(i / P2) * (i % P2)];
  __syncthreads();
  auto issue = [&](int w) {
    const int plane = w / NG, cg = w - plane * NG;
    tc::mbar_expect_tx(bar, bytes);
    for (int r0 = 0; r0 < N; r0 += box_rows) tc::tma_load_3d(stage + (size_t)r0 * CL, &mG, bar, cg * CL, r0, plane);
  };
  if (t == 0 && (int)blockIdx.x < items) issue(blockIdx.x);
  int phase = 0;
  for (int w = blockIdx.x; w < items; w += gridDim.x, phase ^= 1) {
    const int plane = w / NG, cg = w - plane * NG, x0 = cg * CL;
    // One thread decides whether the item's copy arrived and the block
    // follows that decision together.  On a timeout it records the error,
    // waits once more (bounded) for the copy still in flight into this
    // block's shared memory, and the whole block leaves at the same point.
    if (t == 0) {
      bool ok = tc::mbar_wait(bar, phase);
      if (!ok) {
        if (op.err) atomicCAS(op.err, 0, kWaitToepCols);
        tc::mbar_wait(bar, phase);
      }
      *arrived = ok ? 1 : 0;
    }
    __syncthreads();
    if (!*arrived) return;
    const bool skip = done && done[plane / op.nc];
    float2* __restrict__ g = G + (size_t)plane * N * L;  // (b, c) plane [N][L]
    if (!skip)
      for (int jj = t; jj < P1 * CL; jj += NT) {
        const int n1 = jj / CL, ln = jj - n1 * CL;
        float2 z[P2];
#pragma unroll
        for (int n2 = 0; n2 < P2; ++n2) z[n2] = n2 < NIN ? stage[(n1 + P1 * n2) * CL + ln] : make_float2(0.f, 0.f);
        dft_nz<P2, -1, NIN>(z);
#pragma unroll
        for (int k = 0; k < P2; k += 2) {
          const float4 w = *reinterpret_cast<const float4*>(tws + n1 * TS + k);
          buf[k * KS + n1 * CL + ln] = k == 0 ? z[0] : cmul(z[k], make_float2(w.x, w.y));
          buf[(k + 1) * KS + n1 * CL + ln] = cmul(z[k + 1], make_float2(w.z, w.w));
        }
      }
    __syncthreads();  // the staging buffer is free: fetch the next item
    if (t == 0 && w + (int)gridDim.x < items) issue(w + gridDim.x);
    if (!skip) {
      {
        const int k2 = t / CL, ln = t - k2 * CL, kx = x0 + ln;
        float2 y[P1];
        colb_load<P1, P2, CL>(y, k2, ln, buf);
        DFT<P1, -1>::run(y);
#pragma unroll
        for (int k1 = 0; k1 < P1; ++k1) y[k1] = cscale(y[k1], __ldg(op.That + (size_t)(k2 + P2 * k1) * L + kx));
        DFT<P1, 1>::run(y);
        colb_store<P1, P2, CL>(y, k2, ln, buf);
      }
      __syncthreads();
      for (int jj = t; jj < P1 * CL; jj += NT) {
        const int n1 = jj / CL, ln = jj - n1 * CL;
        float2 z[P2];
#pragma unroll
        for (int k = 0; k < P2; k += 2) {
          const float4 w = *reinterpret_cast<const float4*>(tws + n1 * TS + k);
          z[k] = buf[k * KS + n1 * CL + ln];
          if (k > 0) z[k] = cmul_cb(z[k], make_float2(w.x, w.y));
          z[k + 1] = cmul_cb(buf[(k + 1) * KS + n1 * CL + ln], make_float2(w.z, w.w));
        }
        DFT<P2, 1>::run(z);
#pragma unroll
        for (int n2 = 0; n2 < NIN; ++n2) g[(size_t)(n1 + P1 * n2) * L + x0 + ln] = z[n2];  // rows < N only
      }
    }
    __syncthreads();  // buf is rewritten by the next item
  }
}

// ---------------------------------------------------------------------------
// Pass 3: rows: inverse FFT per coil, first N samples, conj(S) combine, + lam p
// ---------------------------------------------------------------------------
// The grid rows of a step arrive by one TMA tensor load per coil, in the
// swizzled exchange layout, and are transformed in place; those of the next
// step are requested as soon as the a-jobs hold their last coil in registers.
// The 128 registers of four blocks per SM do not hold z, y, the accumulators and
// the addresses for P1 >= 20: 128 threads spill 92 bytes a thread at L = 480 padded,
// 164 unpadded, 96 at 384 and 68 at 320 unpadded.  Three blocks of up to 168
// registers without spills are slower all the same, except at 480 x 480 masks
// (inside CG: 96 images of 240 x 240, 20 coils, 505 us with four blocks, 536 with three;
// 48 of a 320 x 320 mask, 15 coils, 283 and 318; 32 of 384 x 384, 8 coils, 171 and
// 183; 24 of 480 x 480, 8 coils, 242 and 222).
template <int P1, int P2, bool CG, bool PAD, int NT>
__global__ void __launch_bounds__(NT, 512 / NT)
    k_toep_rows_inv(SpiralOp op, const __grid_constant__ CUtensorMap mG, const float2* __restrict__ xin,
                    float2* __restrict__ yout, float lam, CgArgs a, int it) {
  using Rp = RowPass<P1, P2, NT>;
  constexpr int RL = Rp::RL, CS = Rp::CS, GA = Rp::GA, CA = Rp::CA;
  constexpr int NIN = PAD ? P2 / 2 : P2;
  constexpr int L = P1 * P2;
  constexpr int N = PAD ? L / 2 : L;
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* ex = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
  float2* sst = reinterpret_cast<float2*>(ex + CS * Rp::slot);  // [CS][RL][N]
  float2* twt = sst + CS * RL * N;                              // [P2][P1]
  uint64_t* bar = reinterpret_cast<uint64_t*>(twt + L);
  __shared__ double red[(NT + 31) / 32];
  __shared__ float sh_beta;
  __shared__ int sh_done;
  const int t = threadIdx.x, b = blockIdx.y, y0 = blockIdx.x * RL;
  if (t == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_init(bar + 1, 1);
    tc::fence_mbar_init();
  }
  for (int i = t; i < L; i += NT) twt[i] = op.tw2[(i / P1) * (i % P1)];
  if (CG) cg_scalars(a, b, it, &sh_done, &sh_beta);
  __syncthreads();
  if (CG && sh_done) return;
  auto issue_g = [&](int c0) {  // grid rows of a step
    const int cn = min(CS, op.nc - c0);
    tc::mbar_expect_tx(bar, (uint32_t)(cn * RL * L * 8));
    for (int l = 0; l < cn * RL; ++l)
      tc::tma_load_3d(ex + l * Rp::line, &mG, bar, 0, 0, (b * op.nc + c0 + l / RL) * N + y0 + l % RL);
  };
  auto issue_s = [&](int c0) {  // its sensitivity rows
    const int cn = min(CS, op.nc - c0);
    tc::mbar_expect_tx(bar + 1, (uint32_t)(cn * RL * N * 8));
    for (int c = 0; c < cn; ++c)
      tc::bulk_load(sst + c * RL * N, op.smaps + ((size_t)(c0 + c) * N + y0) * N, RL * N * 8, bar + 1);
  };
  if (t == 0) issue_g(0);

  const int g = t / (RL * P1), mm = t - g * (RL * P1), ra = mm / P1, n1 = mm - ra * P1;
  const bool ajob = t < Rp::AT;
  const int cb = t / (RL * P2), rb = (t / P2) % RL, k2 = t % P2;
  // each a-thread owns NO image columns of its (row, n1); with several subgroups
  // the owners add the coils' samples in coil order too, so that the sum's bits
  // (and the p^H q partial's, summed as one thread per (row, n1) would) do not
  // depend on the number of threads, that is on the batch
  constexpr int NO = NIN / GA;
  float2 acc[NO];
#pragma unroll
  for (int i = 0; i < NO; ++i) acc[i] = make_float2(0.f, 0.f);
  bool ok = true;
  int phase = 0;
  for (int c0 = 0; c0 < op.nc; c0 += CS, phase ^= 1) {
    if (ok && !tc::mbar_wait(bar, phase)) {  // reported by pico_sync; the block runs on so that its barriers pair up
      ok = false;
      if (op.err) atomicCAS(op.err, 0, kWaitToepRowsInv);
    }
    if (c0 + cb < op.nc) {
      float2 y[P1];
      unsigned char* e = ex + cb * Rp::slot + rb * Rp::line;
#pragma unroll
      for (int m = 0; m < P1; ++m) y[m] = *reinterpret_cast<const float2*>(e + Rp::at(m, k2));
      DFT<P1, 1>::run(y);
#pragma unroll
      for (int m = 0; m < P1; ++m) *reinterpret_cast<float2*>(e + Rp::at(m, k2)) = y[m];
    }
    __syncthreads();  // rows transformed; the sensitivities of the step before were last read before it
    if (t == 0 && ok) issue_s(c0);
#pragma unroll 1
    for (int j = 0; j < CA; ++j) {
      const int cs = j * GA + g;
      const bool on = ajob && c0 + cs < op.nc;
      unsigned char* e = ex + cs * Rp::slot + ra * Rp::line;
      float2 z[P2];
      if (on) {
#pragma unroll
        for (int k = 0; k < P2; k += 2) {
          const float4 v = *reinterpret_cast<const float4*>(e + Rp::at(n1, k));
          z[k] = k == 0 ? make_float2(v.x, v.y) : cmul_cb(make_float2(v.x, v.y), twt[k * P1 + n1]);
          z[k + 1] = cmul_cb(make_float2(v.z, v.w), twt[(k + 1) * P1 + n1]);
        }
      }
      if (GA == 1 && j == CA - 1) {
        tc::fence_proxy_async_smem();  // the in-place writes before the next step's copies
        __syncthreads();               // the slots are free
        if (t == 0 && ok && c0 + CS < op.nc) issue_g(c0 + CS);
      }
      if (on) DFT<P2, 1>::run(z);
      if (j == 0 && ok && !tc::mbar_wait(bar + 1, phase)) {
        ok = false;
        if (op.err) atomicCAS(op.err, 0, kWaitToepRowsInv);
      }
      if (GA == 1) {
        if (on) {
          const float2* S = sst + (cs * RL + ra) * N + n1;
#pragma unroll
          for (int i = 0; i < NO; ++i) acc[i] = cfma_c(acc[i], S[P1 * i], z[i]);
        }
      } else if (on) {  // handed to the owners, in this job's own row
#pragma unroll
        for (int n2 = 0; n2 < NIN; n2 += 2)
          *reinterpret_cast<float4*>(e + Rp::at(n1, n2)) = make_float4(z[n2].x, z[n2].y, z[n2 + 1].x, z[n2 + 1].y);
      }
    }
    if (GA > 1) {
      __syncthreads();
      if (ajob) {
        const int cn = min(CS, op.nc - c0);
#pragma unroll 2
        for (int cs = 0; cs < cn; ++cs) {
          const unsigned char* e = ex + cs * Rp::slot + ra * Rp::line;
          const float2* S = sst + (cs * RL + ra) * N + n1 + P1 * NO * g;
#pragma unroll
          for (int i = 0; i < NO; ++i)
            acc[i] = cfma_c(acc[i], S[P1 * i], *reinterpret_cast<const float2*>(e + Rp::at(n1, NO * g + i)));
        }
      }
      tc::fence_proxy_async_smem();
      __syncthreads();
      if (t == 0 && ok && c0 + CS < op.nc) issue_g(c0 + CS);
    }
  }
  // after a time-out nothing more was requested: wait (bounded) for what was; of
  // each barrier's two parities the completed one returns at once
  if (t == 0 && !ok)
    for (int i = 0; i < 4; ++i) tc::mbar_wait(bar + i / 2, i & 1, 200000000ull);
  float pq = 0.f;
  float* term = reinterpret_cast<float*>(ex);  // [RL P1][NIN] (GA > 1)
  if (ajob) {
    const float2* __restrict__ pin = CG ? a.P : xin;
    float2* __restrict__ out = CG ? a.Q : yout;
#pragma unroll
    for (int i = 0; i < NO; ++i) {
      const size_t idx = ((size_t)b * N + y0 + ra) * N + n1 + P1 * (NO * g + i);
      const float2 pv = pin[idx];
      const float2 q = make_float2(fmaf(lam, pv.x, acc[i].x), fmaf(lam, pv.y, acc[i].y));
      out[idx] = q;
      if (GA == 1)
        pq += cdot_re(pv, q);
      else if (CG)
        term[mm * NIN + NO * g + i] = cdot_re(pv, q);
    }
  }
  if (CG && GA > 1) {
    __syncthreads();
    if (t < RL * P1)
#pragma unroll
      for (int n2 = 0; n2 < NIN; ++n2) pq += term[t * NIN + n2];
  }
  if (CG) {
    const double tot = block_sum_d((double)pq, red);
    if (t == 0) sp_pq(a, b, it)[blockIdx.x] = tot;
  }
}

// ---------------------------------------------------------------------------
// In-place forward FFTs of all rows / all columns of an L x L grid (set-up)
// ---------------------------------------------------------------------------
template <int P1, int P2>
__global__ void __launch_bounds__(Split<P1, P2>::NT, 1) k_fft_rows(float2* __restrict__ plane, const float2* tw2) {
  constexpr int L = P1 * P2;
  constexpr int NT = Split<P1, P2>::NT;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* buf = reinterpret_cast<float2*>(smraw);
  float2* tws = buf + kLines * P2 * Split<P1, P2>::LD;
  const int t = threadIdx.x;
  for (int i = t; i < L; i += NT) tws[i] = tw2[i];
  __syncthreads();
  const int ra = t / P1, n1 = t % P1;
  const int rb = t / P2, k2 = t % P2;
  if (t < kLines * P1) {
    float2 z[P2];
    const float2* row = plane + (size_t)(blockIdx.x * kLines + ra) * L;
#pragma unroll
    for (int n2 = 0; n2 < P2; ++n2) z[n2] = row[n1 + P1 * n2];
    rowa_store<P1, P2, -1>(z, n1, ra, buf, tws);
  }
  __syncthreads();
  if (t < kLines * P2) {
    float2 y[P1];
    rowb_load<P1, P2, -1>(y, k2, rb, buf);
    float2* row = plane + (size_t)(blockIdx.x * kLines + rb) * L;
#pragma unroll
    for (int k1 = 0; k1 < P1; ++k1) row[k2 + P2 * k1] = y[k1];
  }
}

template <int P1, int P2>
__global__ void __launch_bounds__(Split<P1, P2>::NT, 1) k_fft_cols(float2* __restrict__ plane, const float2* tw2) {
  constexpr int L = P1 * P2;
  constexpr int NT = Split<P1, P2>::NT;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* buf = reinterpret_cast<float2*>(smraw);
  float2* tws = buf + L * kLines;
  const int t = threadIdx.x;
  for (int i = t; i < L; i += NT) tws[i] = tw2[i];
  __syncthreads();
  const int ln = t % kLines, job = t / kLines;
  const int kx = blockIdx.x * kLines + ln;
  if (job < P1) {
    float2 z[P2];
#pragma unroll
    for (int n2 = 0; n2 < P2; ++n2) z[n2] = plane[(size_t)(job + P1 * n2) * L + kx];
    cola_store<P1, P2, -1>(z, job, ln, buf, tws);
  }
  __syncthreads();
  if (job < P2) {
    float2 y[P1];
    colb_load<P1, P2>(y, job, ln, buf);
    DFT<P1, -1>::run(y);
#pragma unroll
    for (int k1 = 0; k1 < P1; ++k1) plane[(size_t)(job + P2 * k1) * L + kx] = y[k1];
  }
}

// ---------------------------------------------------------------------------
// PMR adjoint, row pass: inverse row FFT of every grid row, in place; only the
// columns that the centred crop keeps (N of L = 2N) are written.  Blocks of 128
// threads on CS x kRowLines rows in the row passes' exchange layout, four per
// SM, so that one block's loads and stores overlap another's transforms (640
// planes of 480 x 480: one 480-thread block per SM and whole rows written 513 us,
// now 395 us; 1.77 GB, two thirds of the HBM rate).
// ---------------------------------------------------------------------------
template <int P1, int P2>
__global__ void __launch_bounds__(128, 4) k_grid_rows_adjoint(SpiralOp op, float2* __restrict__ data) {
  using Rp = RowPass<P1, P2, 128>;
  constexpr int L = P1 * P2, NT = 128, LINES = Rp::CS * Rp::RL, Q4 = L / 4;
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* ex = smraw;
  float2* twt = reinterpret_cast<float2*>(ex + LINES * Rp::line);  // [P2][P1]
  const int t = threadIdx.x;
  for (int i = t; i < L; i += NT) twt[i] = op.tw2[(i / P1) * (i % P1)];
  __syncthreads();
  float2* __restrict__ rows = data + (size_t)blockIdx.x * LINES * L;
  for (int e = t; e < LINES * P1; e += NT) {
    const int l = e / P1, n1 = e - l * P1;
    float2 z[P2];
#pragma unroll
    for (int n2 = 0; n2 < P2; ++n2) z[n2] = rows[(size_t)l * L + n1 + P1 * n2];
    DFT<P2, 1>::run(z);
    unsigned char* x = ex + l * Rp::line;
#pragma unroll
    for (int k = 0; k < P2; k += 2) {
      const float2 u = k == 0 ? z[0] : cmul_cb(z[k], twt[k * P1 + n1]), v = cmul_cb(z[k + 1], twt[(k + 1) * P1 + n1]);
      *reinterpret_cast<float4*>(x + Rp::at(n1, k)) = make_float4(u.x, u.y, v.x, v.y);
    }
  }
  __syncthreads();
  const int l = t / P2, k2 = t % P2;
  float2 y[P1];
  const unsigned char* x = ex + l * Rp::line;
#pragma unroll
  for (int m = 0; m < P1; ++m) y[m] = *reinterpret_cast<const float2*>(x + Rp::at(m, k2));
  DFT<P1, 1>::run(y);
#pragma unroll
  for (int k1 = 0; k1 < P1; ++k1) {
    const int gx = k2 + P2 * k1;
    if (gx < Q4 || gx >= L - Q4) rows[(size_t)l * L + gx] = y[k1];
  }
}

// ---------------------------------------------------------------------------
// PMR adjoint, last pass: inverse column FFT of the (row-transformed) grid,
// centred crop to the N x N image, deapodisation and conj(S_c) coil combine.
// Image column x reads grid column (x - N/2) mod L; image row y is grid row
// (y - N/2) mod L.  One CTA: 16 image columns of one replica, all coils; P2 x 16
// threads, one b-job each, two blocks per SM or more.  Only the grid rows
// k2 + P2 k1 with k1 in the first or last quarter can lie in the crop, so a
// thread keeps 2 KA accumulators instead of P1 (32 replicas of 20 coils,
// 240 x 240: one 480-thread block per SM, idle in the b-jobs, 661 us; now 199 us,
// at the HBM rate of its 1.18 GB).
// ---------------------------------------------------------------------------
template <int P1, int P2>
__global__ void __launch_bounds__(P2 * kLines, 512 / (P2 * kLines))
    k_grid_cols_adjoint(SpiralOp op, const float2* __restrict__ Q, float2* __restrict__ out) {
  constexpr int L = P1 * P2, NT = P2 * kLines, N = L / 2, KA = (P1 + 3) / 4;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* buf = reinterpret_cast<float2*>(smraw);
  float2* tws = buf + L * kLines;
  const int t = threadIdx.x, b = blockIdx.y;
  for (int i = t; i < L; i += NT) tws[i] = op.tw2[i];
  __syncthreads();
  const int ln = t % kLines, job = t / kLines;
  const int x = blockIdx.x * kLines + ln;  // image column
  const bool xval = x < N;
  const int gx = ((x - N / 2) % L + L) % L;
  const float dax = xval ? op.deapod[x] : 0.f;
  float2 acc[2 * KA];
#pragma unroll
  for (int i = 0; i < 2 * KA; ++i) acc[i] = make_float2(0.f, 0.f);
  for (int c = 0; c < op.nc; ++c) {
    const float2* __restrict__ q = Q + ((size_t)b * op.nc + c) * L * L;
    for (int n1 = job; n1 < P1; n1 += P2) {
      float2 z[P2];
#pragma unroll
      for (int n2 = 0; n2 < P2; ++n2) z[n2] = xval ? q[(size_t)(n1 + P1 * n2) * L + gx] : make_float2(0.f, 0.f);
      cola_store<P1, P2, 1>(z, n1, ln, buf, tws);
    }
    __syncthreads();
    if (xval) {
      float2 y[P1];
      colb_load<P1, P2>(y, job, ln, buf);
      DFT<P1, 1>::run(y);
#pragma unroll
      for (int i = 0; i < 2 * KA; ++i) {
        const int k1 = i < KA ? i : P1 - 2 * KA + i;
        const int gy = job + P2 * k1;
        const int yy = (gy + N / 2) % L;  // image row of grid row gy
        if (yy < N) {
          const float2 s = __ldg(op.smaps + ((size_t)c * N + yy) * N + x);
          acc[i] = cfma_c(acc[i], s, cscale(y[k1], dax * op.deapod[yy]));
        }
      }
    }
    __syncthreads();
  }
  if (xval) {
#pragma unroll
    for (int i = 0; i < 2 * KA; ++i) {
      const int k1 = i < KA ? i : P1 - 2 * KA + i;
      const int gy = job + P2 * k1;
      const int yy = (gy + N / 2) % L;
      if (yy < N) out[((size_t)b * N + yy) * N + x] = acc[i];
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// Row passes (grid: n / RL row blocks per image; the p^H q partials of the
// inverse pass, one per row block, fill the context's slots).
template <int P1, int P2, bool PAD, int NT>
void toep_rows_fwd_launch(const SpiralOp& op, const float2* x, float2* G, int nb, const CgArgs* a, int it,
                          cudaStream_t s) {
  using Rp = RowPass<P1, P2, NT>;
  const size_t sm = Rp::smem(op.n);
  const dim3 grow(op.n / Rp::RL, nb);
  auto k1 = a ? k_toep_rows_fwd<P1, P2, true, PAD, NT> : k_toep_rows_fwd<P1, P2, false, PAD, NT>;
  cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k1<<<grow, NT, sm, s>>>(op, x, G, a ? *a : CgArgs{}, it);
}
template <int P1, int P2, bool PAD, int NT>
bool toep_rows_inv_launch(const SpiralOp& op, const float2* x, float2* y, const float2* G, int nb, float lam,
                          const CgArgs* a, int it, cudaStream_t s) {
  using Rp = RowPass<P1, P2, NT>;
  CUtensorMap mG{};
  if (!encode_row_map(&mG, G, P1, P2, (int64_t)nb * op.nc * op.n)) return false;
  const size_t sm = Rp::smem(op.n);
  const dim3 grow(op.n / Rp::RL, nb);
  auto k3 = a ? k_toep_rows_inv<P1, P2, true, PAD, NT> : k_toep_rows_inv<P1, P2, false, PAD, NT>;
  cudaFuncSetAttribute(k3, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k3<<<grow, NT, sm, s>>>(op, mG, x, y, lam, a ? *a : CgArgs{}, it);
  return true;
}

template <int P1, int P2, bool PAD>
bool toep_cols_launch(const SpiralOp& op, float2* G, int nb, const int* done, int nsm, cudaStream_t s) {
  using Cw = ColsW<P1, P2>;
  CUtensorMap mG{};
  const int box_rows = op.n <= 256 ? op.n : op.n / 2;  // TMA boxes of at most 256 rows
  if (!encode_plane_map(&mG, G, op.n, P1 * P2, (int64_t)nb * op.nc, Cw::CL, box_rows)) return false;
  auto k2 = k_toep_cols_w<P1, P2, PAD>;
  const size_t sm = Cw::smem(op.n);
  static thread_local int bps = 0;
  cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (bps == 0 && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k2, Cw::NT, sm) != cudaSuccess) bps = 1;
  const int64_t items = (int64_t)(P1 * P2 / Cw::CL) * nb * op.nc;
  const int grid = (int)std::min<int64_t>(items, (int64_t)std::max(1, bps) * nsm);
  k2<<<grid, Cw::NT, sm, s>>>(op, mG, G, done, nb * op.nc, box_rows);
  return true;
}

// Threads per block of the row passes: 128 (64 where the a-jobs of four rows fit
// in 64), four (eight) blocks per SM, once the row blocks fill the device; below
// that more coils at once per block, which shortens the serial walk over the
// coils -- 256 threads while every block is resident (two per SM; one where the
// shared memory of 480 x 480 masks allows no more), 512 while one per SM is enough.
// Both row passes with 512 / 256 / 128 threads, 152 SMs: 240 x 240 spiral, 20 coils,
// 120 row blocks 31 / 34 / 42 us, 180 blocks 59 / 53 / 57, 300 blocks 67 / 57 / 63,
// 360 blocks 99 / 96 / 78; 320 x 320 mask, 15 coils, 80 blocks 21 / 25 / 31, 240 blocks
// 41 / 36 / 40, 320 blocks 59 / 55 / 49; 480 x 480 mask, 8 coils, 120 blocks 256 / 128
// threads 20 / 23 us, 240 blocks 36 / 31.
template <int P1, int P2, bool PAD, int NT>
bool toep_normal_nt(const SpiralOp& op, const float2* x, float2* y, float2* G, int nb, float lam, const CgArgs* a,
                    int it, int nsm, cudaStream_t s) {
  toep_rows_fwd_launch<P1, P2, PAD, NT>(op, x, G, nb, a, it, s);
  return toep_cols_launch<P1, P2, PAD>(op, G, nb, a ? a->done : nullptr, nsm, s) &&
         toep_rows_inv_launch<P1, P2, PAD, NT>(op, x, y, G, nb, lam, a, it, s);
}

template <int P1, int P2, bool PAD>
bool toep_normal_impl(const SpiralOp& op, const float2* x, float2* y, float2* G, int nb, float lam, const CgArgs* a,
                      int it, cudaStream_t s) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  nsm = std::max(1, nsm);
  const int64_t blocks = (int64_t)nb * (op.n / kRowLines);
  constexpr bool wide = RowPass<P1, P2, 512>::smem(PAD ? P1 * P2 / 2 : P1 * P2) <= 227 * 1024;
  if constexpr (wide)
    if (blocks <= nsm) return toep_normal_nt<P1, P2, PAD, 512>(op, x, y, G, nb, lam, a, it, nsm, s);
  constexpr int resident = 2 * (RowPass<P1, P2, 256>::smem(PAD ? P1 * P2 / 2 : P1 * P2) + 1024) <= 228 * 1024 ? 2 : 1;
  if (blocks <= resident * nsm) return toep_normal_nt<P1, P2, PAD, 256>(op, x, y, G, nb, lam, a, it, nsm, s);
  return toep_normal_nt<P1, P2, PAD, (kRowLines * P1 <= 64 ? 64 : 128)>(op, x, y, G, nb, lam, a, it, nsm, s);
}

template <int P1, int P2>
bool launch_toep_normal_t(const SpiralOp& op, const float2* x, float2* y, float2* G, int nb, float lam,
                          const CgArgs* a, int it, cudaStream_t s) {
  return op.L == 2 * op.n ? toep_normal_impl<P1, P2, true>(op, x, y, G, nb, lam, a, it, s)
                          : toep_normal_impl<P1, P2, false>(op, x, y, G, nb, lam, a, it, s);
}

template <int P1, int P2>
void launch_fft2_t(float2* plane, const float2* tw2, bool rows, cudaStream_t s) {
  using Sp = Split<P1, P2>;
  constexpr int L = P1 * P2;
  if (rows) {
    const size_t sm = Sp::row_buf + L * sizeof(float2);
    auto k = k_fft_rows<P1, P2>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k<<<L / kLines, Sp::NT, sm, s>>>(plane, tw2);
  } else {
    const size_t sm = Sp::col_buf + L * sizeof(float2);
    auto k = k_fft_cols<P1, P2>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k<<<L / kLines, Sp::NT, sm, s>>>(plane, tw2);
  }
}

template <int P1, int P2>
void launch_grid_rows_adjoint_t(const SpiralOp& op, float2* Q, int nb, cudaStream_t s) {
  using Rp = RowPass<P1, P2, 128>;
  constexpr int lines = Rp::CS * Rp::RL;   // divides L, a multiple of 16
  const size_t sm = (size_t)lines * Rp::line + Rp::tw;
  auto k = k_grid_rows_adjoint<P1, P2>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  const int64_t blocks = (int64_t)nb * op.nc * (P1 * P2 / lines);
  k<<<(unsigned)blocks, 128, sm, s>>>(op, Q);
}

template <int P1, int P2>
void launch_grid_cols_adjoint_t(const SpiralOp& op, const float2* Q, float2* out, int nb, cudaStream_t s) {
  using Sp = Split<P1, P2>;
  constexpr int L = P1 * P2;
  const size_t sm = Sp::col_buf + L * sizeof(float2);
  auto k = k_grid_cols_adjoint<P1, P2>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k<<<dim3((op.n + kLines - 1) / kLines, nb), P2 * kLines, sm, s>>>(op, Q, out);
}

}  // namespace pico
