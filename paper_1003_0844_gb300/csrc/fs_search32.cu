// FP32 search path with compensated (double-float) phases: per-sky constants,
// the per-sky resampling/demodulation (A1) and the host orchestration of the
// transform passes (device code in fs_pass32.cuh).
//
// Per sky (A1): source times t_j of Eq. (eq:Bt), the spline value x~_j (Sec. VI.A),
// a_j, b_j (Sec. II), the heterodyne factor exp(-2 pi i fl phi_m(t_j)) and
// the spindown phase argument Q_j = t_j^2/2 + t_j phi_m(t_j) (Eq. phas) kept
// as a double-float.  The delay, a and b come from polynomials through a few nodes per
// block of samples (k_demod_nodes, k_demod_poly); for a caller's position table, the
// nearest-neighbour resampler and sampling intervals above 16 s every sample takes one
// Newton step from a first delay estimate (k_demod32).  Output per sky: y^a_j, y^b_j
// (float2) and Q_j.
#include <stdio.h>
#include <algorithm>
#include "fs_demod.cuh"
#include "fs_pass32.cuh"

namespace fs {

// ------------------------------------------------------------------ self-test of the bounded waits
__device__ unsigned g_never_incremented = 0;  // nothing writes it

__global__ void k_selftest_wait(uint32_t *flags) {
  if (threadIdx.x == 0) wait_at_least(&g_never_incremented, 1u, flags);
  __syncthreads();
}

cudaError_t selftest_wait(uint32_t *flags, cudaStream_t st) {
  k_selftest_wait<<<1, 32, 0, st>>>(flags);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ set-up of a search
// One launch for everything a search needs before its first demodulation: the per-sky
// constants, the spindowns as double-floats (an FP64 conversion in every transform item
// would occupy the slow FP64 pipe) and the candidate count.  Latency bound (a few
// thousand threads at most): two lanes per sky take the sine and cosine of alpha and of
// delta side by side, everything that depends on the detector alone comes from DetConst.
// With the finalize kernel below and the dependent launches: 43.7 -> 22.5 us for one
// template of a 1-day series, 39.5 -> 21.2 us for six of a 1346-sample one (the constants
// alone took 13 us with all their sines in one thread).
__device__ __forceinline__ void sky_store(const SkyConst64 &k, SkyConst64 *out) { *out = k; }
__device__ __forceinline__ void sky_store(const SkyConst64 &k, SkyConst32 *out) {
  SkyConst32 c;
  c.nx = df_from_double(k.nx);  // the tables carry the factor AU/c
  c.nyp = df_from_double(k.nyp);
  c.nz = df_from_double(k.nz);
  c.ca = (float)k.ca;
  c.sa = (float)k.sa;
  c.rcd = (float)k.rcd;
  c.zsd = (float)k.zsd;
  for (int i = 0; i < 5; i++) c.ea[i] = (float)k.ea[i];
  for (int i = 0; i < 4; i++) c.eb[i] = (float)k.eb[i];
  c.ca2 = df_from_double(k.ca);
  c.sa2 = df_from_double(k.sa);
  c.rcd2 = df_from_double(k.rcd);
  c.zsd2 = df_from_double(k.zsd);
  *out = c;
}

constexpr int kSetupThreads = 64;

template <typename Sky>
__global__ void __launch_bounds__(kSetupThreads) k_setup(const double *alpha, const double *delta, int nsky,
                                                         int sky_blocks, SegGeom g, DetConst dk, Sky *sky,
                                                         const double *f1, int64_t nf1, float2 *f1df,
                                                         unsigned long long *ncand, unsigned *done) {
  pdl_wait();
  if ((int)blockIdx.x < sky_blocks) {
    const int64_t i = blockIdx.x * (int64_t)kSetupThreads + threadIdx.x;
    const int64_t s = min(i >> 1, (int64_t)nsky - 1);
    double sn, cs;
    sincos((i & 1) ? delta[s] : alpha[s], &sn, &cs);
    const double sn2 = __shfl_xor_sync(kFull, sn, 1), cs2 = __shfl_xor_sync(kFull, cs, 1);
    if (!(i & 1) && (i >> 1) < nsky) {
      SkyConst64 k;
      sky_constants_k(cs, sn, cs2, sn2, dk, g, &k);
      sky_store(k, sky + s);
      if (done) done[s] = 0;
    }
    return;
  }
  const int64_t i = (int64_t)(blockIdx.x - sky_blocks) * kSetupThreads + threadIdx.x;
  if (i == 0 && ncand) *ncand = 0;
  if (i < nf1) {
    const df32 d = df_from_double(f1[i]);
    f1df[i] = make_float2(d.hi, d.lo);
  }
}

template <typename Sky>
static cudaError_t setup_search(const fs_ctx *ctx, const double *alpha, const double *delta, int nsky,
                                const SegGeom &g, Sky *sky, const double *f1, int64_t nf1, float2 *f1df,
                                int64_t *ncand, unsigned *done, cudaStream_t st) {
  const int sb = (int)((2 * (int64_t)nsky + kSetupThreads - 1) / kSetupThreads);
  const int64_t fb = (std::max<int64_t>(nf1, 1) + kSetupThreads - 1) / kSetupThreads;
  k_setup<Sky><<<(unsigned)(sb + fb), kSetupThreads, 0, st>>>(alpha, delta, nsky, sb, g, *ctx->detk, sky, f1, nf1,
                                                             f1df, (unsigned long long *)ncand, done);
  return cudaGetLastError();
}

__global__ void k_det_const(fs_detector det, DetConst *out) { *out = det_const(det); }

fs_status device_det_const(const fs_detector &det, DetConst *out) {
  DetConst *d = nullptr;
  if (cudaMalloc(&d, sizeof(DetConst)) != cudaSuccess) {
    cudaGetLastError();
    return FS_ERR_NOMEM;
  }
  k_det_const<<<1, 1>>>(det, d);
  const bool ok = cudaGetLastError() == cudaSuccess &&
                  cudaMemcpy(out, d, sizeof(DetConst), cudaMemcpyDeviceToHost) == cudaSuccess;
  cudaFree(d);
  return ok ? FS_OK : FS_ERR_CUDA;
}

cudaError_t setup_search64(const fs_ctx *ctx, const double *alpha, const double *delta, int nsky, const SegGeom &g,
                           SkyConst64 *sky, int64_t *ncand, cudaStream_t st) {
  return setup_search(ctx, alpha, delta, nsky, g, sky, nullptr, 0, nullptr, ncand, nullptr, st);
}

// ------------------------------------------------------------------ A1: resample + demodulate one sky
// EPH: the delay from the caller's position table (eph0..2: r_m as double-floats
// and v_m on the grid) in place of the analytic orbit and rotation terms.
template <int INTERP, bool EPH>
__global__ void __launch_bounds__(256) k_demod32(DemodArgs A) {
  pdl_wait();
  const int s = blockIdx.y;
  const SkyConst32 K = A.sky[s];
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  float a2 = 0.f, b2 = 0.f;
  if (j < A.npad) {
    float2 oa = make_float2(0.f, 0.f), ob = oa, oq = oa;
    if (j < A.g.n) {
      const ResampledSample r = resample_sample<INTERP, EPH>(A, K, j);
      a2 = r.av * r.av;
      b2 = r.bv * r.bv;
      // 7) heterodyne exp(-2 pi i fl phi_m(t_j))
      const float2 h = expm2pi(df_mul_frac(A.fl, r.phim));
      oa = make_float2(r.xr * r.av * h.x, r.xr * r.av * h.y);
      ob = make_float2(r.xr * r.bv * h.x, r.xr * r.bv * h.y);
      oq = make_float2(r.Q.hi, r.Q.lo);
      if (A.tsrc && s == 0) A.tsrc[j] = (double)r.m1 * A.g.dt + (double)r.tau;
    }
    A.ya[s * A.stride + j] = oa;
    A.yb[s * A.stride + j] = ob;
    A.qq[s * A.stride + j] = oq;
  }
  // deterministic block sums of a^2, b^2 by pairwise trees in FP32 (relative error
  // below 8 roundings of the 256 positive terms); the blocks are summed in FP64 by
  // k_demod_finalize.  (FP64 here would cost half the kernel: its pipe runs at 1/64
  // of the FP32 rate on this GPU.)
  for (int o = 16; o > 0; o >>= 1) {
    a2 += __shfl_down_sync(kFull, a2, o);
    b2 += __shfl_down_sync(kFull, b2, o);
  }
  __shared__ float wa[8], wb[8];
  if ((threadIdx.x & 31) == 0) { wa[threadIdx.x >> 5] = a2; wb[threadIdx.x >> 5] = b2; }
  __syncthreads();
  if (threadIdx.x == 0) {
    const float sa = ((wa[0] + wa[1]) + (wa[2] + wa[3])) + ((wa[4] + wa[5]) + (wa[6] + wa[7]));
    const float sb = ((wb[0] + wb[1]) + (wb[2] + wb[3])) + ((wb[4] + wb[5]) + (wb[6] + wb[7]));
    A.partial[(int64_t)s * gridDim.x + blockIdx.x] = make_float2(sa, sb);
  }
}

// <a^2>, <b^2> over the n output samples and the F normalisation (cF / <a^2>, cF / <b^2>)
// of one sky with cF = 2 dt^2 / (S0 To) = 2 dt / (S0 n), from its nb block sums, by all
// threads of a block (a multiple of 32, at most 256).  Latency bound: the sums meet through
// warp shuffles and one exchange (a tree of eight shared-memory steps and four divisions in
// one thread took 4.3 us).
__device__ __forceinline__ void finish_sky(const float2 *partial, int nb, int64_t n, double dt, double S0, float2 *norm,
                                           double2 *ab2) {
  double sa = 0.0, sb = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    const float2 v = __ldcg(partial + i);  // (written by other blocks of this launch)
    sa += v.x;
    sb += v.y;
  }
  for (int o = 16; o > 0; o >>= 1) {
    sa += __shfl_down_sync(kFull, sa, o);
    sb += __shfl_down_sync(kFull, sb, o);
  }
  __shared__ double red[2][8];
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = sa; red[1][threadIdx.x >> 5] = sb; }
  __syncthreads();
  if (threadIdx.x < 2) {  // thread 0: signal a, thread 1: signal b
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += red[threadIdx.x][w];
    if (norm) (&norm->x)[threadIdx.x] = (float)(2.0 * dt / (S0 * t));  // cF / (t / n)
    if (ab2) (&ab2->x)[threadIdx.x] = t / (double)n;
  }
}

// After k_demod32, one block per sky; the blocks also clear the transform queue's counters.
__global__ void __launch_bounds__(256) k_demod_finalize(const float2 *partial, int nb, int64_t n, double dt,
                                                        double S0, float2 *norm, double2 *ab2, unsigned *ctr,
                                                        int64_t nctr) {
  pdl_wait();
  const int s = blockIdx.x;
  for (int64_t i = (int64_t)s * 256 + threadIdx.x; i < nctr; i += (int64_t)gridDim.x * 256) ctr[i] = 0;
  finish_sky(partial + (int64_t)s * nb, nb, n, dt, S0, norm ? norm + s : nullptr, ab2 ? ab2 + s : nullptr);
}

// ------------------------------------------------------------------ A1 by nodes
// The delay phi_m(t_j) of an output sample, and a and b at its source time, vary a few
// times per day: over a block of at most 512 s they are their interpolating polynomials
// through 6 Chebyshev nodes (error below (Omega_r 256 s)^6 / (6! 2^5) = 2e-15 of the
// diurnal delay's 0.02 s, (2 Omega_r 256 s)^6 / (6! 2^5) = 1e-13 of a, b).  k_demod_nodes
// solves Eq. (eq:Bt) at the nodes only, k_demod_poly evaluates three polynomials per
// sample, and with tau = j dt and t_j = tau - phi the spindown argument is
// Q_j = t_j (t_j/2 + phi) = (tau^2 - phi^2) / 2.
// Per sample ~190 instructions instead of ~430 (k_demod32, which solves for every sample
// and stays for position tables, the nearest-neighbour resampler and sampling intervals
// above 16 s).  The delay is more accurate than one FP32 Newton step's (1e-12 against 1e-9
// s): F's error against 64 bits falls from 1.9e-6 to 5e-7.  k_demod_poly is bound by issue
// (0.66 of the slots; 24 warps per SM) beside 24 bytes of output per sample that spill
// past L2 (2.4 TB/s).  Measured, 256 sky positions x 86,164 samples: 22 us at the nodes and
// 173 us per sample (193 us with one sample per thread), 244 + 6 us with k_demod32; 1024 x
// 43,082: 63 + 347 us, 494 + 20 us before.  One sky position takes 2 us longer (a launch
// more; the path does not hang on the number of positions, so that F does not either).
size_t demod_nodes_bytes(const fs_seg *seg) {
  const int K = seg->d.precision == FS_PREC_F32 && seg->d.interp == FS_INTERP_SPLINE2X ? dem_block(seg->g.dt) : 0;
  if (!K) return 0;
  const size_t nb = (size_t)((seg->g.n + K - 1) / K);
  return nb * 8 * (2 * sizeof(float4) + sizeof(float2)) + 64 * sizeof(float2);
}

DemNodes demod_nodes(const fs_seg *seg) {
  DemNodes d;
  if (!seg->demn) {
    d.lam = d.tht = nullptr;
    d.wlag = d.lag = nullptr;
    return d;
  }
  d.K = dem_block(seg->g.dt);
  d.nb = (int)((seg->g.n + d.K - 1) / d.K);
  const float4 *b = (const float4 *)seg->demn;
  d.lam = b;
  d.tht = b + (size_t)d.nb * 8;
  d.wlag = (const float2 *)(d.tht + (size_t)d.nb * 8);
  d.lag = d.wlag + (size_t)d.nb * 8;
  return d;
}

__device__ inline double dem_place(int q) { return -cospi((2 * q + 1) / (2.0 * kDemNodes)); }

__global__ void k_demod_node_tables(SegGeom g, DemNodes d) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)d.nb * 8) return;
  const int64_t b = i >> 3;
  const int q = (int)(i & 7) < kDemNodes ? (int)(i & 7) : 0;
  // Lagrange polynomial l_q in powers of s
  double c[kDemNodes] = {1.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int deg = 0;
  for (int j = 0; j < kDemNodes; j++) {
    if (j == q) continue;
    const double sj = dem_place(j), inv = 1.0 / (dem_place(q) - sj);
    deg++;
    for (int m = deg; m >= 0; m--) c[m] = ((m > 0 ? c[m - 1] : 0.0) - sj * c[m]) * inv;
  }
  auto two = [](double x) {
    const df32 v = df_from_double(x);
    return make_float2(v.hi, v.lo);
  };
  const double t = ((double)(b * d.K) + 0.5 * (d.K - 1) + dem_place(q) * (0.5 * d.K)) * g.dt;
  double sl, cl, sth, cth, w = 0.0;
  sincos(g.lambda0 + kOmegaO * t, &sl, &cl);
  sincos(g.theta0 + kOmegaR * t, &sth, &cth);
  const float2 x = two(kAUls * cl), y = two(kAUls * sl), u = two(cth), v = two(sth);
  ((float4 *)d.lam)[i] = make_float4(x.x, x.y, y.x, y.y);
  ((float4 *)d.tht)[i] = make_float4(u.x, u.y, v.x, v.y);
  const int64_t have = g.n - b * d.K < d.K ? g.n - b * d.K : d.K;
  for (int64_t j = 0; j < have; j++) {
    const double s1 = (2.0 * j + 1.0) / d.K - 1.0;
    double p = c[kDemNodes - 1];
    for (int m = kDemNodes - 2; m >= 0; m--) p = fma(p, s1, c[m]);
    w += p;
  }
  ((float2 *)d.wlag)[i] = make_float2((i & 7) < kDemNodes ? (float)w : 0.f, 0.f);
  if (b == 0)
    for (int m = 0; m < 8; m++)
      ((float2 *)d.lag)[i * 8 + m] = m < kDemNodes && i < kDemNodes ? two(c[m]) : make_float2(0.f, 0.f);
}

cudaError_t demod_node_tables(const fs_seg *seg, cudaStream_t st) {
  const DemNodes d = demod_nodes(seg);
  const int64_t n = (int64_t)d.nb * 8;
  k_demod_node_tables<<<(unsigned)((n + 63) / 64), 64, 0, st>>>(seg->g, d);
  return cudaGetLastError();
}

// Eight lanes per (sky, block): lane q < 6 solves t + phi_m(t) = tau at node q, two FP32
// evaluations of phi = f(phi) = phi_m(tau - phi) from phi = 0 (each takes the error down by
// |d phi_m/dt| < 1.1e-4) and one in double-float with a Newton step (left: 1e-18 s); then
// lane m forms the coefficients of s^m.  The sums of a^2, b^2 are the nodes' own, with the
// weights of the samples they stand for.
// SETUP: a search of few sky positions (kSetupSkies) without k_setup: every block takes the
// constants of its sky itself (two lanes, two sines and cosines in FP64: ~2 us of latency,
// against a launch of its own), the grid converts the spindowns and clears the candidate
// count, and the finished-block counters are the context's own, left at zero by the last
// block.
struct SetupArgs {
  const double *alpha, *delta, *f1;
  int64_t nf1;
  float2 *f1df;
  unsigned long long *ncand;
  DetConst dk;
};
constexpr int kSetupSkies = 16;

template <bool SETUP>
__global__ void __launch_bounds__(128) k_demod_nodes(DemodArgs A, SetupArgs U) {
  pdl_wait();
  const int sky = blockIdx.y;
  __shared__ SkyConst32 sk;
  if constexpr (SETUP) {
    if (threadIdx.x < 32) {
      double sn = 0.0, cs = 1.0;
      if (threadIdx.x < 2) sincos(threadIdx.x ? U.delta[sky] : U.alpha[sky], &sn, &cs);
      const double sd = __shfl_sync(kFull, sn, 1), cd = __shfl_sync(kFull, cs, 1);
      if (threadIdx.x == 0) {
        SkyConst64 k;
        sky_constants_k(cs, sn, cd, sd, U.dk, A.g, &k);
        sky_store(k, &sk);
      }
    }
    const int64_t i = ((int64_t)sky * gridDim.x + blockIdx.x) * 128 + threadIdx.x;
    if (i == 0) *U.ncand = 0;
    for (int64_t q = i; q < U.nf1; q += (int64_t)gridDim.x * gridDim.y * 128) {
      const df32 d = df_from_double(U.f1[q]);
      U.f1df[q] = make_float2(d.hi, d.lo);
    }
    __syncthreads();
  }
  for (int64_t c = ((int64_t)sky * gridDim.x + blockIdx.x) * 128 + threadIdx.x; c < A.nctr;
       c += (int64_t)gridDim.x * gridDim.y * 128)
    A.ctr[c] = 0;
  const int i = blockIdx.x * 128 + threadIdx.x;
  const int b = i >> 3, q = i & 7;
  const bool in = b < A.nodes.nb;
  const int node = (in ? b : 0) * 8 + q;
  const SkyConst32 K = SETUP ? sk : A.sky[sky];
  const float4 Lm = A.nodes.lam[node], Th = A.nodes.tht[node];
  const df32 C{Lm.x, Lm.y}, S{Lm.z, Lm.w}, ct{Th.x, Th.y}, sn{Th.z, Th.w};
  // orbit P = n0 . (C, S), its derivative with the longitude R; cos, sin of alpha - theta
  const df32 P = df_add(df_mul(K.nx, C), df_mul(K.nyp, S)), R = df_sub(df_mul(K.nx, S), df_mul(K.nyp, C));
  const df32 cx = df_add(df_mul(K.ca2, ct), df_mul(K.sa2, sn)), sx = df_sub(df_mul(K.sa2, ct), df_mul(K.ca2, sn));
  constexpr float wo = (float)kOmegaO, wr = (float)kOmegaR;
  float ph = P.hi + fmaf(K.rcd, cx.hi, K.zsd);
  {
    const float eo = wo * ph, er = wr * ph, c1 = fmaf(-0.5f * er, er, 1.f), s1 = er - er * er * er * (1.f / 6.f);
    ph = fmaf(eo, R.hi, fmaf(-0.5f * eo * eo, P.hi, P.hi)) + fmaf(K.rcd, fmaf(cx.hi, c1, -sx.hi * s1), K.zsd);
  }
  // at source time t = tau - ph: longitude and sidereal angle turned back by Omega ph
  const df32 eo = df_mul_f(df_from_double(kOmegaO), ph), er = df_mul_f(df_from_double(kOmegaR), ph);
  const df32 orb = df_add(P, df_add_f(df_mul(eo, R), -0.5f * eo.hi * eo.hi * (P.hi + eo.hi * R.hi * (1.f / 3.f))));
  const df32 er2 = df_mul(er, er);
  const df32 ce = df_add_f(df_scale(er2, -0.5f), er2.hi * er2.hi * (1.f / 24.f));                // cos - 1
  const df32 se = df_add_f(er, er.hi * er2.hi * fmaf(er2.hi, 1.f / 120.f, -1.f / 6.f));
  const df32 cxt = df_add(cx, df_sub(df_mul(cx, ce), df_mul(sx, se)));
  const df32 sxt = df_add(sx, df_add(df_mul(sx, ce), df_mul(cx, se)));
  const df32 f = df_add(orb, df_add(df_mul(K.rcd2, cxt), K.zsd2));
  const float phidot = fmaf(-wo, R.hi - eo.hi * P.hi, K.rcd * wr * sxt.hi);  // d phi_m / dt at t
  const df32 r = df_add_f(f, -ph);
  const float dl = (r.hi + r.lo) / (1.f + phidot);
  const df32 phi = df_add_f(df32{ph, 0.f}, dl);  // t moved by -dl
  const float eta = -wr * dl;
  const float cj = fmaf(sxt.hi, eta, cxt.hi), sj = fmaf(-cxt.hi, eta, sxt.hi);
  const float c2 = fmaf(cj, cj, -sj * sj), s2 = 2.f * sj * cj;
  const float av = fmaf(K.ea[0], c2, fmaf(K.ea[1], s2, fmaf(K.ea[2], cj, fmaf(K.ea[3], sj, K.ea[4]))));
  const float bv = fmaf(K.eb[0], c2, fmaf(K.eb[1], s2, fmaf(K.eb[2], cj, K.eb[3] * sj)));
  // coefficients: of phi relative to node 2
  const df32 ref{__shfl_sync(kFull, phi.hi, 2, 8), __shfl_sync(kFull, phi.lo, 2, 8)};
  const df32 d = df_sub(phi, ref);
  df32 cphi{0.f, 0.f};
  float ca = 0.f, cb = 0.f;
#pragma unroll
  for (int n = 0; n < kDemNodes; n++) {
    const float2 l = A.nodes.lag[n * 8 + q];
    const df32 dn{__shfl_sync(kFull, d.hi, n, 8), __shfl_sync(kFull, d.lo, n, 8)};
    cphi = df_add(cphi, df_mul(df32{l.x, l.y}, dn));
    ca = fmaf(l.x, __shfl_sync(kFull, av, n, 8), ca);
    cb = fmaf(l.x, __shfl_sync(kFull, bv, n, 8), cb);
  }
  if (q == 0) cphi = df_add(cphi, ref);
  const float w = A.nodes.wlag[node].x;
  float sa = w * av * av, sb = w * bv * bv;
  for (int o = 4; o > 0; o >>= 1) {
    sa += __shfl_down_sync(kFull, sa, o, 8);
    sb += __shfl_down_sync(kFull, sb, o, 8);
  }
  if (in) {
    // [0, 8): c0 hi, lo, c1 hi, lo, c2 .. c5 of phi; [8, 14) of a, [14, 20) of b
    float *o = (float *)(A.dcoef + ((int64_t)sky * A.nodes.nb + b) * kDemCoef);
    if (q < 2) {
      o[2 * q] = cphi.hi;
      o[2 * q + 1] = cphi.lo;
    } else if (q < kDemNodes) {
      o[2 + q] = cphi.hi;
    }
    if (q < kDemNodes) {
      o[8 + q] = ca;
      o[14 + q] = cb;
    }
    if (q == 0) A.partial[(int64_t)sky * A.nodes.nb + b] = make_float2(sa, sb);
  }
  // the sky's last block forms its normalisation (in block order: the same sums every time)
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(A.done + sky, 1u) == gridDim.x - 1;
    if (SETUP && last) A.done[sky] = 0;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  finish_sky(A.partial + (int64_t)sky * A.nodes.nb, A.nodes.nb, A.g.n, A.g.dt, A.g.S0, A.norm ? A.norm + sky : nullptr,
             A.ab2 ? A.ab2 + sky : nullptr);
}

// Two neighbouring samples per thread: one set of coefficients, two independent gathers in
// flight, 16-byte stores.
__global__ void __launch_bounds__(256) k_demod_poly(DemodArgs A) {
  pdl_wait();
  const int s = blockIdx.y;
  const int j0 = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);  // FP32 series hold at most 2^20 samples
  if (j0 >= (int)A.npad) return;
  const int n = (int)A.g.n, K = A.nodes.K;
  float4 oa = make_float4(0.f, 0.f, 0.f, 0.f), ob = oa, oq = oa;
  if (j0 < n) {
    const float4 *cf = A.dcoef + ((int64_t)s * A.nodes.nb + j0 / K) * kDemCoef;
    const float4 f0 = cf[0], f1 = cf[1], a0 = cf[2], ab = cf[3], b1 = cf[4];
    const float inv_k = 1.f / (float)K;
    float2 ra[2], rb[2], rq[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int j = j0 + h, jj = j & (K - 1);
      ra[h] = rb[h] = rq[h] = make_float2(0.f, 0.f);
      const float u = fmaf((float)(2 * jj + 1), inv_k, -1.f);  // exact
      const float p = f0.z * u, hi = u * u * fmaf(u, fmaf(u, fmaf(u, f1.w, f1.z), f1.y), f1.x);
      const df32 ps = two_sum(f0.x, p);
      const df32 phi = quick_two_sum(ps.hi, ps.lo + (f0.y + (fmaf(f0.z, u, -p) + fmaf(f0.w, u, hi))));
      const float av = fmaf(u, fmaf(u, fmaf(u, fmaf(u, fmaf(u, ab.y, ab.x), a0.w), a0.z), a0.y), a0.x);
      const float bv = fmaf(u, fmaf(u, fmaf(u, fmaf(u, fmaf(u, b1.w, b1.z), b1.y), b1.x), ab.w), ab.z);
      unsigned i;
      float f;
      float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
      if (spline_place(phi, A.two_over_dt2, j, n, &i, &f)) c = A.coef[i];
      const float xr = fmaf(f, fmaf(f, fmaf(f, c.w, c.z), c.y), c.x);
      const float2 e = expm2pi(df_mul_frac(A.fl, phi));  // heterodyne
      const df32 tau = df_mul_f(A.dt2, (float)j);        // exact index
      const df32 Q = df_scale(df_sub(df_mul(tau, tau), df_mul(phi, phi)), 0.5f);
      if (j < n) {
        ra[h] = make_float2(xr * av * e.x, xr * av * e.y);
        rb[h] = make_float2(xr * bv * e.x, xr * bv * e.y);
        rq[h] = make_float2(Q.hi, Q.lo);
        if (A.tsrc && s == 0) A.tsrc[j] = (double)j * A.g.dt - ((double)phi.hi + (double)phi.lo);
      }
    }
    oa = make_float4(ra[0].x, ra[0].y, ra[1].x, ra[1].y);
    ob = make_float4(rb[0].x, rb[0].y, rb[1].x, rb[1].y);
    oq = make_float4(rq[0].x, rq[0].y, rq[1].x, rq[1].y);
  }
  const int64_t o = s * A.stride + j0;  // stride and j0 are even: 16-byte aligned
  *(float4 *)(A.ya + o) = oa;
  *(float4 *)(A.yb + o) = ob;
  *(float4 *)(A.qq + o) = oq;
}

// ------------------------------------------------------------------ host orchestration
static int log2_exact(int64_t v) {
  int p = 0;
  while (p < 62 && ((int64_t)1 << p) < v) p++;
  return ((int64_t)1 << p) == v ? p : -1;
}
// Default split of a sub-transform of length 2^p: N1 = 2^ceil(p/2), N2 = 2^floor(p/2).
static FftShape default_split(int p) { return FftShape{1 << ((p + 1) / 2), 1 << (p / 2)}; }

// Transform splits N1 x N2 the library instantiates for the persistent kernel.
static const int kSplits[][2] = {
    {64, 64},    {128, 64},  {128, 128},  {256, 64},   {256, 128}, {256, 256},  {512, 128},
    {128, 512},  {512, 256}, {256, 512},  {1024, 128}, {512, 512}, {1024, 256}, {256, 1024},
    {1024, 512}, {512, 1024}, {1024, 1024}};

bool split_instantiated(int N1, int N2) {
  for (const auto &s : kSplits)
    if (s[0] == N1 && s[1] == N2) return true;
  return false;
}

cudaError_t dispatch_passes(int N1, int N2, const Pass1Args &a1, const Pass2Args &a2, const QueueArgs &qa,
                            const QueueStream &st) {
  const int64_t nf = (int64_t)N1 * N2;
  if (nf <= (1 << 16)) return dispatch_passes_small(N1, N2, a1, a2, qa, st);
  if (nf <= (1 << 18)) return dispatch_passes_mid(N1, N2, a1, a2, qa, st);
  return dispatch_passes_large(N1, N2, a1, a2, qa, st);
}
int passes_blocks_per_sm(int N1, int N2) {
  const int64_t nf = (int64_t)N1 * N2;
  if (nf <= (1 << 16)) return passes_blocks_per_sm_small(N1, N2);
  if (nf <= (1 << 18)) return passes_blocks_per_sm_mid(N1, N2);
  return passes_blocks_per_sm_large(N1, N2);
}

// Sub-transform split: 2^vshift sub-transforms of at most 2^20 points.
static bool sub_transform(int64_t nfft, int *vshift, int *psub) {
  const int p = log2_exact(nfft);
  if (p < 12 || p > 21) return false;
  *vshift = p > 20 ? p - 20 : 0;
  *psub = p - *vshift;
  return true;
}

bool tuning_valid(int64_t nfft, const fs_tuning &t) {
  int vs = 0, ps = 0;
  if (!sub_transform(nfft, &vs, &ps)) return false;
  if (t.n1 < 0 || t.queue_round < 0 || t.queue_lag < 0 || t.group_skies < 0) return false;
  if (t.queue_lag > 64 || t.queue_round > 4096) return false;
  if (t.n1 == 0) return true;
  const int64_t ns = (int64_t)1 << ps;
  return ns % t.n1 == 0 && split_instantiated(t.n1, (int)(ns / t.n1));
}

static QueueShape queue_shape(const fs_ctx *ctx, const fs_tuning *t, const FftShape &sh) {
  QueueShape q{};
  queue_tiles(sh.N1, sh.N2, kPersistThreads, &q.tiles1, &q.tiles2);
  const int nsm = ctx->nsm;
  int bps = passes_blocks_per_sm(sh.N1, sh.N2);
  if (bps < 1) bps = 1;
  const int ctas = bps * (nsm > 0 ? nsm : 1);
  const int qr = (t && t->queue_round > 0) ? t->queue_round : ctx->queue_round;
  // a round's pass-1 items: a little more than the resident CTAs.  A template's second pass
  // comes a round after its first, so the round has to outlast the items in flight; the
  // ring of lag + 2 rounds should stay in L2 (100 MB at 1.15 x for 2^18).  Measured at 0.85
  // / 1.15 / 1.3 / 1.6 x: 2-day grid (3 CTAs per SM) 9.03 / 8.94 / 8.98 / 9.36 ms,
  // interbinning 2.04 / 1.90 / 1.89 / 1.89, 2^20 segments (2 CTAs per SM, 1, 1, 2 and 2
  // templates) 8.74 / 8.70 / 8.52 / 8.60, 2^21 7.22 / 7.22 / 7.18 / 7.18.
  q.kr = qr > 0 ? qr : (int)((bps >= 3 ? 1.15 : 1.3) * ctas / q.tiles1 + 0.5);
  if (q.kr < 1) q.kr = 1;
  const int lg = (t && t->queue_lag > 0) ? t->queue_lag : ctx->queue_lag;
  q.lag = lg > 0 ? lg : 1;
  const int need = (q.lag + 2) * q.kr;
  q.slots = ctx->z_slots > need ? ctx->z_slots : need;
  return q;
}

fs_status config32(const fs_ctx *ctx, const fs_seg *seg, int nsky, int64_t nbins, Cfg32 *c) {
  int ps = 0;
  if (!sub_transform(seg->g.nfft, &c->vshift, &ps)) return FS_ERR_SHAPE;
  c->nsub = (int64_t)1 << ps;
  if (seg->g.n > c->nsub) return FS_ERR_SHAPE;
  const int p = ps + c->vshift;
  const fs_tuning *t = ctx->tuned[p] ? &ctx->tune[p] : nullptr;
  c->sh = default_split(ps);
  // interbinning with an odd power: the split with the shorter first pass where its
  // items are built (2^17: 256 x 512 measured 15% faster than 512 x 256)
  if ((seg->d.options & FS_OPT_INTERBIN) && (ps & 1) && passes_ib_instantiated(c->sh.N1 / 2, c->sh.N2 * 2))
    c->sh = FftShape{c->sh.N1 / 2, c->sh.N2 * 2};
  if (t && t->n1 > 0) c->sh = FftShape{t->n1, (int)(c->nsub / t->n1)};
  c->n1max = (int)((seg->g.n + c->sh.N2 - 1) / c->sh.N2);
  c->npad = (int64_t)c->n1max * c->sh.N2;
  const int gsk = (t && t->group_skies > 0) ? t->group_skies : ctx->group_skies;
  c->G = gsk < nsky ? gsk : nsky;
  c->interbin = (seg->d.options & FS_OPT_INTERBIN) != 0;
  if (c->interbin && (c->vshift || nbins != seg->g.nfft)) return FS_ERR_SHAPE;
  c->full = (nbins == seg->g.nfft);
  // interbinning runs from the persistent queue for the splits built with its items
  c->persistent = ctx->persistent && (c->interbin ? passes_ib_instantiated(c->sh.N1, c->sh.N2) : !c->full);
  c->qs = queue_shape(ctx, t, c->sh);
  c->B = c->persistent ? c->qs.slots : ctx->batch_templates;
  return FS_OK;
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

fs_status workspace32(fs_ctx *ctx, int slot, const fs_seg *seg, const Cfg32 &c, int nsky, int nspin,
                      bool may_alloc, cudaStream_t st, Ws32 *w) {
  if (slot < 0 || slot >= fs_ctx::kWsSlots) return FS_ERR_ARG;
  const int G = c.G;
  const int64_t stride = (c.npad + 63) & ~(int64_t)63;
  const DemNodes dn = demod_nodes(seg);
  const int nblk = dn.K ? dn.nb : (int)((c.npad + 255) / 256);
  const size_t vt = ((size_t)G * nspin) << c.vshift;  // virtual templates of a group
  size_t off = 0;
  size_t o_sky = off; off = align256(off + sizeof(SkyConst32) * (nsky > G ? nsky : G));
  size_t o_ya = off; off = align256(off + sizeof(float2) * stride * G);
  size_t o_yb = off; off = align256(off + sizeof(float2) * stride * G);
  size_t o_qq = off; off = align256(off + sizeof(float2) * stride * G);
  size_t o_nm = off; off = align256(off + sizeof(float2) * G);
  size_t o_ab = off; off = align256(off + sizeof(double2) * G);
  size_t o_pa = off; off = align256(off + sizeof(float2) * (size_t)nblk * G);
  size_t o_dc = off; off = align256(off + sizeof(float4) * kDemCoef * (size_t)(dn.K ? dn.nb : 0) * G);
  size_t o_dn = off; off = align256(off + sizeof(unsigned) * (size_t)nsky);
  size_t o_f1 = off; off = align256(off + sizeof(float2) * (size_t)nsky * nspin);
  const size_t gb = kDebug ? kGuardBytes : 0;  // debug builds: guard words around the ring
  size_t o_g0 = off; off = align256(off + gb);
  size_t o_z = off; off = align256(off + sizeof(float2) * 2 * (size_t)c.nsub * c.B);
  size_t o_g1 = off; off = align256(off + gb);
  const size_t xn = !c.interbin ? 0
                    : c.persistent ? vt * (size_t)ib_edge_stride(c.sh.N1, c.sh.N2, kPersistThreads)
                                   : 2 * (size_t)c.nsub * c.B;
  size_t o_x = off; off = align256(off + sizeof(float2) * xn);
  size_t o_ct = off; off = align256(off + sizeof(unsigned) * (1 + 2 * vt));
  size_t o_g2 = off; off = align256(off + gb);
  if (may_alloc) {
    fs_status s = ensure_buffer(&ctx->ws[slot], &ctx->ws_bytes[slot], off, st);
    if (s != FS_OK) return s;
  } else if (ctx->ws_bytes[slot] < off || !ctx->ws[slot]) {
    return FS_ERR_NOMEM;
  }
  char *base = (char *)ctx->ws[slot];
  w->skyc = (SkyConst32 *)(base + o_sky);
  w->ya = (float2 *)(base + o_ya);
  w->yb = (float2 *)(base + o_yb);
  w->qq = (float2 *)(base + o_qq);
  w->norm = (float2 *)(base + o_nm);
  w->ab2 = (double2 *)(base + o_ab);
  w->partial = (float2 *)(base + o_pa);
  w->dcoef = (float4 *)(base + o_dc);
  w->done = (unsigned *)(base + o_dn);
  w->f1df = (float2 *)(base + o_f1);
  w->Z = (float2 *)(base + o_z);
  w->X = c.interbin ? (float2 *)(base + o_x) : nullptr;
  w->counters = (unsigned *)(base + o_ct);
  w->small_done = ctx->small_done + slot * kSetupSkies;
  w->stride = stride;
  w->nblk_a1 = nblk;
  w->guard[0] = kDebug ? (uint32_t *)(base + o_g0) : nullptr;
  w->guard[1] = kDebug ? (uint32_t *)(base + o_g1) : nullptr;
  w->guard[2] = kDebug ? (uint32_t *)(base + o_g2) : nullptr;
  return FS_OK;
}

// Debug builds: fill the guard words of a workspace before a search and check
// them after it (an overwritten word latches ERRF_CORRUPT).
__global__ void k_guard(uint32_t *g0, uint32_t *g1, uint32_t *g2, int check, uint32_t *flags) {
  constexpr int W = (int)(kGuardBytes / sizeof(uint32_t));
  uint32_t *g[3] = {g0, g1, g2};
  for (int i = threadIdx.x; i < 3 * W; i += blockDim.x) {
    uint32_t *p = g[i / W] + (i % W);
    if (!check) *p = kGuardWord;
    else if (*p != kGuardWord) atomicOr(flags, ERRF_CORRUPT);
  }
}

static cudaError_t guards(const Ws32 &w, bool check, uint32_t *flags, cudaStream_t st) {
  if (!w.guard[0]) return cudaSuccess;
  k_guard<<<1, 256, 0, st>>>(w.guard[0], w.guard[1], w.guard[2], check ? 1 : 0, flags);
  return cudaGetLastError();
}

static DemodArgs demod_args(const fs_seg *seg, const Ws32 &w, int64_t npad) {
  DemodArgs A{};
  A.g = seg->g;
  A.dt2 = df_from_double(seg->g.dt);
  A.dt = (float)seg->g.dt;
  A.inv_dt = (float)(1.0 / seg->g.dt);
  A.two_over_dt = (float)(2.0 / seg->g.dt);
  A.fl = df_from_double(seg->g.fl);
  A.sky = w.skyc;
  A.tab0 = seg->tab0;
  A.tab1 = seg->tab1;
  A.eph0 = seg->eph0;
  A.eph1 = seg->eph1;
  A.eph2 = seg->eph2;
  A.coef = (const float4 *)seg->coef;
  A.x32 = seg->x32;
  A.ya = w.ya;
  A.yb = w.yb;
  A.qq = w.qq;
  A.stride = w.stride;
  A.npad = npad;
  A.partial = w.partial;
  A.tsrc = nullptr;
  A.nodes = demod_nodes(seg);
  A.dcoef = w.dcoef;
  A.done = w.done;
  A.norm = w.norm;
  A.ab2 = w.ab2;
  A.ctr = nullptr;
  A.nctr = 0;
  A.two_over_dt2 = df_from_double(2.0 / seg->g.dt);
  return A;
}

// One group of skies: demodulation, normalisation (A.norm, A.ab2) and the transform queue's
// counters (A.ctr).  Returns the launches in *launches.
// setup: NULL, or what a search of few sky positions hands to k_demod_nodes.
static cudaError_t launch_demod(const DemodArgs &A, int nsky, int nblk_sums, int interp, int64_t *launches,
                                cudaStream_t st, const SetupArgs *setup = nullptr) {
  const int nblk = (int)((A.npad + 255) / 256);
  *launches += 2;
  if (A.nodes.K) {
    const dim3 grid((unsigned)((A.nodes.nb * 8 + 127) / 128), nsky);
    const cudaError_t e = launch_pdl(setup ? k_demod_nodes<true> : k_demod_nodes<false>, grid, dim3(128), 0, st, A,
                                     setup ? *setup : SetupArgs{});
    return e == cudaSuccess ? launch_pdl(k_demod_poly, dim3((nblk + 1) / 2, nsky), dim3(256), 0, st, A) : e;
  }
  const bool eph = A.eph0 != nullptr;
  auto kern = interp == FS_INTERP_NEAREST ? (eph ? k_demod32<FS_INTERP_NEAREST, true> : k_demod32<FS_INTERP_NEAREST, false>)
                                          : (eph ? k_demod32<FS_INTERP_SPLINE2X, true> : k_demod32<FS_INTERP_SPLINE2X, false>);
  const cudaError_t e = launch_pdl(kern, dim3(nblk, nsky), dim3(256), 0, st, A);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_demod_finalize, dim3(nsky), dim3(256), 0, st, A.partial, nblk_sums, A.g.n, A.g.dt, A.g.S0, A.norm,
                    A.ab2, A.ctr, A.nctr);
}

static void pass_args(const fs_seg *seg, const Cfg32 &c, const Ws32 &w, int nspin, float thr,
                      fs_candidate *cand, int64_t cap, int64_t *ncand, uint32_t *flags, Pass1Args *p1,
                      Pass2Args *p2) {
  *p1 = Pass1Args{};
  p1->ya = w.ya;
  p1->yb = w.yb;
  p1->qq = w.qq;
  p1->sky_stride = w.stride;
  p1->f1df = w.f1df;  // filled by k_setup or k_demod_nodes<true> before the transform
  p1->nspin = nspin;
  p1->nspin_fd = make_fastdiv((uint32_t)nspin);
  p1->N2 = c.sh.N2;
  p1->n1max = c.n1max;
  p1->nfft = c.nsub;
  p1->vshift = c.vshift;
  p1->inv_nfft_total = (float)(1.0 / (double)seg->g.nfft);
  p1->Z = w.Z;
  p1->z_elems = 2 * c.nsub * (int64_t)c.B;
  p1->yq_elems = w.stride * (int64_t)c.G;
  p1->flags = flags;
  *p2 = Pass2Args{};
  p2->Z = w.Z;
  p2->N1 = c.sh.N1;
  p2->N2 = c.sh.N2;
  p2->nfft = c.nsub;
  p2->norm = w.norm;
  p2->nspin = nspin;
  p2->nspin_fd = make_fastdiv((uint32_t)nspin);
  p2->vshift = c.vshift;
  p2->thr = thr;
  p2->cand = cand;
  p2->cap = cap;
  p2->ncand = (unsigned long long *)ncand;
  p2->flags = flags;
  p2->z_elems = 2 * c.nsub * (int64_t)c.B;
}

fs_status search32_run(fs_ctx *ctx, fs_seg *seg, const Cfg32 &c, const Ws32 &w, const double *alpha,
                       const double *delta, int nsky, const double *f1, int nspin, float thr, float *F,
                       int64_t nbins, fs_candidate *cand, int64_t cap, int64_t *ncand, cudaStream_t st,
                       const double *lat_offset) {
  if (lat_offset && !c.persistent) return FS_ERR_UNSUPPORTED;
  if (guards(w, false, ctx->d_flags, st) != cudaSuccess) return FS_ERR_CUDA;
  DemodArgs DA = demod_args(seg, w, c.npad);
  const int64_t nf1 = lat_offset ? (int64_t)nsky * nspin : nspin;
  // few sky positions and blocks: no launch of its own for the set-up (19.2 against 22.5 us
  // for one template of a 1-day series; beyond two blocks per SM the constants would be
  // taken more often than that saves)
  const bool small = DA.nodes.K && nsky <= kSetupSkies && nsky <= c.G &&
                     (int64_t)nsky * ((DA.nodes.nb * 8 + 127) / 128) <= 2 * (int64_t)ctx->nsm;
  SetupArgs su{};
  if (small) {
    su = SetupArgs{alpha, delta, f1, nf1, w.f1df, (unsigned long long *)ncand, *ctx->detk};
  } else {
    ProfScope ps(ctx, PROF_OTHER, st);
    if (setup_search(ctx, alpha, delta, nsky, seg->g, w.skyc, f1, nf1, w.f1df, ncand, w.done, st) != cudaSuccess)
      return FS_ERR_CUDA;
    ctx->launches += 1;
  }
  Pass1Args p1;
  Pass2Args p2;
  pass_args(seg, c, w, nspin, thr, cand, cap, ncand, ctx->d_flags, &p1, &p2);
  p2.nbins = nbins;
  for (int g0 = 0; g0 < nsky; g0 += c.G) {
    const int gs = (nsky - g0) < c.G ? (nsky - g0) : c.G;
    const int ntm = (gs * nspin) << c.vshift;  // virtual templates of the group
    DA.sky = w.skyc + g0;
    DA.done = small ? w.small_done : w.done + g0;
    DA.ctr = w.counters;
    DA.nctr = c.persistent ? 1 + 2 * (int64_t)ntm : 0;
    {
      NvtxRange nv("fs.demodulate");
      ProfScope ps(ctx, PROF_DEMOD, st);
      if (launch_demod(DA, gs, w.nblk_a1, seg->d.interp, &ctx->launches, st, small ? &su : nullptr) != cudaSuccess)
        return FS_ERR_CUDA;
    }
    p2.sky_base = g0;
    if (lat_offset) {  // the group's rows of per-template spindowns and bin offsets
      p1.f1df = w.f1df + (int64_t)g0 * nspin;
      p1.bin_offset = lat_offset + (int64_t)g0 * nspin;
    }
    p2.F = F ? F + (int64_t)g0 * nspin * nbins : nullptr;
    p2.f_elems = (int64_t)(nsky - g0) * nspin * nbins;
    if (c.persistent) {
      QueueArgs qa{};
      qa.ntm = ntm;
      qa.tiles1 = c.qs.tiles1;
      qa.tiles2 = c.qs.tiles2;
      qa.kr = ntm < c.qs.kr ? ntm : c.qs.kr;  // (no empty places in a round of few templates)
      qa.lag = c.qs.lag;
      qa.slots = c.qs.slots;
      qa.ipr_fd = make_fastdiv((uint32_t)(qa.kr * (qa.tiles1 + qa.tiles2)));
      qa.slots_fd = make_fastdiv((uint32_t)qa.slots);
      qa.counter = w.counters;
      {
        NvtxRange nv("fs.transform");
        ProfScope ps(ctx, PROF_PASS2, st);
        if (c.interbin) {
          p2.X = w.X;
          p2.eb_stride = ib_edge_stride(c.sh.N1, c.sh.N2, kPersistThreads);
          const bool in_queue = edges_in_queue(
              seg->d.nfft, (size_t)ntm * ((p2.F ? sizeof(float) * nbins : 0) + sizeof(float2) * p2.eb_stride));
          if ((in_queue ? dispatch_passes_ibq : dispatch_passes_ib)(
                  c.sh.N1, c.sh.N2, p1, p2, qa, QueueStream{st, &ctx->blocks_per_sm, ctx->nsm}) != cudaSuccess)
            return FS_ERR_CUDA;
          ctx->launches += !in_queue;  // the kernel of the edge bins
        } else if (lat_offset) {
          if (dispatch_passes_lat(c.sh.N1, c.sh.N2, p1, p2, qa, QueueStream{st, &ctx->blocks_per_sm, ctx->nsm}) != cudaSuccess) return FS_ERR_CUDA;
        } else if (dispatch_passes(c.sh.N1, c.sh.N2, p1, p2, qa, QueueStream{st, &ctx->blocks_per_sm, ctx->nsm}) != cudaSuccess) {
          return FS_ERR_CUDA;
        }
      }
      ctx->launches += 1;
      continue;
    }
    NvtxRange nv("fs.transform");
    for (int b0 = 0; b0 < ntm; b0 += c.B) {
      const int nb = (ntm - b0) < c.B ? (ntm - b0) : c.B;
      p1.tmpl0 = b0;
      p2.tmpl0 = b0;
      {
        ProfScope ps(ctx, PROF_PASS1, st);
        if (dispatch_pass1(c.sh.N1, p1, nb, st) != cudaSuccess) return FS_ERR_CUDA;
      }
      if (c.interbin) {
        ProfScope ps(ctx, PROF_PASS2, st);
        p2.X = w.X;
        if (dispatch_pass2x(c.sh.N2, p2, nb, st) != cudaSuccess) return FS_ERR_CUDA;
        if (launch_interbin(p2, nb, st) != cudaSuccess) return FS_ERR_CUDA;
        ctx->launches += 1;
      } else {
        ProfScope ps(ctx, PROF_PASS2, st);
        if (dispatch_pass2(c.sh.N2, c.full, p2, nb, st) != cudaSuccess) return FS_ERR_CUDA;
      }
      ctx->launches += 2;
    }
  }
  if (guards(w, true, ctx->d_flags, st) != cudaSuccess) return FS_ERR_CUDA;
  return FS_OK;
}

// Lattice templates run as lattice items of the persistent queue: the split's items
// must be built, and 2^21 takes its sub-transforms on the 1024 x 1024 split only.
bool lattice_supported(const Cfg32 &c) {
  if (c.interbin || c.full || !c.persistent || !passes_lat_instantiated(c.sh.N1, c.sh.N2)) return false;
  return !c.vshift || (c.vshift == 1 && c.sh.N1 == 1024 && c.sh.N2 == 1024);
}

fs_status search32_lattice(fs_ctx *ctx, fs_seg *seg, const double *alpha, const double *delta, int nsky,
                           const double *f1, const double *offset, int nspin, float thr, float *F, int64_t nbins,
                           fs_candidate *cand, int64_t cap, int64_t *ncand, cudaStream_t st) {
  Cfg32 c;
  fs_status s = config32(ctx, seg, nsky, nbins, &c);
  if (s != FS_OK) return s;
  if (!lattice_supported(c)) return FS_ERR_UNSUPPORTED;
  Ws32 w;
  s = workspace32(ctx, 0, seg, c, nsky, nspin, true, st, &w);
  if (s != FS_OK) return s;
  return search32_run(ctx, seg, c, w, alpha, delta, nsky, f1, nspin, thr, F, nbins, cand, cap, ncand, st, offset);
}

fs_status search32(fs_ctx *ctx, fs_seg *seg, const double *alpha, const double *delta, int nsky,
                   const double *f1, int nspin, float thr, float *F, int64_t nbins, fs_candidate *cand,
                   int64_t cap, int64_t *ncand, cudaStream_t st) {
  Cfg32 c;
  fs_status s = config32(ctx, seg, nsky, nbins, &c);
  if (s != FS_OK) return s;
  Ws32 w;
  s = workspace32(ctx, 0, seg, c, nsky, nspin, true, st, &w);
  if (s != FS_OK) return s;
  return search32_run(ctx, seg, c, w, alpha, delta, nsky, f1, nspin, thr, F, nbins, cand, cap, ncand, st);
}

// Stage access: A1 for one sky, widened to double.
__global__ void k_widen(const float2 *ya, const float2 *yb, double *oa, double *ob, int64_t n) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= n) return;
  oa[2 * j] = ya[j].x;
  oa[2 * j + 1] = ya[j].y;
  ob[2 * j] = yb[j].x;
  ob[2 * j + 1] = yb[j].y;
}

fs_status demod32_debug(fs_ctx *ctx, fs_seg *seg, double alpha, double delta, double *ya, double *yb,
                        double *tsrc, double *ab2, cudaStream_t st) {
  const int64_t n = seg->g.n;
  Cfg32 c{};
  c.G = 1;
  c.npad = n;
  c.nsub = 0;
  c.B = 0;
  Ws32 w;
  fs_status s = workspace32(ctx, 0, seg, c, 1, 1, true, st, &w);
  if (s != FS_OK) return s;
  // alpha/delta are host values: stage them through the partial buffer's tail is not
  // possible before allocation, so use a small device copy.
  double hd[2] = {alpha, delta};
  double *dd = (double *)w.ab2;  // 16 bytes, overwritten by finalize afterwards
  if (cudaMemcpyAsync(dd, hd, sizeof(hd), cudaMemcpyHostToDevice, st) != cudaSuccess) return FS_ERR_CUDA;
  if (setup_search(ctx, dd, dd + 1, 1, seg->g, w.skyc, nullptr, 0, nullptr, nullptr, w.done, st) != cudaSuccess)
    return FS_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return FS_ERR_CUDA;  // hd is on the stack
  DemodArgs A = demod_args(seg, w, n);
  A.npad = (n + 1) & ~(int64_t)1;  // whole pairs (the stride holds them)
  A.tsrc = tsrc;
  A.norm = nullptr;
  A.ab2 = (double2 *)ab2;
  if (launch_demod(A, 1, w.nblk_a1, seg->d.interp, &ctx->launches, st) != cudaSuccess) return FS_ERR_CUDA;
  k_widen<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w.ya, w.yb, ya, yb, n);
  return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------------------ allocation-free search
// The working memory of fs_search_noalloc: one fixed array per device, alive
// until the process exits.  In host code the symbol is only a host-side stand-in
// for the array: fs_create looks up its device address once for each context,
// with the context's device current, and the searches pass that address on.
static __device__ __align__(256) unsigned char g_noalloc_scratch[FS_NOALLOC_SCRATCH_BYTES];

fs_status noalloc_address(unsigned char **addr) {
  void *p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess || !p) {
    cudaGetLastError();
    *addr = nullptr;
    return FS_ERR_CUDA;
  }
  *addr = (unsigned char *)p;
  return FS_OK;
}

// offset non-NULL: lattice templates (f1 and offset [nsky][nspin]), one sky row per launch
fs_status search32_noalloc(fs_ctx *ctx, fs_seg *seg, const double *alpha, const double *delta, int nsky,
                           const double *f1, int nspin, float thr, float *F, int64_t nbins, fs_candidate *cand,
                           int64_t cap, int64_t *ncand, cudaStream_t st, const double *offset) {
  if (seg->d.precision != FS_PREC_F32 || nbins != seg->g.nfft / 2) return FS_ERR_UNSUPPORTED;
  int vshift = 0, ps = 0;
  if (!sub_transform(seg->g.nfft, &vshift, &ps) || seg->g.n > seg->g.nfft) return FS_ERR_SHAPE;
  if (vshift) return FS_ERR_SCRATCH;  // a 2^21 transform ring alone exceeds the array
  const FftShape sh = default_split(ps);
  if (offset && !passes_lat_instantiated(sh.N1, sh.N2)) return FS_ERR_UNSUPPORTED;
  const int64_t n = seg->g.n;
  const int n1max = (int)((n + sh.N2 - 1) / sh.N2);
  const int64_t npad = (int64_t)n1max * sh.N2;
  const int64_t stride = (npad + 63) & ~(int64_t)63;
  DemNodes dn = demod_nodes(seg);
  const int lag = 4, slots = 6;  // one sky per launch: a short ring suffices
  // layout inside the fixed array (one sky at a time); a request that does not fit with the
  // nodes' coefficients (up to 0.3 MB more) runs sample by sample instead of being refused
  size_t o_sky, o_ya, o_yb, o_qq, o_nm, o_ab, o_pa, o_dc, o_f1, o_z, o_ct;
  int nblk;
  for (;;) {
    nblk = dn.K ? dn.nb : (int)((npad + 255) / 256);
    size_t off = 0;
    o_sky = off; off = align256(off + sizeof(SkyConst32));
    o_ya = off; off = align256(off + sizeof(float2) * stride);
    o_yb = off; off = align256(off + sizeof(float2) * stride);
    o_qq = off; off = align256(off + sizeof(float2) * stride);
    o_nm = off; off = align256(off + sizeof(float2));
    o_ab = off; off = align256(off + sizeof(double2));
    o_pa = off; off = align256(off + sizeof(float2) * (size_t)nblk);
    o_dc = off; if (dn.K) off = align256(off + sizeof(float4) * kDemCoef * (size_t)dn.nb);
    o_f1 = off; off = align256(off + sizeof(float2) * (size_t)nspin);
    o_z = off; off = align256(off + sizeof(float2) * 2 * (size_t)seg->g.nfft * slots);
    o_ct = off; off = align256(off + sizeof(unsigned) * (1 + 2 * (size_t)nspin));
    if (off <= (size_t)FS_NOALLOC_SCRATCH_BYTES) break;
    if (!dn.K) return FS_ERR_SCRATCH;
    dn.K = 0;
  }
  const size_t o_dn = o_nm + 128;  // in the padding of the norm's 256 bytes
  unsigned char *base = ctx->noalloc;
  if (!base) return FS_ERR_CUDA;
  Ws32 w{};
  w.skyc = (SkyConst32 *)(base + o_sky);
  w.ya = (float2 *)(base + o_ya);
  w.yb = (float2 *)(base + o_yb);
  w.qq = (float2 *)(base + o_qq);
  w.norm = (float2 *)(base + o_nm);
  w.ab2 = (double2 *)(base + o_ab);
  w.partial = (float2 *)(base + o_pa);
  w.dcoef = (float4 *)(base + o_dc);
  w.done = (unsigned *)(base + o_dn);
  w.f1df = (float2 *)(base + o_f1);
  w.Z = (float2 *)(base + o_z);
  w.counters = (unsigned *)(base + o_ct);
  w.stride = stride;
  w.nblk_a1 = nblk;
  DemodArgs DA = demod_args(seg, w, npad);
  DA.nodes = dn;
  for (int g0 = 0; g0 < nsky; g0++) {
    {  // this sky's constants and (lattice) its row of spindowns; the first sky clears the count
      ProfScope ps(ctx, PROF_OTHER, st);
      const double *f1s = offset ? f1 + (int64_t)g0 * nspin : f1;
      if (setup_search(ctx, alpha + g0, delta + g0, 1, seg->g, w.skyc, f1s, nspin, w.f1df, g0 ? nullptr : ncand,
                       w.done, st) !=
          cudaSuccess)
        return FS_ERR_CUDA;
    }
    {
      NvtxRange nv("fs.demodulate");
      ProfScope ps(ctx, PROF_DEMOD, st);
      // the array keeps the previous call's contents: the queue counters start at zero
      DA.ctr = w.counters;
      DA.nctr = 1 + 2 * (int64_t)nspin;
      if (launch_demod(DA, 1, nblk, seg->d.interp, &ctx->launches, st) != cudaSuccess) return FS_ERR_CUDA;
    }
    Cfg32 c{};
    c.sh = sh;
    c.vshift = 0;
    c.nsub = seg->g.nfft;
    c.n1max = n1max;
    c.npad = npad;
    Pass1Args p1;
    Pass2Args p2;
    pass_args(seg, c, w, nspin, thr, cand, cap, ncand, ctx->d_flags, &p1, &p2);
    p2.sky_base = g0;
    p2.F = F ? F + (int64_t)g0 * nspin * nbins : nullptr;
    p2.nbins = nbins;
    p1.z_elems = p2.z_elems = 2 * seg->g.nfft * (int64_t)slots;
    p1.yq_elems = stride;
    p2.f_elems = (int64_t)(nsky - g0) * nspin * nbins;
    QueueArgs qa{};
    qa.ntm = nspin;
    queue_tiles(sh.N1, sh.N2, kPersistThreads, &qa.tiles1, &qa.tiles2);
    qa.kr = 1;
    qa.lag = lag;
    qa.slots = slots;
    qa.ipr_fd = make_fastdiv((uint32_t)(qa.kr * (qa.tiles1 + qa.tiles2)));
    qa.slots_fd = make_fastdiv((uint32_t)qa.slots);
    qa.counter = w.counters;
    {
      NvtxRange nv("fs.transform");
      ProfScope ps(ctx, PROF_PASS2, st);
      if (offset) {
        p1.bin_offset = offset + (int64_t)g0 * nspin;
        if (dispatch_passes_lat(sh.N1, sh.N2, p1, p2, qa, QueueStream{st, &ctx->blocks_per_sm, ctx->nsm}) != cudaSuccess) return FS_ERR_CUDA;
      } else if (dispatch_passes(sh.N1, sh.N2, p1, p2, qa, QueueStream{st, &ctx->blocks_per_sm, ctx->nsm}) != cudaSuccess) {
        return FS_ERR_CUDA;
      }
    }
    ctx->launches += 2;
  }
  return FS_OK;
}

}  // namespace fs
