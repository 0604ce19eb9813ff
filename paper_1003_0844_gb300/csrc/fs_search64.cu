// Plain FP64 form of the search: the analytic model in double at each source time (two FP32
// evaluations bring the first estimate near it, source_time64) or the caller's position
// table, the spline in double, and the zero-padded transform in double on chip
// (k_fft64_cols, k_fft64_rows; 2^21 points by the radix-16 passes of fs_fft64.cu).  It is
// the FP64 comparison for the FP32 path on the same GPU; against sums in 64-bit mantissas
// (1500 to 258,492 samples) F is right to 2e-11 .. 8e-11, as with five FP64 evaluations per sample:
// the FP64 phase of 2e5 cycles decides it.
#include <type_traits>
#include "fs_internal.h"
#include "fs_model.cuh"
#include "fs_blockdft.cuh"

namespace fs {

constexpr unsigned kFull64 = 0xffffffffu;

// eph: NULL (analytic Earth) or the caller's position table of the segment.
__global__ void __launch_bounds__(256) k_demod64(SegGeom g, const SkyConst64 *sky, const dcoef4 *coef,
                                                 const double *x64, int interp, double2 *ya, double2 *yb,
                                                 double *qq, int64_t stride, double *partial, double *tsrc,
                                                 const dbl4 *eph) {
  pdl_wait();
  const int s = blockIdx.y;
  const SkyConst64 K = sky[s];
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double a2 = 0.0, b2 = 0.0;
  if (j < g.n) {
    Geo64 geo;
    const double t = source_time64((double)j * g.dt, K, g, &geo, eph);
    double xr = 0.0;
    if (interp == FS_INTERP_SPLINE2X) {
      if (t >= 0.0 && t <= (double)(g.n - 1) * g.dt) {
        const double u = 2.0 * geo.t1 / g.dt, du = 2.0 * geo.d / g.dt;
        int64_t i = (int64_t)floor(u + du);
        if (i > 2 * g.n - 2) i = 2 * g.n - 2;
        if (i < 0) i = 0;
        const double f = (u - (double)i) + du;
        const dcoef4 c = coef[i];
        xr = fma(f, fma(f, fma(f, c.w, c.z), c.y), c.x);
      }
    } else {
      const int64_t kk = (int64_t)rint(t / g.dt);
      if (kk >= 0 && kk < g.n) xr = x64[kk];
    }
    double av, bv;
    ab_eval64(K, geo.cx, geo.sx, &av, &bv);
    a2 = av * av;
    b2 = bv * bv;
    double cyc = g.fl * geo.phi;
    cyc -= floor(cyc);
    cyc = fma(g.fl, geo.dphi, cyc);
    double sp, cp;
    sincospi(2.0 * cyc, &sp, &cp);
    ya[s * stride + j] = make_double2(xr * av * cp, -xr * av * sp);
    yb[s * stride + j] = make_double2(xr * bv * cp, -xr * bv * sp);
    qq[s * stride + j] = t * (0.5 * t + (geo.phi + geo.dphi));
    if (tsrc && s == 0) tsrc[j] = t;
  }
  for (int o = 16; o > 0; o >>= 1) {
    a2 += __shfl_down_sync(kFull64, a2, o);
    b2 += __shfl_down_sync(kFull64, b2, o);
  }
  __shared__ double wa[8], wb[8];
  if ((threadIdx.x & 31) == 0) { wa[threadIdx.x >> 5] = a2; wb[threadIdx.x >> 5] = b2; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sa = 0.0, sb = 0.0;
    for (int w = 0; w < 8; w++) { sa += wa[w]; sb += wb[w]; }
    double *p = partial + ((int64_t)s * gridDim.x + blockIdx.x) * 2;
    p[0] = sa;
    p[1] = sb;
  }
}

__global__ void __launch_bounds__(256) k_finalize64(const double *partial, int nb, int64_t n, double dt, double S0,
                                                    double2 *norm, double2 *ab2) {
  pdl_wait();
  const int s = blockIdx.x;
  double sa = 0.0, sb = 0.0;
  for (int i = threadIdx.x; i < nb; i += 256) {
    sa += partial[((int64_t)s * nb + i) * 2];
    sb += partial[((int64_t)s * nb + i) * 2 + 1];
  }
  for (int o = 16; o > 0; o >>= 1) {
    sa += __shfl_down_sync(kFull64, sa, o);
    sb += __shfl_down_sync(kFull64, sb, o);
  }
  __shared__ double red[2][8];
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = sa; red[1][threadIdx.x >> 5] = sb; }
  __syncthreads();
  if (threadIdx.x < 2) {  // thread 0: signal a, thread 1: signal b
    const double *r = red[threadIdx.x];
    const double t = ((r[0] + r[1]) + (r[2] + r[3])) + ((r[4] + r[5]) + (r[6] + r[7]));
    if (norm) (&norm[s].x)[threadIdx.x] = 2.0 * dt / (S0 * t);  // cF / (t / n)
    if (ab2) (&ab2[s].x)[threadIdx.x] = t / (double)n;
  }
}

// ------------------------------------------------------------------ transform on chip
// Transforms of nfft = N1 N2 = 2^12 .. 2^20 points (n = N2 n1 + n2, k = k1 + N1 k2) in two
// launches per sky position: k_fft64_cols chirps the demodulated series and takes the DFTs
// over n1 of a few columns, both signals; k_fft64_rows takes those over n2 of a few rows and
// forms F (or stores the bins for interbinning).  Eight values per thread, the factors of a
// transform exchanged through shared memory (fs_blockdft.cuh).  Bound by the FP64 pipe (one
// warp instruction per 16 clocks and SM) and, for one template, by the latency of a launch:
// the two take the place of the chirp kernel, four radix-16 passes through global memory
// and the F kernel.  Measured, a search of one template of 2^16: 63.6 us, 89.2 us before (57
// of them in those six kernels).
constexpr int kDft64Seq = 4;  // sequences per block at least: two columns (rows) of both signals

// exp(-2 pi i e / nfft) from the table of e < nfft/2, 0 <= e < nfft
__device__ __forceinline__ double2 tw64_at(const double2 *tw, int64_t e, int64_t half) {
  const double2 w = tw[e < half ? e : e - half];
  return e < half ? w : make_double2(-w.x, -w.y);
}
template <int LEN>
__device__ __forceinline__ void load_table64(double2 *dst, const double2 *tw, int64_t nfft) {
  const int64_t step = nfft / LEN;
  for (int e = threadIdx.x; e < LEN; e += blockDim.x) dst[e] = tw64_at(tw, e * step, nfft / 2);
}

// The chirp exp(-2 pi i f1 Q_j), with lattice templates times exp(-2 pi i d j / nfft)
__device__ __forceinline__ double2 chirp64(double f1, double d, bool lattice, const double *qq, int64_t j,
                                           int64_t nfft) {
  double cyc = f1 * qq[j];
  cyc -= floor(cyc);
  if (lattice) {
    cyc += d * ((double)j / (double)nfft);
    cyc -= floor(cyc);
  }
  double sp, cp;
  sincospi(2.0 * cyc, &sp, &cp);
  return make_double2(cp, -sp);
}

// Grid: x = column group, y = spindown.  The lanes of a column's two signals share the
// chirps: each computes every other one.
template <int LEN>
__global__ void __launch_bounds__(BlockDft<LEN, kDft64Seq>::THREADS)
    k_fft64_cols(const double2 *ya, const double2 *yb, const double *qq, const double *f1, const double *offset, int64_t n,
                 int N2, const double2 *tw, double2 *out) {
  using C = BlockDft<LEN, kDft64Seq>;
  constexpr int CW = C::SEQ / 2;
  extern __shared__ double2 sm64[];
  double2 *tab = sm64 + C::SEQ * C::STRIDE;
  const int64_t nfft = (int64_t)LEN * N2;
  load_table64<LEN>(tab, tw, nfft);  // the segment's, complete before the search began
  pdl_wait();
  const int c = threadIdx.x % C::SEQ, t = threadIdx.x / C::SEQ;
  const int col = c % CW, sig = c / CW;
  const int n2 = blockIdx.x * CW + col, spin = blockIdx.y;
  const double2 *y = sig ? yb : ya;
  const double f = f1[spin], d = offset ? offset[spin] : 0.0;
  double2 v[8];
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int64_t j = (int64_t)N2 * (t + C::T * m) + n2;
    v[m] = j < n ? y[j] : make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int m = 0; m < 8; m += 2) {
    const int64_t j = (int64_t)N2 * (t + C::T * (m + sig)) + n2;
    const double2 mine = j < n ? chirp64(f, d, offset != nullptr, qq, j, nfft) : make_double2(0.0, 0.0);
    const double2 other = make_double2(__shfl_xor_sync(kFull64, mine.x, CW), __shfl_xor_sync(kFull64, mine.y, CW));
    v[m] = cmul(v[m], sig ? other : mine);
    v[m + 1] = cmul(v[m + 1], sig ? mine : other);
  }
  block_dft<LEN, -1>(v, t, sm64 + c * C::STRIDE, tab);
  double2 *o = out + (2 * (int64_t)spin + sig) * nfft;
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int k1 = t + C::T * m;
    o[(int64_t)k1 * N2 + n2] = cmul(v[m], tw64_at(tw, ((int64_t)n2 * k1) & (nfft - 1), nfft / 2));
  }
}

// One threshold crossing per lane with hit set (called by whole warps).
__device__ __forceinline__ void emit64(bool hit, double Fv, int sky, int spin, int64_t k, fs_candidate *cand, int64_t cap,
                                       unsigned long long *ncand, uint32_t *flags) {
  const int lane = threadIdx.x & 31;
  const unsigned msk = __ballot_sync(kFull64, hit);
  if (!msk) return;
  const int leader = __ffs(msk) - 1;
  unsigned long long base = 0;
  if (lane == leader) base = atomicAdd(ncand, (unsigned long long)__popc(msk));
  base = __shfl_sync(kFull64, base, leader);
  if (hit) {
    const unsigned long long idx = base + __popc(msk & ((1u << lane) - 1u));
    if ((long long)idx < cap) {
      fs_candidate c;
      c.sky = (uint32_t)sky;
      c.spin = (uint32_t)spin;
      c.bin = (uint32_t)k;
      c.F = (float)Fv;
      cand[idx] = c;
    } else {
      atomicOr(flags, ERRF_CAPACITY);
    }
  }
}

// Grid: x = row group, y = spindown.  X non-NULL: the bins in natural order instead of F.
template <int LEN>
__global__ void __launch_bounds__(BlockDft<LEN, kDft64Seq>::THREADS)
    k_fft64_rows(const double2 *in, int N1, const double2 *tw, const double2 *nrmp, int64_t nbins, double *F, double2 *X,
                 int sky, float thr, fs_candidate *cand, int64_t cap, unsigned long long *ncand, uint32_t *flags) {
  using C = BlockDft<LEN, kDft64Seq>;
  extern __shared__ double2 sm64[];
  double2 *tab = sm64 + C::SEQ * C::STRIDE;
  const int64_t nfft = (int64_t)N1 * LEN;
  load_table64<LEN>(tab, tw, nfft);
  pdl_wait();
  const int c = threadIdx.x / C::T, t = threadIdx.x % C::T;
  const int sig = c & 1, k1 = blockIdx.x * (C::SEQ / 2) + (c >> 1), spin = blockIdx.y;
  const double2 *r = in + (2 * (int64_t)spin + sig) * nfft + (int64_t)k1 * LEN;
  double2 v[8];
#pragma unroll
  for (int m = 0; m < 8; m++) v[m] = r[t + C::T * m];
  block_dft<LEN, -1>(v, t, sm64 + c * C::STRIDE, tab);
  if (X) {
    double2 *o = X + (2 * (int64_t)spin + sig) * nfft + k1;
#pragma unroll
    for (int m = 0; m < 8; m++) o[(int64_t)N1 * (t + C::T * m)] = v[m];
    return;
  }
  const double2 nrm = *nrmp;
  double *P = (double *)sm64 + (c >> 1) * LEN;  // the row's |X_b|^2 / <b^2>
  __syncthreads();
  if (sig) {
#pragma unroll
    for (int m = 0; m < 8; m++) P[t + C::T * m] = (v[m].x * v[m].x + v[m].y * v[m].y) * nrm.y;
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int k2 = t + C::T * m;
    const int64_t k = k1 + (int64_t)N1 * k2;
    double Fv = 0.0;
    const bool ok = !sig && k < nbins;
    if (ok) {
      Fv = (v[m].x * v[m].x + v[m].y * v[m].y) * nrm.x + P[k2];
      if (F) F[(int64_t)spin * nbins + k] = Fv;
    }
    emit64(ok && Fv > (double)thr, Fv, sky, spin, k, cand, cap, ncand, flags);
  }
}

static bool fft64_split(int64_t nfft, int *N1, int *N2) {
  if (nfft < (1 << 12) || nfft > (1 << 20)) return false;
  int q = 0;
  while (((int64_t)1 << q) < nfft) q++;
  *N1 = 1 << ((q + 1) / 2);
  *N2 = 1 << (q / 2);
  return true;
}

template <int LEN, typename... KArgs, typename... Args>
static cudaError_t launch_fft64(void (*kern)(KArgs...), int groups, int nspin, cudaStream_t st, Args... args) {
  using C = BlockDft<LEN, kDft64Seq>;
  if constexpr (C::SMEM > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(kern, dim3(groups, nspin), dim3(C::THREADS), C::SMEM, st, args...);
}

template <typename F>
static cudaError_t by_length64(int len, F &&f) {
  switch (len) {
    case 64: return f(std::integral_constant<int, 64>{});
    case 128: return f(std::integral_constant<int, 128>{});
    case 256: return f(std::integral_constant<int, 256>{});
    case 512: return f(std::integral_constant<int, 512>{});
    case 1024: return f(std::integral_constant<int, 1024>{});
  }
  return cudaErrorInvalidValue;
}

// buf[(m*2 + sig)][k] = y^sig_k exp(-2 pi i f1_m Q_k) for k < n, 0 up to nfft; with
// lattice templates (offset non-NULL) also exp(-2 pi i d_m k / nfft), which moves bin
// j of the transform to the frequency (j + d_m) / (nfft dt)
__global__ void k_modulate64(const double2 *ya, const double2 *yb, const double *qq, const double *f1,
                             const double *offset, int nspin, int64_t n, int64_t nfft, double2 *buf) {
  pdl_wait();
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int m = blockIdx.y;
  if (k >= nfft || m >= nspin) return;
  double2 va = make_double2(0.0, 0.0), vb = va;
  if (k < n) {
    const double2 c = chirp64(f1[m], offset ? offset[m] : 0.0, offset != nullptr, qq, k, nfft);
    va = cmul(ya[k], c);
    vb = cmul(yb[k], c);
  }
  buf[(2 * (int64_t)m) * nfft + k] = va;
  buf[(2 * (int64_t)m + 1) * nfft + k] = vb;
}

// F on bin k < nbins; with interbinning (ib) on the half-bin grid: output j
// takes X(j/2) for even j and (X(j/2+1) - X(j/2))/sqrt(2) for odd j (Eq. intbin).
__global__ void k_fstat64(const double2 *buf, int nspin, int64_t nfft, int64_t nbins, const double2 *nrmp, double *F,
                          int sky, float thr, fs_candidate *cand, int64_t cap, unsigned long long *ncand,
                          uint32_t *flags, int ib) {
  pdl_wait();
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int m = blockIdx.y;
  double Fv = 0.0;
  const bool ok = (k < nbins);
  const double2 nrm = *nrmp;
  if (ok) {
    const double2 *ba = buf + (2 * (int64_t)m) * nfft, *bb = ba + nfft;
    const int64_t q = ib ? (k >> 1) : k;
    double2 xa = ba[q], xb = bb[q];
    if (ib && (k & 1)) {
      const double2 ya = ba[q + 1], yb = bb[q + 1];
      xa = make_double2((ya.x - xa.x) * 0.70710678118654752440, (ya.y - xa.y) * 0.70710678118654752440);
      xb = make_double2((yb.x - xb.x) * 0.70710678118654752440, (yb.y - xb.y) * 0.70710678118654752440);
    }
    Fv = (xa.x * xa.x + xa.y * xa.y) * nrm.x + (xb.x * xb.x + xb.y * xb.y) * nrm.y;
    if (F) F[(int64_t)m * nbins + k] = Fv;
  }
  emit64(ok && Fv > (double)thr, Fv, sky, m, k, cand, cap, ncand, flags);
}

struct Ws64 {
  SkyConst64 *skyc;
  double2 *ya, *yb, *norm, *ab2, *buf, *tmp;
  double *qq, *partial;
  int nblk;
};

static size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

static fs_status workspace64(fs_ctx *ctx, const fs_seg *seg, int nspin, cudaStream_t st, Ws64 *w) {
  const int64_t n = seg->g.n, nfft = seg->g.nfft;
  const int nblk = (int)((n + 255) / 256);
  size_t off = 0;
  size_t o_sky = off; off = al256(off + sizeof(SkyConst64));
  size_t o_ya = off; off = al256(off + sizeof(double2) * n);
  size_t o_yb = off; off = al256(off + sizeof(double2) * n);
  size_t o_qq = off; off = al256(off + sizeof(double) * n);
  size_t o_nm = off; off = al256(off + sizeof(double2));
  size_t o_ab = off; off = al256(off + sizeof(double2));
  size_t o_pa = off; off = al256(off + sizeof(double) * 2 * nblk);
  size_t o_bf = off; off = al256(off + sizeof(double2) * 2 * (size_t)nspin * nfft);
  size_t o_tm = off; off = al256(off + sizeof(double2) * 2 * (size_t)nspin * nfft);
  fs_status s = ensure_buffer(&ctx->ws64, &ctx->ws64_bytes, off, st);
  if (s != FS_OK) return s;
  char *b = (char *)ctx->ws64;
  w->skyc = (SkyConst64 *)(b + o_sky);
  w->ya = (double2 *)(b + o_ya);
  w->yb = (double2 *)(b + o_yb);
  w->qq = (double *)(b + o_qq);
  w->norm = (double2 *)(b + o_nm);
  w->ab2 = (double2 *)(b + o_ab);
  w->partial = (double *)(b + o_pa);
  w->buf = (double2 *)(b + o_bf);
  w->tmp = (double2 *)(b + o_tm);
  w->nblk = nblk;
  return FS_OK;
}

// offset non-NULL: lattice templates, f1 and offset [nsky][nspin] (row sk for sky sk)
fs_status search64(fs_ctx *ctx, fs_seg *seg, const double *alpha, const double *delta, int nsky,
                   const double *f1, int nspin, float thr, double *F, int64_t nbins, fs_candidate *cand,
                   int64_t cap, int64_t *ncand, cudaStream_t st, const double *offset) {
  const int64_t n = seg->g.n, nfft = seg->g.nfft;
  Ws64 w;
  fs_status s = workspace64(ctx, seg, nspin, st, &w);
  if (s != FS_OK) return s;
  for (int sk = 0; sk < nsky; sk++) {
    if (setup_search64(ctx, alpha + sk, delta + sk, 1, seg->g, w.skyc, sk ? nullptr : ncand, st) != cudaSuccess)
      return FS_ERR_CUDA;
    cudaError_t e = launch_pdl(k_demod64, dim3(w.nblk, 1), dim3(256), 0, st, seg->g, w.skyc,
                               (const dcoef4 *)seg->coef, seg->x64, seg->d.interp, w.ya, w.yb, w.qq, 0, w.partial,
                               nullptr, seg->eph);
    if (e == cudaSuccess)
      e = launch_pdl(k_finalize64, dim3(1), dim3(256), 0, st, w.partial, w.nblk, n, seg->g.dt, seg->g.S0, w.norm,
                     w.ab2);
    ctx->launches += 5;  // sky constants, demodulation, finalize, modulation, F epilogue
    const double *f1s = offset ? f1 + (int64_t)sk * nspin : f1;
    const double *ds = offset ? offset + (int64_t)sk * nspin : nullptr;
    double *Fs = F ? F + (int64_t)sk * nspin * nbins : nullptr;
    const int ib = (seg->d.options & FS_OPT_INTERBIN) ? 1 : 0;
    double2 *X = nullptr;  // the bins, where F is formed from them by a launch of its own
    int N1 = 0, N2 = 0;
    if (fft64_split(nfft, &N1, &N2)) {
      double2 *out = ib ? w.tmp : nullptr;
      if (e == cudaSuccess)
        e = by_length64(N1, [&](auto len) {
          constexpr int LEN = decltype(len)::value;
          return launch_fft64<LEN>(k_fft64_cols<LEN>, N2 / (BlockDft<LEN, kDft64Seq>::SEQ / 2), nspin, st, w.ya, w.yb,
                                   w.qq, f1s, ds, n, N2, seg->tw64, w.buf);
        });
      if (e == cudaSuccess)
        e = by_length64(N2, [&](auto len) {
          constexpr int LEN = decltype(len)::value;
          return launch_fft64<LEN>(k_fft64_rows<LEN>, N1 / (BlockDft<LEN, kDft64Seq>::SEQ / 2), nspin, st, w.buf, N1,
                                   seg->tw64, w.norm, nbins, Fs, out, sk, thr, cand, cap, (unsigned long long *)ncand,
                                   ctx->d_flags);
        });
      X = out;
    } else {  // 2^21: the passes through global memory
      if (e == cudaSuccess)
        e = launch_pdl(k_modulate64, dim3((unsigned)((nfft + 255) / 256), nspin), dim3(256), 0, st, w.ya, w.yb, w.qq,
                       f1s, ds, nspin, n, nfft, w.buf);
      if (e == cudaSuccess) e = fft64(w.buf, w.tmp, seg->tw64, nfft, 2 * nspin, -1, st, &ctx->launches, &X);
    }
    if (X && e == cudaSuccess)
      e = launch_pdl(k_fstat64, dim3((unsigned)((nbins + 255) / 256), nspin), dim3(256), 0, st, X, nspin, nfft, nbins,
                     w.norm, Fs, sk, thr, cand, cap, (unsigned long long *)ncand, ctx->d_flags, ib);
    if (e != cudaSuccess) return FS_ERR_CUDA;
  }
  return cuda_status(cudaGetLastError());
}

__global__ void k_copy_pairs(const double2 *y, double *o, int64_t n) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j < n) { o[2 * j] = y[j].x; o[2 * j + 1] = y[j].y; }
}

fs_status demod64_debug(fs_ctx *ctx, fs_seg *seg, double alpha, double delta, double *ya, double *yb,
                        double *tsrc, double *ab2, cudaStream_t st) {
  const int64_t n = seg->g.n;
  Ws64 w;
  fs_status s = workspace64(ctx, seg, 1, st, &w);
  if (s != FS_OK) return s;
  double hd[2] = {alpha, delta};
  double *dd = (double *)w.ab2;
  if (cudaMemcpyAsync(dd, hd, sizeof(hd), cudaMemcpyHostToDevice, st) != cudaSuccess) return FS_ERR_CUDA;
  if (setup_search64(ctx, dd, dd + 1, 1, seg->g, w.skyc, nullptr, st) != cudaSuccess) return FS_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return FS_ERR_CUDA;
  k_demod64<<<dim3(w.nblk, 1), 256, 0, st>>>(seg->g, w.skyc, (const dcoef4 *)seg->coef, seg->x64,
                                              seg->d.interp, w.ya, w.yb, w.qq, 0, w.partial, tsrc,
                                              seg->eph);
  k_finalize64<<<1, 256, 0, st>>>(w.partial, w.nblk, n, seg->g.dt, seg->g.S0, nullptr, (double2 *)ab2);
  k_copy_pairs<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w.ya, ya, n);
  k_copy_pairs<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w.yb, yb, n);
  return cuda_status(cudaGetLastError());
}

}  // namespace fs
