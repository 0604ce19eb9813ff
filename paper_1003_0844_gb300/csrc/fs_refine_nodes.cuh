// The fine search's sums over a few nodes per block of samples in place of every sample
// (included by fs_refine.cu).
//
// Every sum of the fine search has the form sum_k x_k exp(-2 pi i Phi_k) g(t_k) or
// sum_k g(t_k), g a product of the amplitude modulation, the delay, t and their
// derivatives: smooth in time (a few cycles per day), unlike the phase and the data.  On
// a block of kNodeSub * sb samples, at most 512 s long, g is its interpolating polynomial
// through kNodes Chebyshev nodes t_q, so that
//   sum_k x_k exp(-2 pi i Phi_k) g(t_k) = sum_q W_q g(t_q),
//   W_q = sum_k x_k exp(-2 pi i Phi_k) l_q(s_k) = sum_m l_qm S_m,
//   S_m = sum_k x_k exp(-2 pi i Phi_k) s_k^m,
// with l_q the Lagrange polynomials, s in (-1, 1) the place in the block.  k_moments forms
// W_q once per point and block; the 26 + 46 sums of F, its gradient and its Hessian then
// run over 6 nodes per block (one node for 43 samples at dt = 2 s) with W_q in the place
// of x_k exp(-2 pi i Phi_k).  The error of the interpolation is below
// (2 Omega_r 256 s)^6 / (6! 2^5) = 1.2e-13 of g's scale (products with a second harmonic of
// the day; the third and fourth have amplitudes below 1e-4 of it).  The derivatives with
// f1 hold t^2, and f1's second one t^4, beside a and b: over a block of length h a series of
// length T bends these by (h/T)^2 and (h/T)^3 of their scale, times
// 15 (2 Omega_r 256 s)^4 / (6! 2^5) = 1.2e-9, so a series is cut into 32 blocks at least
// (node_sub).
//
// The phase is needed at every sample, but it too is a polynomial on the block, through
// its values at the same nodes: (f0 + fl) times the diurnal delay's sixth-order term is
// below 1e-13 cycles.  Its linear and f1's quadratic part are taken out with exactly known
// rates, the small rest is interpolated, and the phase then advances from sample to sample
// by two 64-bit integer additions (units of 2^-64 cycles: reduction modulo 1 is free).
//
// Accuracy (19 lengths from 1024 samples to 6 days at 0.5 to 16 s, against sums in 64-bit
// mantissas, worst of four points each): F 4e-14 .. 2e-11, the gradient 1e-14 .. 4e-11 and the
// Hessian 6e-14 .. 2e-11 of F times the phase derivatives that meet in them; over every
// sample it is F 1e-11 .. 3e-10, gradient 4e-12 .. 3e-10, Hessian 2e-12 .. 1e-9, bound by the
// FP64 phase of each sample (3e-11 cycles).  With blocks of 512 s whatever the length (one of
// 256 samples for a series of 200) the gradient was off by up to 1e-8, the Hessian by 3e-7.
// The sky gradient, whose parts cancel, ends at 2e-9 .. 5e-8 of F (3e-8 .. 2e-7 over every
// sample, with FP32 derivatives of a and b).
// Measured, 256 points of a 2-day series at 2 s with gradient and Hessian: 4.72 ms over every
// sample, 0.28 ms this way, about half of it k_moments and half the sums over nodes.
#pragma once

namespace fs {

constexpr int kNodes = 6;     // nodes per block
constexpr int kNodeSub = 8;   // sub-blocks per block, one warp each in k_moments
constexpr int kNodeSubMin = 4, kNodeSubMax = 128;  // samples per sub-block

// Blocks a series is cut into at least.  The derivatives with f1 hold t^2 and t^4 beside a
// and b, whose curvature over a block is the larger the fewer blocks there are.
constexpr int kNodeBlocks = 32;

// Samples per sub-block for a sampling interval and a length: the largest power of two
// within 64 s, at most 128, that leaves kNodeBlocks blocks.  0 (the sums run over every
// sample): dt above 16 s, where a block would hold no more than five samples per node and
// the interpolation no longer pays, and series below kNodeBlocks of the smallest blocks,
// 1024 samples.
static int node_sub(double dt, int64_t n) {
  if (!(dt <= 16.0) || n < (int64_t)kNodeBlocks * kNodeSub * kNodeSubMin) return 0;
  int sb = kNodeSubMin;
  while (2 * sb <= kNodeSubMax && 2 * sb * dt <= 64.0 && n >= (int64_t)kNodeBlocks * kNodeSub * 2 * sb) sb *= 2;
  return sb;
}

// Per-segment node tables (geometry only; one allocation).
struct NodeTab {
  int sb, nb, nn;     // samples per sub-block, blocks, nodes (kNodes nb)
  double cr, sr;      // (cos, sin) of the orbital longitude at the segment's middle
  double2 *E;         // (cos, sin) of the orbital longitude at the nodes less (cr, sr)
  double *n64;        // node times in samples (exact: places are multiples of 2^-8 samples)
  float4 *L, *T;      // orbital longitude and sidereal angle as double-floats (Etab32)
  float2 *t;          // node times as double-floats
  float2 *w;          // sum of l_q over the block's samples
  float4 *SC;         // exp(-2 pi i j / 1024) as (cos hi, cos lo, sin hi, sin lo), j < 1024
  float2 *lag;        // l_qm [kNodes][kNodes]
  float2 *sub;        // [kNodeSub][4][kNodes]: the phase's cubic on each sub-block from its node values
  double *u;          // [kNodes]: node places in samples from the block's first
};
constexpr int kNodeSc = 1024;

static __host__ __device__ inline double node_ref_longitude(const SegGeom &g) {
  return g.lambda0 + kOmegaO * (0.5 * (double)g.n * g.dt);
}

static size_t node_tab_view(const SegGeom &g, int sb, char *base, NodeTab *v) {
  const int64_t K = (int64_t)kNodeSub * sb, nb = (g.n + K - 1) / K, nn = nb * kNodes;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = (off + bytes + 255) & ~(size_t)255;
    return base + o;
  };
  v->sb = sb;
  v->nb = (int)nb;
  v->nn = (int)nn;
  const double lr = node_ref_longitude(g);
  v->cr = cos(lr);
  v->sr = sin(lr);
  v->E = (double2 *)take(sizeof(double2) * nn);
  v->n64 = (double *)take(sizeof(double) * nn);
  v->L = (float4 *)take(sizeof(float4) * nn);
  v->T = (float4 *)take(sizeof(float4) * nn);
  v->t = (float2 *)take(sizeof(float2) * nn);
  v->w = (float2 *)take(sizeof(float2) * nn);
  v->SC = (float4 *)take(sizeof(float4) * kNodeSc);
  v->lag = (float2 *)take(sizeof(float2) * kNodes * kNodes);
  v->sub = (float2 *)take(sizeof(float2) * kNodeSub * 4 * kNodes);
  v->u = (double *)take(sizeof(double) * kNodes);
  return off;
}

__device__ __forceinline__ float2 f2_from_double(double x) {
  const df32 d = df_from_double(x);
  return make_float2(d.hi, d.lo);
}
// Chebyshev nodes, moved to a multiple of 2^-8 samples (K samples per block).
__device__ inline double node_place(int q, int K) {
  const double half = 0.5 * K, s = -cospi((2 * q + 1) / (2.0 * kNodes));
  return (rint((0.5 * (K - 1) + s * half) * 256.0) / 256.0 - 0.5 * (K - 1)) / half;
}

// Coefficients of the Lagrange polynomial l_q in powers of s.
__device__ inline void node_lagrange(int q, int K, double (&c)[kNodes]) {
  for (int m = 0; m < kNodes; m++) c[m] = m == 0 ? 1.0 : 0.0;
  const double sq = node_place(q, K);
  int deg = 0;
  for (int j = 0; j < kNodes; j++) {
    if (j == q) continue;
    const double sj = node_place(j, K), inv = 1.0 / (sq - sj);
    deg++;
    for (int m = deg; m >= 0; m--) c[m] = ((m > 0 ? c[m - 1] : 0.0) - sj * c[m]) * inv;
  }
}

__global__ void k_node_tables(SegGeom g, NodeTab v) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int K = kNodeSub * v.sb;
  if (i < v.nn) {
    const int64_t b = i / kNodes;
    const int q = (int)(i - b * kNodes);
    const double nq = (double)(b * K) + (0.5 * (K - 1) + node_place(q, K) * (0.5 * K));
    const double t = nq * g.dt;
    double sl, cl, sth, cth;
    sincos(g.lambda0 + kOmegaO * t, &sl, &cl);
    sincos(g.theta0 + kOmegaR * t, &sth, &cth);
    // cos a - cos b and sin a - sin b as products: full relative accuracy
    const double hd = 0.5 * kOmegaO * (t - 0.5 * (double)g.n * g.dt);
    double sm, cm;
    sincos(node_ref_longitude(g) + hd, &sm, &cm);
    const double sh = 2.0 * sin(hd);
    v.E[i] = make_double2(-sm * sh, cm * sh);
    v.n64[i] = nq;
    const float2 c = f2_from_double(cl), s = f2_from_double(sl), ct = f2_from_double(cth), st = f2_from_double(sth);
    v.L[i] = make_float4(c.x, c.y, s.x, s.y);
    v.T[i] = make_float4(ct.x, ct.y, st.x, st.y);
    v.t[i] = f2_from_double(t);
    // sum of l_q over the samples the block holds (all K but in the last block)
    double c6[kNodes], w = 0.0;
    const double inv_k = 1.0 / K;
    node_lagrange(q, K, c6);
    const int64_t have = g.n - b * K < K ? g.n - b * K : K;
    for (int64_t j = 0; j < have; j++) {
      const double s1 = fma(2.0 * j + 1.0, inv_k, -1.0);
      double p = c6[kNodes - 1];
      for (int m = kNodes - 2; m >= 0; m--) p = fma(p, s1, c6[m]);
      w += p;
    }
    v.w[i] = f2_from_double(w);
  }
  if (i < kNodeSc) {
    double sj, cj;
    sincospi((double)i / (kNodeSc / 2), &sj, &cj);
    const float2 c = f2_from_double(cj), s = f2_from_double(sj);
    v.SC[i] = make_float4(c.x, c.y, s.x, s.y);
  }
  if (i < kNodes) {
    double c[kNodes];
    node_lagrange((int)i, K, c);
    v.u[i] = 0.5 * (K - 1) + node_place((int)i, K) * (0.5 * K);
    for (int m = 0; m < kNodes; m++) v.lag[i * kNodes + m] = f2_from_double(c[m]);
    for (int w = 0; w < kNodeSub; w++) {
      // l_q(s_w + sigma / 8) in powers of sigma, the fourth and fifth by their least-squares
      // cubic on (-1, 1), sigma^4 ~ 6/7 sigma^2 - 3/35, sigma^5 ~ 10/9 sigma^3 - 5/21 sigma:
      // what that leaves of the phase (2e-12 cycles) has no mean over a sub-block, where the
      // nearest cubic's shows as a phase error of 6e-13 rad with the period of a day
      const double sw = (2.0 * w + 1.0) / kNodeSub - 1.0;
      double d[kNodes], scale = 1.0;
      for (int e = 0; e < kNodes; e++) {
        double acc = 0.0, pw = 1.0, binom = 1.0;
        for (int m = e; m < kNodes; m++) {
          acc += c[m] * binom * pw;
          pw *= sw;
          binom = binom * (m + 1) / (m + 1 - e);
        }
        d[e] = acc * scale;
        scale /= kNodeSub;
      }
      const double r[4] = {d[0] - d[4] * 3.0 / 35.0, d[1] - d[5] * 5.0 / 21.0, d[2] + d[4] * 6.0 / 7.0,
                           d[3] + d[5] * 10.0 / 9.0};
      for (int e = 0; e < 4; e++) v.sub[(w * 4 + e) * kNodes + i] = f2_from_double(r[e]);
    }
  }
}

// ------------------------------------------------------------------ moments
__device__ __forceinline__ long long df_fix64(df32 x) {  // cycles -> 2^-64 cycles
  constexpr float k = 18446744073709551616.f;
  return __float2ll_rn(x.hi * k) + __float2ll_rn(x.lo * k);
}
// Pairs (re, im) in packed FP32 instructions (fs_dft.cuh): the moments' arithmetic is the
// same for both halves, and a pair takes one issue slot instead of two.
#ifdef FS_X2
__device__ __forceinline__ float2 x2b(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 x2neg(float2 a) { return make_float2(-a.x, -a.y); }
// a + b = s + e by halves
__device__ __forceinline__ void x2_two_sum(float2 a, float2 b, float2 *s, float2 *e) {
  *s = x2add(a, b);
  const float2 bb = x2sub(*s, a);
  *e = x2add(x2sub(a, x2sub(*s, bb)), x2sub(b, bb));
}
// acc += v for a sum whose low word is not normalised between additions
__device__ __forceinline__ void x2_acc(float2 &hi, float2 &lo, float2 vh, float2 vl) {
  float2 s, e;
  x2_two_sum(hi, vh, &s, &e);
  hi = s;
  lo = x2add(lo, x2add(e, vl));
}
// acc += k (vh + vl), k an exact FP32 factor
__device__ __forceinline__ void x2_acc_scaled(float2 &hi, float2 &lo, float k, float2 vh, float2 vl) {
  const float2 kk = x2b(k), p = x2mul(kk, vh);
  x2_acc(hi, lo, p, x2fma(kk, vl, x2fma(kk, vh, x2neg(p))));
}
#endif

// Phase [cycles] of a sample by FP64 throughout, for points whose phase the block's
// polynomial does not follow.
__device__ __noinline__ long long phase_direct(const FastConst &c, const SegGeom &g, int64_t k) {
  const double t = (double)k * g.dt;
  double sl, cl, sth, cth;
  sincos(g.lambda0 + kOmegaO * t, &sl, &cl);
  sincos(g.theta0 + kOmegaR * t, &sth, &cth);
  auto d = [](df32 v) { return (double)v.hi + (double)v.lo; };
  const double phi = c.nxA * cl + c.nyA * sl + d(c.rcd) * (d(c.ca) * cth + d(c.sa) * sth) + d(c.zsd);
  double p = c.F0L * phi + c.f0 * t + d(c.f1) * t * (0.5 * t + phi);
  p -= rint(p);
  return __double2ll_rn(p * 18446744073709551616.0);
}

constexpr int kMomThreads = 32 * kNodeSub;
constexpr int kMomComp = 12;  // S_0 .. S_5, re and im

struct MomShared {
  float4 sc[kNodeSc];
  float red[kMomComp + 6][kNodeSub][32];  // S_0..S_2 in two words, S_3..S_5 in one
  float2 mom[kMomComp][32];
  float2 d[kNodes][32];                   // the phase's rest at the nodes relative to node 2
  long long r[kNodes][32];
  long long nu[32], kap[32];
  float nuf[32];
  int bad[32];
  float2 lag[kNodes * kNodes];
  float2 sub[kNodeSub * 4 * kNodes];
};

// W_q of 32 points (lanes) on one block of samples, sub-block w in warp w.  Grid: x =
// block of samples, y = group of points.
//
// Bound by the FMA pipe and issue: about 110 FP32 results per sample and point (the table
// sine and cosine 40, the double-float products with the data and the sums S_0, S_1, S_2
// 68) and a dozen integer instructions for the phase, against ~3500 for the 72 sums
// themselves.  The real and the imaginary part go through packed pairs: 288 -> 274 us for a
// step on 256 points (k_moments itself 140 us with scalar instructions, issue 0.65 busy).
// S_3 to S_5 enter with g's third and higher powers over a block, below 2e-5 of the result
// with 32 blocks, and are FP32.  A point per lane makes the data,
// the place s and its powers the same for the whole warp (broadcast reads), and leaves
// nothing to reduce across lanes.
__global__ void __launch_bounds__(kMomThreads, 4) k_moments(SegGeom g, NodeTab v, const float2 *X,
                                                         const FastConst *fcs, int npt, float2 *W) {
  extern __shared__ __align__(16) unsigned char mom_smem[];
  MomShared &S = *(MomShared *)mom_smem;
  float4 *sx = (float4 *)(mom_smem + sizeof(MomShared));  // (x.hi, x.lo, s, sigma^3) per sample
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = blockIdx.x, sb = v.sb, K = kNodeSub * sb;
  const int pt = blockIdx.y * 32 + lane;
  const FastConst &c = fcs[min(pt, npt - 1)];
  for (int i = threadIdx.x; i < kNodeSc; i += kMomThreads) S.sc[i] = v.SC[i];
  for (int i = threadIdx.x; i < kNodes * kNodes; i += kMomThreads) S.lag[i] = v.lag[i];
  for (int i = threadIdx.x; i < kNodeSub * 4 * kNodes; i += kMomThreads) S.sub[i] = v.sub[i];
  const float inv_sb = 1.0f / (float)sb;
  pdl_wait();  // (the tables above are the segment's)
  for (int j = threadIdx.x; j < K; j += kMomThreads) {
    const int64_t k = (int64_t)b * K + j;
    const float2 x = k < g.n ? X[k] : make_float2(0.f, 0.f);
    const float s = (float)(2 * j + 1) * (0.125f * inv_sb) - 1.f;                    // exact
    const float sg = (float)(2 * (j & (sb - 1)) + 1) * inv_sb - 1.f;  // exact
    sx[j] = make_float4(x.x, x.y, s, sg * sg * sg);
  }
  double ph = 0.0;
  if (w < kNodes) {
    // the phase at node w, modulo 1.  An error here is shared by the node's 43 samples or
    // more, so it is kept below FP64's rounding of the phase itself (2.5e5 cycles: 3e-11):
    // the orbital delay as its value at the segment's middle (a constant of the point,
    // c.Pref) and the difference to it, f0 t with its rounding error.
    const int i = b * kNodes + w;
    const double2 e = v.E[i];
    const float4 Tq = v.T[i];
    const double n = v.n64[i], t = n * g.dt;
    const double dphi = fma(c.nxA, e.x, c.nyA * e.y);
    const double f0dt = c.f0 * g.dt, p0 = f0dt * n;
    double P = (p0 - rint(p0)) + fma(f0dt, n, -p0) + fma(c.f0, g.dt, -f0dt) * n;
    const double po = c.F0L * dphi;
    P += (po - rint(po)) + c.Pref;
    const df32 cx = df_add(df_mul(c.ca, df32{Tq.x, Tq.y}), df_mul(c.sa, df32{Tq.z, Tq.w}));
    const df32 phid = df_add(df_mul(c.rcd, cx), c.zsd);
    const df32 pd = df_mul(c.F0L2, phid);
    const double phi = c.phir + dphi + ((double)phid.hi + (double)phid.lo);
    const double ps = ((double)c.f1.hi + (double)c.f1.lo) * (t * fma(0.5, t, phi));
    ph = P + (ps - rint(ps)) + ((double)pd.hi + (double)pd.lo);
  } else if (w == kNodes) {
    // the rate at the block's first sample and f1's curvature, cycles per sample (and
    // squared); whatever FP32 loses stays in the rest
    const int i = b * kNodes + 2;
    const float4 Lq = v.L[i], Tq = v.T[i];
    const float dt = c.dt.hi, f1 = c.f1.hi, F0L = (float)c.F0L;
    const float sxn = c.sa.hi * Tq.x - c.ca.hi * Tq.z, cxn = c.ca.hi * Tq.x + c.sa.hi * Tq.z;
    const float phidot = (float)kOmegaO * (c.nyA2.hi * Lq.x - c.nxA2.hi * Lq.z) + (float)kOmegaR * c.rcd.hi * sxn;
    const float phi = c.nxA2.hi * Lq.x + c.nyA2.hi * Lq.z + c.rcd.hi * cxn + c.zsd.hi;
    const float t0 = (float)b * ((float)K * dt), tm = t0 + 0.5f * (float)K * dt;
    const float kap = 0.5f * f1 * dt * dt;
    const float H = 0.5f * (float)K * dt;
    const float nu = (float)(c.f0 * g.dt) + (F0L * phidot + f1 * (tm + phi + tm * phidot)) * dt - kap * (float)K;
    // the Doppler curvature must stay well inside half a cycle over the block (1.4e-10
    // s^-1 bounds the delay's second derivative); a rate of 4 cycles per sample and more
    // would cost the rest digits, here and in FP32 above
    const bool ok = fabsf(F0L) * (1.4e-10f * 0.5f) * H * H < 0.1f && fabsf(F0L) * dt * 1.1e-4f < 4.f &&
                    fabsf(f1) * (t0 + 1e3f) * dt < 4.f && fabsf(nu) < 4.f && fabsf(kap) < 1e-3f;
    // whole turns per sample count at the nodes, which lie between samples, but not at the
    // samples
    S.nuf[lane] = nu;
    S.nu[lane] = __double2ll_rn((double)(nu - rintf(nu)) * 18446744073709551616.0);
    S.kap[lane] = __double2ll_rn((double)kap * 18446744073709551616.0);
    S.bad[lane] = ok ? 0 : isfinite(c.F0L) && isfinite(c.f0) && isfinite(f1) ? 1 : 2;
  }
  __syncthreads();
  if (w < kNodes) {  // what the known rates leave of it
    const double u = v.u[w], k64 = 1.0 / 18446744073709551616.0;
    double r = ph - (double)S.nuf[lane] * u - ((double)S.kap[lane] * k64) * (u * u);
    r -= rint(r);
    S.r[w][lane] = __double2ll_rn(r * 18446744073709551616.0);
  }
  __syncthreads();
  if (w < kNodes) {
    const long long d = S.r[w][lane] - S.r[2][lane];  // modulo 1, small
    const float hi = (float)((double)d * (1.0 / 18446744073709551616.0));
    const float lo = (float)((double)d * (1.0 / 18446744073709551616.0) - (double)hi);
    S.d[w][lane] = make_float2(hi, lo);
  }
  __syncthreads();
  const float2 zero = make_float2(0.f, 0.f);
  float2 h0 = zero, l0 = zero, h1 = zero, l1 = zero, h2 = zero, l2 = zero, m3 = zero, m4 = zero, m5 = zero;
  {
    df32 rho[4];
#pragma unroll
    for (int e = 0; e < 4; e++) {
      df32 a{0.f, 0.f};
#pragma unroll
      for (int q = 0; q < kNodes; q++) {
        if (q == 2) continue;  // d = 0 there; the l_q sum to one
        const float2 mq = S.sub[(w * 4 + e) * kNodes + q], dq = S.d[q][lane];
        a = df_add(a, df_mul(df32{mq.x, mq.y}, df32{dq.x, dq.y}));
      }
      rho[e] = a;
    }
    // sigma = sg0 + j 2/sb (all exact): the quadratic as a phase, its first and second difference
    const float sg0 = inv_sb - 1.f, h = 2.f * inv_sb;
    const df32 a0 = df_add(rho[0], df_add(df_mul_f(rho[1], sg0), df_mul_f(rho[2], sg0 * sg0)));
    const df32 a1 = df_scale(df_add(rho[1], df_scale(df_mul_f(rho[2], sg0), 2.f)), h);
    const df32 a2 = df_scale(rho[2], h * h);
    const long long j0 = (long long)w * sb, nu = S.nu[lane], kap = S.kap[lane], a2f = df_fix64(a2);
    unsigned long long phase = (unsigned long long)S.r[2][lane] + (unsigned long long)df_fix64(a0) +
                               (unsigned long long)nu * (unsigned long long)j0 +
                               (unsigned long long)kap * (unsigned long long)(j0 * j0);
    unsigned long long step = (unsigned long long)nu + (unsigned long long)kap * (unsigned long long)(2 * j0 + 1) +
                              (unsigned long long)df_fix64(a1) + (unsigned long long)a2f;
    const unsigned long long curv = 2ull * ((unsigned long long)kap + (unsigned long long)a2f);
    const float c3 = 6.283185307f * rho[3].hi;
    const float4 *xs = sx + w * sb;
    // one sample: its phase (2^-64 cycles, and the cubic rest in radians) and data
    auto add_sample = [&](unsigned long long phase, float cubic, const float4 &xv) {
      const unsigned hi = (unsigned)(phase >> 32), lo = (unsigned)phase;
      // nearest table angle and the remainder x = xh + xl [rad], |x| <= pi / 1024
      const unsigned idx = (hi + (1u << 21)) >> 22;
      const int rh = (int)(hi - (idx << 22));
      const float fh = __int_as_float(0x4B400000 + rh) - 12582912.f;        // exact
      const float fl = __int_as_float(0x4B000000 | (lo >> 9)) - 8388608.f;  // units of 2^-55 cycles
      constexpr float k32h = 1.46291807926716e-09f;                         // 2 pi / 2^32 in two words
      constexpr float k32l = (float)(6.283185307179586476925286766559 / 4294967296.0 - (double)1.46291807926716e-09f);
      constexpr float k55 = (float)(6.283185307179586476925286766559 / 36028797018963968.0);
      const float xh = fh * k32h;
      const float xl = fmaf(fh, k32h, -xh) + (fmaf(fh, k32l, fl * k55) + cubic);
      const float xx = xh * xh;
      // cos x - 1 and sin x = xh + sl (dropped: x^5/120 and the like, below 3e-15)
      const float cm = fmaf(-xh, xl, xx * fmaf(xx, 1.f / 24.f, -0.5f));
      const float sl = fmaf(xh * xx, -1.f / 6.f, xl);
      const float4 tq = S.sc[idx & (kNodeSc - 1)];
#ifdef FS_X2
      // (cos, sin) = (C, S) (1 + cm) + (-S, C) sin x
      const float2 T = make_float2(tq.x, tq.z), Tl = make_float2(tq.y, tq.w);
      const float2 xs = make_float2(-xh, xh), ts = x2swap(T);
      const float2 pr = x2mul(ts, xs), er = x2fma(ts, xs, x2neg(pr));
      float2 c, ce;
      x2_two_sum(T, pr, &c, &ce);
      const float2 cl = x2add(ce, x2add(x2fma(T, x2b(cm), Tl),
                                        x2fma(ts, make_float2(-sl, sl), x2fma(x2swap(Tl), xs, er))));
      // z = x (cos, sin)
      const float2 xb = x2b(xv.x), z = x2mul(xb, c);
      const float2 zl = x2fma(xb, cl, x2fma(x2b(xv.y), c, x2fma(xb, c, x2neg(z))));
      x2_acc(h0, l0, z, zl);
      const float s1 = xv.z, s2 = s1 * s1, s3 = s2 * s1;  // s and s^2 exact
      x2_acc_scaled(h1, l1, s1, z, zl);
      x2_acc_scaled(h2, l2, s2, z, zl);
      m3 = x2fma(x2b(s3), z, m3);
      m4 = x2fma(x2b(s3 * s1), z, m4);
      m5 = x2fma(x2b(s3 * s2), z, m5);
#endif
    };
    const bool bad = S.bad[lane] != 0;
    if (!__any_sync(0xffffffffu, bad)) {
#pragma unroll 4
      for (int j = 0; j < sb; j++) {
        const float4 xv = xs[j];
        add_sample(phase, c3 * xv.w, xv);
        phase += step;
        step += curv;
      }
    } else {
#pragma unroll 1
      for (int j = 0; j < sb; j++) {
        const float4 xv = xs[j];
        unsigned long long p = phase;
        if (bad) p = (unsigned long long)phase_direct(c, g, min((int64_t)b * K + w * sb + j, g.n - 1));
        add_sample(p, bad ? 0.f : c3 * xv.w, xv);
        phase += step;
        step += curv;
      }
    }
  }
  {
    // S.red[2 q], [2 q + 1]: words of component q = 2 m (re), 2 m + 1 (im)
    const float v[kMomComp + 6] = {h0.x, l0.x, h0.y, l0.y, h1.x, l1.x, h1.y, l1.y, h2.x,
                                   l2.x, h2.y, l2.y, m3.x, m3.y, m4.x, m4.y, m5.x, m5.y};
#pragma unroll
    for (int q = 0; q < kMomComp + 6; q++) S.red[q][w][lane] = v[q];
  }
  __syncthreads();
  for (int q = w; q < kMomComp; q += kNodeSub) {  // component 2 m (re), 2 m + 1 (im) over the sub-blocks
    df32 a{0.f, 0.f};
#pragma unroll
    for (int k = 0; k < kNodeSub; k++)
      a = q < 6 ? df_add(a, quick_two_sum(S.red[2 * q][k][lane], S.red[2 * q + 1][k][lane]))
                : df_add_f(a, S.red[q + 6][k][lane]);
    S.mom[q][lane] = make_float2(a.hi, a.lo);
  }
  __syncthreads();
  if (pt < npt) {
    for (int o = w; o < 2 * kNodes; o += kNodeSub) {  // W_q, re and im
      const int q = o >> 1, im = o & 1;
      df32 a{0.f, 0.f};
#pragma unroll
      for (int m = 0; m < kNodes; m++) {
        const float2 l = S.lag[q * kNodes + m], sm = S.mom[2 * m + im][lane];
        a = df_add(a, df_mul(df32{l.x, l.y}, df32{sm.x, sm.y}));
      }
      if (S.bad[lane] == 2) a.hi = __int_as_float(0x7fffffff);  // f0 or f1 is not a number: nor is F
      W[2 * ((int64_t)pt * v.nn + b * kNodes + q) + im] = make_float2(a.hi, a.lo);
    }
  }
}

// ------------------------------------------------------------------ sums over the nodes
__device__ __forceinline__ FastSample node_sample(const FastConst &c, const NodeTab &v, const float4 *W, int i) {
  FastSample s;
  const float4 Lq = v.L[i], Tq = v.T[i], Wq = W[i];
  const float2 tq = v.t[i], wq = v.w[i];
  s.cl = df32{Lq.x, Lq.y};
  s.sl = df32{Lq.z, Lq.w};
  s.t = df32{tq.x, tq.y};
  sample_geometry(c, df32{Tq.x, Tq.y}, df32{Tq.z, Tq.w}, &s);
  s.x = df32{1.f, 0.f};
  s.cp = df32{Wq.x, Wq.y};  // sum of x cos(2 pi Phi) l_q
  s.sp = df32{Wq.z, Wq.w};  // sum of x sin(2 pi Phi) l_q
  s.wt = df32{wq.x, wq.y};
  return s;
}

__global__ void __launch_bounds__(kPtThreads) k_nodes_fg(NodeTab v, const FastConst *fcs, const float4 *W,
                                                         double *partial, int NA) {
  pdl_wait();
  __shared__ FastConst c;
  const int pt = blockIdx.x;
  load_fast_const(fcs + pt, &c);
  __syncthreads();
  df32 acc[26];
#pragma unroll
  for (int q = 0; q < 26; q++) acc[q] = df32{0.f, 0.f};
  int64_t k0, k1;
  block_range(v.nn, &k0, &k1);
  for (int64_t k = k0 + threadIdx.x; k < k1; k += kPtThreads)
    fg_sample<true>(c, node_sample(c, v, W + (int64_t)pt * v.nn, (int)k), acc);
  fast_reduce<26>(acc, 0, NA, partial, pt);
}

template <int SIG>
__global__ void __launch_bounds__(kPtThreads) k_nodes_h(NodeTab v, const FastConst *fcs, const float4 *W,
                                                        double *partial, int NA, int q0) {
  pdl_wait();
  __shared__ FastConst c;
  const int pt = blockIdx.x;
  load_fast_const(fcs + pt, &c);
  __syncthreads();
  df32 acc[23];
#pragma unroll
  for (int q = 0; q < 23; q++) acc[q] = df32{0.f, 0.f};
  int64_t k0, k1;
  block_range(v.nn, &k0, &k1);
  for (int64_t k = k0 + threadIdx.x; k < k1; k += kPtThreads)
    hess_sample<SIG, true>(c, node_sample(c, v, W + (int64_t)pt * v.nn, (int)k), acc);
  fast_reduce<20>(acc, q0 + 20 * SIG, NA, partial, pt);
  fast_reduce<3>(acc + 20, q0 + 40 + 3 * SIG, NA, partial, pt);
}

}  // namespace fs
