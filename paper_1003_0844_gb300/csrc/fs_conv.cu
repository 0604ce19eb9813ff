// The Fourier x2 upsampler's convolution with blocks that keep their transforms on chip.
//
// The odd samples of the upsampled series are the circular convolution of the real data
// with a real kernel (fs_prep.cu), of length M = 2 L.  Two real samples form one complex
// value, z[n] = x[2n] + i x[2n + 1], so the transforms have length L = N1 N2, taken in
// two steps (n = N2 n1 + n2, bin k = k1 + N1 k2) in double-float arithmetic:
//  k_conv_cols_fwd  DFTs over n1 of a few columns n2 straight from the data, twiddle;
//  k_conv_rows      DFTs over n2 of the rows k1 and N1 - k1, which hold each bin k with
//                   its mirror L - k; there the spectrum of the real series is unpacked,
//                   multiplied by the kernel's and packed again, and the inverse DFTs of
//                   the same rows follow, twiddle;
//  k_conv_cols_inv  inverse DFTs over k1, the upsampled series out.
// With Z = DFT_L(z), E' = Z[k] + conj Z[L-k], O' = (Z[k] - conj Z[L-k]) / i and the
// kernel's spectrum H (length M) as He = (H[k] + H[k+L])/2, Ho = W_M^-k (H[k] - H[k+L])/2,
//   Ec = E' He + O' W_L^k Ho,  Oc = O' He + E' Ho,
//   Y[k] = Ec + i Oc,  Y[L-k] = conj(Ec - i Oc)
// is the packed spectrum of the convolution.
//
// What bounds it: the double-float butterflies (about 20 FP32 instructions per real
// addition) and, at these sizes (2^16 to 2^20), the latency of a pass; so three launches
// with every factor of a length-N1 or -N2 transform in shared memory take the place of
// twelve to fifteen radix-16 passes through global memory on transforms of twice the
// length.  Eight values per thread: 64 to 128 threads per sequence, two (1024, 512 points)
// to sixteen (64 points) sequences per block, which gives 128 to 256 blocks at L = 2^17 and
// 2^18.
// Measured for 6 days at 2 s (N = 258,492, L = 2^18): 14.5 + 27 + 12 us, against
// 107 us for fifteen launches of the radix-16 form (kept for series below 2049 samples,
// where it takes fewer and shorter passes, and above 2^20, which these kernels' two
// factors of 1024 do not reach).
#include <type_traits>
#include "fs_internal.h"
#include "fs_blockdft.cuh"

namespace fs {

namespace {

// W_M^e (M = 2 L) from the table of e < L, 0 <= e < M
__device__ __forceinline__ dfc tw_m(const float4 *tw, int64_t e, int64_t L) {
  const dfc w = dfc_ld(tw[e < L ? e : e - L]);
  return e < L ? w : dfc{df_neg(w.re), df_neg(w.im)};
}

// W_LEN^e, e < LEN, of the block from the table of W_M
template <int LEN>
__device__ __forceinline__ void load_table(float4 *dst, const float4 *tw, int64_t L) {
  const int64_t step = 2 * L / LEN;
  for (int e = threadIdx.x; e < LEN; e += BlockDft<LEN>::THREADS) dst[e] = dfc_st(tw_m(tw, e * step, L));
}

// x (n samples of type X) to z, its columns' DFTs; x64, x32: the series as the other
// kernels read it (values that are not finite latch ERRF_NONFINITE and read as zero).
template <int LEN, typename X>
__global__ void __launch_bounds__(BlockDft<LEN>::THREADS) k_conv_cols_fwd(const X *x, double *x64, float *x32,
                                                                          int64_t n, const float4 *tw, float4 *out,
                                                                          int N2, uint32_t *flags) {
  using C = BlockDft<LEN>;
  extern __shared__ float4 sm[];
  float4 *tab = sm + C::SEQ * C::STRIDE;
  const int64_t L = (int64_t)LEN * N2;
  const int c = threadIdx.x % C::SEQ, t = threadIdx.x / C::SEQ;
  const int n2 = blockIdx.x * C::SEQ + c;
  float4 *s = sm + c * C::STRIDE;
  pdl_wait();
  load_table<LEN>(tab, tw, L);
  auto get = [&](int64_t i) {
    if (i >= n) return df32{0.f, 0.f};
    X d = x[i];
    if (!isfinite(d)) {
      atomicOr(flags, ERRF_NONFINITE);
      d = X(0);
    }
    x64[i] = (double)d;
    const float f = (float)d;
    x32[i] = f;
    return sizeof(X) == 4 ? df32{f, 0.f} : df32{f, (float)(d - (X)f)};
  };
  dfc v[8];
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int64_t i = 2 * ((int64_t)N2 * (t + C::T * m) + n2);
    v[m] = dfc{get(i), get(i + 1)};
  }
  block_dft<LEN, -1>(v, t, s, tab);  // its first barrier also covers the table
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int k1 = t + C::T * m;
    const int64_t q = ((int64_t)n2 * k1) & (L - 1);
    out[(int64_t)k1 * N2 + n2] = dfc_st(dfc_mul(v[m], tw_m(tw, 2 * q, L)));
  }
}

// Rows b and N1 - b (block 0: rows 0 and N1/2): forward DFTs, product with the kernel's
// spectrum, inverse DFTs, in place.  kern: He, Ho and W_L^k Ho of the rows 0 .. N1/2 one
// after the other ((N1/2 + 1) N2 values each).
template <int LEN>
__global__ void __launch_bounds__(BlockDft<LEN>::THREADS) k_conv_rows(float4 *buf, const float4 *kern,
                                                                      const float4 *tw, int N1) {
  using C = BlockDft<LEN>;
  constexpr int N2 = LEN;
  extern __shared__ float4 sm[];
  float4 *tab = sm + C::SEQ * C::STRIDE;
  const int64_t L = (int64_t)N1 * N2;
  const int c = threadIdx.x / C::T, t = threadIdx.x % C::T;
  const int b = blockIdx.x * (C::SEQ / 2) + (c >> 1);
  const int row = (c & 1) ? (b == 0 ? N1 / 2 : N1 - b) : b;
  float4 *s = sm + c * C::STRIDE;
  float4 *r = buf + (int64_t)row * N2;
  dfc v[8];
  load_table<LEN>(tab, tw, L);  // the plan's, complete before the columns began
  pdl_wait();
#pragma unroll
  for (int m = 0; m < 8; m++) v[m] = dfc_ld(r[t + C::T * m]);
  block_dft<LEN, -1>(v, t, s, tab);
  __syncthreads();
#pragma unroll
  for (int m = 0; m < 8; m++) s[pad8(t + C::T * m)] = dfc_st(v[m]);
  __syncthreads();
  // the pairs (k, L - k) of the two rows, spread over their 2 T threads
  {
    float4 *s0 = sm + (c & ~1) * C::STRIDE, *s1 = s0 + C::STRIDE;
    const int64_t plane = (int64_t)(N1 / 2 + 1) * N2;
    const int pairs = b == 0 ? N2 + 1 : N2;
    for (int i = (c & 1) * C::T + t; i < pairs; i += 2 * C::T) {
      float4 *p, *q;
      int64_t kk;  // position in a plane of kern
      if (b) {
        p = s0 + pad8(i);
        q = s1 + pad8(N2 - 1 - i);
        kk = (int64_t)b * N2 + i;
      } else if (i <= N2 / 2) {  // row 0
        p = s0 + pad8(i);
        q = s0 + pad8((N2 - i) & (N2 - 1));
        kk = i;
      } else {  // row N1/2
        const int j = i - N2 / 2 - 1;
        p = s1 + pad8(j);
        q = s1 + pad8(N2 - 1 - j);
        kk = (int64_t)(N1 / 2) * N2 + j;
      }
      const dfc z = dfc_ld(*p), zm = dfc_conj(dfc_ld(*q));
      const dfc he = dfc_ld(kern[kk]), ho = dfc_ld(kern[plane + kk]), wo = dfc_ld(kern[2 * plane + kk]);
      const dfc e = dfc_add(z, zm), o = dfc_rot(dfc_sub(z, zm), -1);
      const dfc ec = dfc_add(dfc_mul(e, he), dfc_mul(o, wo));
      const dfc io = dfc_rot(dfc_add(dfc_mul(o, he), dfc_mul(e, ho)), +1);
      *p = dfc_st(dfc_add(ec, io));
      if (q != p) *q = dfc_st(dfc_conj(dfc_sub(ec, io)));
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < 8; m++) v[m] = dfc_ld(s[pad8(t + C::T * m)]);
  block_dft<LEN, +1>(v, t, s, tab);
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int n2 = t + C::T * m;
    const int64_t q = ((int64_t)n2 * row) & (L - 1);
    r[n2] = dfc_st(dfc_mul(v[m], dfc_conj(tw_m(tw, 2 * q, L))));
  }
}

// The inverse columns and the upsampled series: x2[2m] = x[m], x2[2m + 1] = c[m], as
// doubles and (ydf) as double-floats.
template <int LEN, typename X>
__global__ void __launch_bounds__(BlockDft<LEN>::THREADS) k_conv_cols_inv(const float4 *in, const double *x64,
                                                                          const float *x32, const float4 *tw,
                                                                          double *x2, float2 *ydf, int64_t n, int N2) {
  using C = BlockDft<LEN>;
  extern __shared__ float4 sm[];
  float4 *tab = sm + C::SEQ * C::STRIDE;
  const int64_t L = (int64_t)LEN * N2;
  const int c = threadIdx.x % C::SEQ, t = threadIdx.x / C::SEQ;
  const int n2 = blockIdx.x * C::SEQ + c;
  float4 *s = sm + c * C::STRIDE;
  dfc v[8];
  load_table<LEN>(tab, tw, L);
  pdl_wait();
#pragma unroll
  for (int m = 0; m < 8; m++) v[m] = dfc_ld(in[(int64_t)(t + C::T * m) * N2 + n2]);
  block_dft<LEN, +1>(v, t, s, tab);
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int64_t i = 2 * ((int64_t)N2 * (t + C::T * m) + n2);
#pragma unroll
    for (int h = 0; h < 2; h++) {
      if (i + h >= n) continue;
      const df32 o = h ? v[m].im : v[m].re;
      const double e = x64[i + h];
      const df32 ed = sizeof(X) == 4 ? df32{x32[i + h], 0.f} : df_from_double(e);  // FP32 data is its own high word
      x2[2 * (i + h)] = e;
      x2[2 * (i + h) + 1] = (double)o.hi + (double)o.lo;
      ydf[2 * (i + h)] = make_float2(ed.hi, ed.lo);
      ydf[2 * (i + h) + 1] = make_float2(o.hi, o.lo);
    }
  }
}

// The kernel's spectrum H (length M = 2 L, natural order) as the planes of k_conv_rows.
__global__ void k_conv_kernel(const float4 *H, const float4 *tw, float4 *kern, int N1, int N2) {
  const int64_t L = (int64_t)N1 * N2, plane = (int64_t)(N1 / 2 + 1) * N2;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= plane) return;
  const int64_t k = i / N2 + N1 * (i % N2);
  const dfc a = dfc_ld(H[k]), b = dfc_ld(H[k + L]), w = dfc_ld(tw[k]);
  auto half = [](const dfc &v) { return dfc{df_scale(v.re, 0.5f), df_scale(v.im, 0.5f)}; };
  const dfc wo = half(dfc_mul(dfc_sub(a, b), w));  // W_L^k Ho = W_M^k (H[k] - H[k + L]) / 2
  kern[i] = dfc_st(half(dfc_add(a, b)));
  kern[plane + i] = dfc_st(half(dfc_mul(dfc_sub(a, b), dfc_conj(w))));
  kern[2 * plane + i] = dfc_st(wo);
}

void conv_split(int64_t L, int *N1, int *N2) {
  int q = 0;
  while (((int64_t)1 << q) < L) q++;
  *N1 = 1 << ((q + 1) / 2);
  *N2 = 1 << (q / 2);
}

template <int LEN, typename K, typename... Args>
cudaError_t launch_conv(K *kern, int grid, cudaStream_t st, Args... args) {
  using C = BlockDft<LEN>;
  if constexpr (C::SMEM > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(kern, dim3(grid), dim3(C::THREADS), C::SMEM, st, args...);
}

template <typename F>
cudaError_t by_length(int len, F &&f) {
  switch (len) {
    case 64: return f(std::integral_constant<int, 64>{});
    case 128: return f(std::integral_constant<int, 128>{});
    case 256: return f(std::integral_constant<int, 256>{});
    case 512: return f(std::integral_constant<int, 512>{});
    case 1024: return f(std::integral_constant<int, 1024>{});
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool conv_supported(int64_t M) { return M >= (1 << 13) && M <= (1 << 21); }

int64_t conv_kernel_elems(int64_t M) {
  int N1, N2;
  conv_split(M / 2, &N1, &N2);
  return 3 * (int64_t)(N1 / 2 + 1) * N2;
}

cudaError_t conv_plan(const float4 *H, const float4 *tw, float4 *kern, int64_t M, cudaStream_t st) {
  int N1, N2;
  conv_split(M / 2, &N1, &N2);
  const int64_t plane = (int64_t)(N1 / 2 + 1) * N2;
  k_conv_kernel<<<(unsigned)((plane + 255) / 256), 256, 0, st>>>(H, tw, kern, N1, N2);
  return cudaGetLastError();
}

cudaError_t conv_upsample(const void *x, bool x_double, double *x64, float *x32, int64_t n, int64_t M,
                          const float4 *kern, const float4 *tw, float4 *buf, double *x2, float2 *ydf, uint32_t *flags,
                          cudaStream_t st) {
  int N1, N2;
  conv_split(M / 2, &N1, &N2);
  cudaError_t e = by_length(N1, [&](auto len) {
    constexpr int LEN = decltype(len)::value;
    const int grid = N2 / BlockDft<LEN>::SEQ;
    return x_double ? launch_conv<LEN>(k_conv_cols_fwd<LEN, double>, grid, st, (const double *)x, x64, x32, n, tw, buf,
                                       N2, flags)
                    : launch_conv<LEN>(k_conv_cols_fwd<LEN, float>, grid, st, (const float *)x, x64, x32, n, tw, buf,
                                       N2, flags);
  });
  if (e != cudaSuccess) return e;
  e = by_length(N2, [&](auto len) {
    constexpr int LEN = decltype(len)::value;
    return launch_conv<LEN>(k_conv_rows<LEN>, N1 / BlockDft<LEN>::SEQ, st, buf, kern, tw, N1);
  });
  if (e != cudaSuccess) return e;
  return by_length(N1, [&](auto len) {
    constexpr int LEN = decltype(len)::value;
    const int grid = N2 / BlockDft<LEN>::SEQ;
    const float4 *in = buf;
    const double *xd = x64;
    const float *xf = x32;
    return x_double ? launch_conv<LEN>(k_conv_cols_inv<LEN, double>, grid, st, in, xd, xf, tw, x2, ydf, n, N2)
                    : launch_conv<LEN>(k_conv_cols_inv<LEN, float>, grid, st, in, xd, xf, tw, x2, ydf, n, N2);
  });
}

}  // namespace fs
