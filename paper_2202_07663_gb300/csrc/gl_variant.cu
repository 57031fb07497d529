// gl_variant.cu - the likelihood with the observed-image variance of
// arXiv:2202.07663, Sec. 2.1.2 (sigma_tot^2 = sigma_bkg^2 + I_obs/(G t_exp),
// negative observed pixels counted as zero), profiled over the two light
// amplitudes. With a parameter-independent variance the model is linear in
// (I_l, I_s), M = I_l A_l + I_s A_s, and the amplitudes maximising log L solve
//   [<A_l,A_l> <A_l,A_s>; <A_s,A_l> <A_s,A_s>] [I_l; I_s] = [<A_l,D>; <A_s,D>],
// <a,b> = sum_pixels a b / sigma_tot^2. The basis images A come from the
// simulation path at unit amplitudes (one ray pass for both, k_ray_fwd_basis);
// these kernels reduce and solve the 2x2 systems (FP64), evaluate log L and
// d log L / d M of the profiled model, and zero the amplitude entries of the
// profiled gradient.
#include <cuda_runtime.h>

#include "gl_internal.h"

namespace {

constexpr int kIL = 14, kIS = 21;
constexpr double kSingular = 1e-12;   // relative size below which a self-product or det counts as zero
constexpr int kSolveThreads = 512;

__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < int(blockDim.x >> 5); ++i) t += sh[i];
  return t;   // valid in thread 0
}

// A number as an unevaluated sum of two floats, h = fl(h + l): about 48 bits.
// The FP64 pipe issues two lanes a clock on an SM, the FP32 pipe 128, so the
// weighted inner products run in these (the error-free sum and product of
// Dekker 1971 and Knuth, TAOCP 4.2.2, the product's error from one FMA).
struct F2Sum {
  float h, l;
};
__device__ __forceinline__ F2Sum two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ void add_to(F2Sum& s, float h, float l) {
  const float t = __fadd_rn(s.h, h);
  const float bb = __fsub_rn(t, s.h);
  const float e = __fadd_rn(__fsub_rn(s.h, __fsub_rn(t, bb)), __fsub_rn(h, bb));
  s.h = t;
  s.l = __fadd_rn(s.l, __fadd_rn(e, l));
}
// a b + c's low part: (a.h + a.l) b as a pair
__device__ __forceinline__ F2Sum times(F2Sum a, float b) {
  const F2Sum p = two_prod(a.h, b);
  return {p.h, __fmaf_rn(a.l, b, p.l)};
}

// The five weighted inner products of the block's images over its threads, in
// pairs of floats: <Al,Al>, <Al,As>, <As,As>, <Al,D>, <As,D>, weights
// scale / sigma2 (scale, a power of two near the smallest sigma2, keeps them
// near 1; the solution does not depend on it). out is valid in every thread
// after the call.
__device__ void inner_products(int HW, const float* Al, const float* As, const float* data, const float* sigma2,
                               double (*sh)[5], double* out) {
  __shared__ float s_min[kSolveThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float m = 3.4e38f;
  for (int i = threadIdx.x; i < HW; i += blockDim.x) m = fminf(m, sigma2[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) s_min[w] = m;
  __syncthreads();
  for (int i = 0; i < nw; ++i) m = fminf(m, s_min[i]);
  const float inv_scale = exp2f(-float(ilogbf(m)));   // exact
  F2Sum acc[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) acc[q] = {0.f, 0.f};
#pragma unroll 4
  for (int i = threadIdx.x; i < HW; i += blockDim.x) {
    const float v = sigma2[i] * inv_scale, al = Al[i], as = As[i], d = data[i];
    const float wh = __fdiv_rn(1.f, v);
    const F2Sum wt = {wh, __fmul_rn(wh, __fmaf_rn(-wh, v, 1.f))};   // one Newton step's residual
    const F2Sum wl = times(wt, al), ws = times(wt, as);
    F2Sum t = times(wl, al);
    add_to(acc[0], t.h, t.l);
    t = times(wl, as);
    add_to(acc[1], t.h, t.l);
    t = times(ws, as);
    add_to(acc[2], t.h, t.l);
    t = times(wl, d);
    add_to(acc[3], t.h, t.l);
    t = times(ws, d);
    add_to(acc[4], t.h, t.l);
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h = __shfl_xor_sync(0xffffffffu, acc[q].h, o), l = __shfl_xor_sync(0xffffffffu, acc[q].l, o);
      add_to(acc[q], h, l);
    }
    if (lane == 0) sh[w][q] = double(acc[q].h) + double(acc[q].l);
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    double v = 0.0;
    for (int i = 0; i < nw; ++i) v += sh[i][threadIdx.x];
    sh[nw][threadIdx.x] = v;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 5; ++q) out[q] = sh[nw][q];
}

// The same in FP64, for images outside the range in which the pairs carry
// their precision.
__device__ void inner_products_fp64(int HW, const float* Al, const float* As, const float* data, const float* sigma2,
                                    double* red, double (*sh)[5], double* out) {
  double g[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int i = threadIdx.x; i < HW; i += blockDim.x) {
    const double w = 1.0 / double(sigma2[i]);
    const double al = Al[i], as = As[i], d = data[i];
    g[0] += w * al * al;
    g[1] += w * al * as;
    g[2] += w * as * as;
    g[3] += w * al * d;
    g[4] += w * as * d;
  }
  for (int q = 0; q < 5; ++q) {
    const double v = block_sum(g[q], red);
    if (threadIdx.x == 0) sh[0][q] = v;
  }
  __syncthreads();
  for (int q = 0; q < 5; ++q) out[q] = sh[0][q];
}

// One block per vector: the five weighted inner products, the 2x2 solve, the
// amplitudes (FP64) and the parameter row with the amplitudes substituted;
// then, with loglik set, the model M = I_l A_l + I_s A_s (the PSF convolution
// is linear, so the convolved basis images give the convolved model), log L
// and chi^2 (FP32 per pixel and thread, FP64 across threads) and, with dldm
// set, d log L / d M per pixel into dldm[b] (the next pass correlates it with
// the PSF for the gradient). The inner products were bound by the FP64 pipe
// (a division and some twenty operations per pixel): 300 vectors of 80 x 80
// 77 us, 28 us with pairs of floats and 512 threads (with launch gaps, between
// events).
__global__ void __launch_bounds__(kSolveThreads) k_amp_solve(int B, int HW, const float* __restrict__ images,
                                                             const float* __restrict__ data,
                                                             const float* __restrict__ sigma2,
                                                             const float* __restrict__ params,
                                                             float* __restrict__ params_out,
                                                             double* __restrict__ amps, float inv_gain,
                                                             double* __restrict__ loglik,
                                                             double* __restrict__ chi2, float* __restrict__ dldm) {
  __shared__ double sh[kSolveThreads / 32];
  __shared__ double sh5[kSolveThreads / 32 + 1][5];
  __shared__ double s_amp[2];
  const int b = blockIdx.x;
  if (b >= B) return;
  const float* Al = images + size_t(2 * b) * HW;
  const float* As = images + size_t(2 * b + 1) * HW;
  double g[5];
  inner_products(HW, Al, As, data, sigma2, sh5, g);
  // a pair's low part is lost below about 2^-126 and the high part overflows
  // at 2^128; the sums are the same in every thread, so the block agrees
  const double big = fmax(g[0], g[2]);
  if (!(big > 1e-20 && big < 1e36)) inner_products_fp64(HW, Al, As, data, sigma2, sh, sh5, g);
  if (threadIdx.x == 0) {
    const double gll = g[0], gls = g[1], gss = g[2], rl = g[3], rs = g[4];
    double il = 0.0, is = 0.0;
    const double gmax = fmax(gll, gss);
    const bool live_l = gll > kSingular * gmax, live_s = gss > kSingular * gmax;
    const double det = gll * gss - gls * gls;
    if (live_l && live_s && det > kSingular * gll * gss) {
      il = (gss * rl - gls * rs) / det;
      is = (gll * rs - gls * rl) / det;
    } else if (live_l || live_s) {
      if (live_l && (!live_s || gll >= gss)) {
        il = rl / gll;
      } else {
        is = rs / gss;
      }
    }
    amps[2 * b] = il;
    amps[2 * b + 1] = is;
    s_amp[0] = il;
    s_amp[1] = is;
  }
  for (int j = threadIdx.x; j < gl::NPARAM; j += blockDim.x) {
    // thread 0 wrote amps above; the other rows are copies of the input
    if (j != kIL && j != kIS) params_out[size_t(b) * gl::NPARAM + j] = params[size_t(b) * gl::NPARAM + j];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    params_out[size_t(b) * gl::NPARAM + kIL] = float(s_amp[0]);
    params_out[size_t(b) * gl::NPARAM + kIS] = float(s_amp[1]);
  }
  if (!loglik) return;
  // the amplitudes as the model evaluation uses them (the substituted FP32 row)
  const float il = float(s_amp[0]), is = float(s_amp[1]);
  float ll = 0.f, c2 = 0.f;
#pragma unroll 4
  for (int i = threadIdx.x; i < HW; i += blockDim.x) {
    const float M = fmaf(il, Al[i], is * As[i]);
    const float v = fmaf(M, inv_gain, sigma2[i]);
    const float res = data[i] - M;
    const float iv = 1.0f / v;
    const float t2 = res * res * iv;
    c2 += t2;
    ll += t2 + logf(6.28318530717958648f * v);
    // d log L / d M = res/v + (res^2/v^2 - 1/v) / (2 G t_exp)
    if (dldm) dldm[size_t(b) * HW + i] = fmaf(0.5f * inv_gain, fmaf(t2, iv, -iv), res * iv);
  }
  // the threads' sums as pairs of floats within a warp, FP64 across warps
  F2Sum sum[2] = {{ll, 0.f}, {c2, 0.f}};
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h = __shfl_xor_sync(0xffffffffu, sum[q].h, o), l = __shfl_xor_sync(0xffffffffu, sum[q].l, o);
      add_to(sum[q], h, l);
    }
  if ((threadIdx.x & 31) == 0) {
    sh5[threadIdx.x >> 5][0] = double(sum[0].h) + double(sum[0].l);
    sh5[threadIdx.x >> 5][1] = double(sum[1].h) + double(sum[1].l);
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double v = 0.0;
    for (int i = 0; i < int(blockDim.x >> 5); ++i) v += sh5[i][threadIdx.x];
    if (threadIdx.x == 0) loglik[b] = -0.5 * v;
    if (threadIdx.x == 1 && chi2) chi2[b] = v;
  }
}

__global__ void k_zero_amp_grad(int B, double* __restrict__ grad) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) {
    grad[size_t(b) * gl::NPARAM + kIL] = 0.0;
    grad[size_t(b) * gl::NPARAM + kIS] = 0.0;
  }
}

int grid_for(long long n, int threads) {
  long long g = (n + threads - 1) / threads;
  return int(g < 1 ? 1 : (g > 4096 ? 4096 : g));
}

}  // namespace

namespace gl_internal {

cudaError_t launch_amp_solve(int B, int HW, const float* images, const float* data, const float* sigma2,
                             const float* params, float* params_out, double* amps, float inv_gain, double* loglik,
                             double* chi2, float* dldm, cudaStream_t st) {
  hooks()->before(GL_K_OTHER, st);
  k_amp_solve<<<B, kSolveThreads, 0, st>>>(B, HW, images, data, sigma2, params, params_out, amps, inv_gain, loglik,
                                           chi2, dldm);
  return hooks()->after(GL_K_OTHER, st);
}

cudaError_t launch_zero_amp_grad(int B, double* grad, cudaStream_t st) {
  hooks()->before(GL_K_OTHER, st);
  k_zero_amp_grad<<<grid_for(B, 128), 128, 0, st>>>(B, grad);
  return hooks()->after(GL_K_OTHER, st);
}

}  // namespace gl_internal
