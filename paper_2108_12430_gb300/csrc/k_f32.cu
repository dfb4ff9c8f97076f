// FP32 SIMT kernels of the plain-FP32 path besides the convs (k_conv_f32.cu):
// FIR, pool + head, range of a tensor.
#include "gw_internal.h"

namespace gw {

namespace {

constexpr int kThreads = 256;

// FIR over one row:
//   y[r][n] = scale * sum_k h'[k] x[r][n + k + x_off],  x zero outside [0, x_len),
// h' = h (rev = 0) or h reversed (rev = 1).  Valid mode: x_off = 0,
// x_len = lout + ntaps - 1.  Its adjoint (dx[m] = sum_k h[k] dy[m - k]) is
// x_off = -(ntaps - 1), rev = 1.
// CTA: kFirTile outputs, kFirThreads threads of kFirOut consecutive outputs
// each.  Taps go in blocks of 8 (zero-padded): per block a thread loads the 8
// taps and the 16 inputs its outputs read as float4 vectors from shared
// memory, so that every loaded value feeds 4-8 FMAs.  Each output's sum runs
// over the taps in order.
constexpr int kFirThreads = 128, kFirOut = 8, kFirTile = kFirThreads * kFirOut;
__global__ void __launch_bounds__(kFirThreads) fir_f32_kernel(const float* __restrict__ x, int64_t x_row,
                                                              float* __restrict__ y, int64_t y_row,
                                                              const float* __restrict__ h, int ntaps, int lout,
                                                              int x_off, int x_len, int rev, float scale) {
  extern __shared__ __align__(16) float smem[];
  const int npad = (ntaps + 7) / 8 * 8;
  float* hs = smem;         // [npad]
  float* xs = smem + npad;  // [kFirTile + npad + 8]
  const int r = blockIdx.y, n0 = blockIdx.x * kFirTile;
  const float* xr = x + (int64_t)r * x_row;
  const int span = kFirTile + npad + 8;
  for (int e = threadIdx.x; e < npad; e += kFirThreads) hs[e] = e < ntaps ? h[rev ? ntaps - 1 - e : e] : 0.f;
  for (int e = threadIdx.x; e < span; e += kFirThreads) {
    const int q = n0 + e + x_off;
    xs[e] = (q >= 0 && q < x_len) ? xr[q] : 0.f;
  }
  __syncthreads();
  float acc[kFirOut];
#pragma unroll
  for (int j = 0; j < kFirOut; ++j) acc[j] = 0.f;
  const float* xt = xs + threadIdx.x * kFirOut;
  for (int kb = 0; kb < npad; kb += 8) {
    float hv[8], xv[16];
    const float4 h0 = *reinterpret_cast<const float4*>(hs + kb), h1 = *reinterpret_cast<const float4*>(hs + kb + 4);
    hv[0] = h0.x, hv[1] = h0.y, hv[2] = h0.z, hv[3] = h0.w, hv[4] = h1.x, hv[5] = h1.y, hv[6] = h1.z, hv[7] = h1.w;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(xt + kb + 4 * q);
      xv[4 * q] = v.x, xv[4 * q + 1] = v.y, xv[4 * q + 2] = v.z, xv[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
#pragma unroll
      for (int j = 0; j < kFirOut; ++j) acc[j] = fmaf(hv[kk], xv[j + kk], acc[j]);
  }
#pragma unroll
  for (int j = 0; j < kFirOut; ++j) {
    const int n = n0 + threadIdx.x * kFirOut + j;
    if (n < lout) y[(int64_t)r * y_row + n] = scale * acc[j];
  }
}

// Global average pool over time followed by the linear head; one CTA per item.
__global__ void __launch_bounds__(kThreads) gap_linear_f32_kernel(const float* __restrict__ h, int64_t hb,
                                                                  int64_t hc, int C, int L,
                                                                  const float* __restrict__ w,
                                                                  const float* __restrict__ bias,
                                                                  float* __restrict__ out) {
  __shared__ float red[kThreads / 32];
  const int b = blockIdx.x;
  float part = 0.f;
  for (int c = threadIdx.x; c < C; c += kThreads) {
    const float* row = h + (int64_t)b * hb + (int64_t)c * hc;
    float sum = 0.f;
    for (int t = 0; t < L; ++t) sum += row[t];
    part = fmaf(sum / (float)L, w[c], part);
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    float v = 0.f;
    for (int i = 0; i < kThreads / 32; ++i) v += red[i];
    out[b] = v + bias[0];
  }
}

// *amax = max(*amax, max_i |x[i]|): block maximum, then an atomic max on the
// bit pattern (non-negative floats order like their bits as integers, and a
// maximum does not depend on the order it is taken in).
__global__ void __launch_bounds__(kThreads) absmax_kernel(const float* __restrict__ x, int64_t n,
                                                         float* __restrict__ amax) {
  __shared__ float red[kThreads / 32];
  float m = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads)
    m = fmaxf(m, fabsf(x[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kThreads / 32; ++i) m = fmaxf(m, red[i]);
    atomicMax(reinterpret_cast<int*>(amax), __float_as_int(m));
  }
}

}  // namespace

void launch_absmax(const float* x, int64_t n, float* amax, cudaStream_t st) {
  const int64_t blocks = std::min<int64_t>((n + kThreads - 1) / kThreads, 1216);
  absmax_kernel<<<(int)std::max<int64_t>(blocks, 1), kThreads, 0, st>>>(x, n, amax);
  GW_LAUNCH_CHECK();
}

void launch_fir_f32(const float* x, int64_t x_row, float* y, int64_t y_row, int rows, const float* taps,
                    int ntaps, int lout, cudaStream_t st, int x_off, int x_len, int rev, float scale) {
  if (x_len < 0) x_len = lout + ntaps - 1;
  const int npad = (ntaps + 7) / 8 * 8;
  const size_t smem = (size_t)(npad + kFirTile + npad + 8) * 4;
  GW_CHECK_ARG(smem <= 200 * 1024, "FIR too long for the FP32 kernel");
  set_smem_limit_once(fir_f32_kernel, 200 * 1024);
  dim3 grid((lout + kFirTile - 1) / kFirTile, rows);
  fir_f32_kernel<<<grid, kFirThreads, smem, st>>>(x, x_row, y, y_row, taps, ntaps, lout, x_off, x_len, rev, scale);
  GW_LAUNCH_CHECK();
}

void launch_gap_linear_f32(const float* h, int64_t hb, int64_t hc, int B, int C, int L, const float* w,
                           const float* b, float* out, cudaStream_t st) {
  gap_linear_f32_kernel<<<B, kThreads, 0, st>>>(h, hb, hc, C, L, w, b, out);
  GW_LAUNCH_CHECK();
}

}  // namespace gw
