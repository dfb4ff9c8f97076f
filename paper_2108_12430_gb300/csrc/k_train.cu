// Training kernels (FP32): BatchNorm fold and its chain rule, the band-limited
// loss and Adam (weight gradients: k_wgrad_f32.cu, k_wgrad_tc.cu).
//
// Data gradients reuse the forward conv kernel (a conv's data gradient is a
// transposed conv with the transposed weights and vice versa), with the
// activation derivative fused into its epilogue.  Every reduction here runs
// in a fixed order, so a gradient is bitwise reproducible.
#include "gw_train.h"

namespace gw {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  float t = 0.f;
  if (threadIdx.x == 0)
    for (int i = 0; i < nw; ++i) t += red[i];
  return t;  // valid in thread 0
}

// Folded weights of one layer in the conv kernel's layout [C_in][K][C_out
// padded] (wf), the same values with the channels exchanged, [C_out][K][C_in
// padded] (wT, the data gradient's weights), and the folded bias (bf); the
// padding is zero from the start and never written:
//   sc[o] = gamma[o] / sqrt(var[o] + eps),  w' = w sc[o],  b' = (b - mean) sc + beta.
// One CTA per (layer, output channel): the channel's factor takes an FP64
// square root and division, which this chip does slowly, so one thread does it
// (per element it made the eight layers take 8.7 us, this takes 6 us).
__device__ __forceinline__ void fold_body(const FoldArgs& f, int o) {
  __shared__ double s_sc;
  if (threadIdx.x == 0) {
    const double sc = f.bn ? (double)f.p[f.off_g + o] / sqrt((double)f.p[f.off_var + o] + (double)kBnEps) : 1.0;
    const double b = f.p[f.off_b + o];
    f.bf[o] = f.bn ? (float)((b - (double)f.p[f.off_mu + o]) * sc + (double)f.p[f.off_be + o]) : (float)b;
    s_sc = sc;
  }
  __syncthreads();
  const double sc = s_sc;
  for (int e = threadIdx.x; e < f.cin * f.K; e += blockDim.x) {
    const int i = e / f.K, k = e - i * f.K;
    const int64_t raw = f.transposed ? ((int64_t)i * f.cout + o) * f.K + k : (int64_t)o * f.cin * f.K + e;
    const float w = (float)((double)f.p[f.off_w + raw] * sc);
    f.wf[((int64_t)i * f.K + k) * conv_f32_cop(f.cout) + o] = w;
    if (f.wT) f.wT[((int64_t)o * f.K + k) * conv_f32_cop(f.cin) + i] = w;
  }
}
struct FoldList {
  FoldArgs f[kFoldMax];
};
__global__ void fold_many_kernel(const __grid_constant__ FoldList l) {
  const FoldArgs& f = l.f[blockIdx.y];
  if ((int)blockIdx.x < f.cout) fold_body(f, blockIdx.x);
}

// Chain rule from the folded parameters' gradients (dWf in the layer's
// gradient layout, dbf) to the raw ones; one CTA per output channel o:
//   dw = dWf sc,  db = dbf sc,  dbeta = dbf,
//   dgamma = a (sum_{i,k} w dWf + dbf (b - mean)),  a = 1 / sqrt(var + eps);
// running mean and variance are not trained (gradient 0).
__device__ __forceinline__ void unfold_body(const FoldArgs& f, const float* __restrict__ dWf, int dw_in_major,
                                            const float* __restrict__ dbf, float* __restrict__ dp, int o) {
  __shared__ float red[kThreads / 32];
  __shared__ double s_a;  // one FP64 square root and division per channel
  if (threadIdx.x == 0) s_a = f.bn ? 1.0 / sqrt((double)f.p[f.off_var + o] + (double)kBnEps) : 1.0;
  __syncthreads();
  const double a = s_a, sc = f.bn ? (double)f.p[f.off_g + o] * a : 1.0;
  float dot = 0.f;
  for (int j = threadIdx.x; j < f.cin * f.K; j += blockDim.x) {
    const int i = j / f.K, k = j % f.K;
    const int64_t g = dw_in_major ? ((int64_t)i * f.cout + o) * f.K + k : ((int64_t)o * f.cin + i) * f.K + k;
    const int64_t raw = f.transposed ? ((int64_t)i * f.cout + o) * f.K + k : ((int64_t)o * f.cin + i) * f.K + k;
    const float d = dWf[g];
    dp[f.off_w + raw] = (float)((double)d * sc);
    dot = fmaf(f.p[f.off_w + raw], d, dot);
  }
  dot = block_sum(dot, red);
  if (threadIdx.x == 0) {
    const double db = dbf[o];
    dp[f.off_b + o] = (float)(db * sc);
    if (f.bn) {
      dp[f.off_g + o] = (float)(a * ((double)dot + db * ((double)f.p[f.off_b + o] - (double)f.p[f.off_mu + o])));
      dp[f.off_be + o] = (float)db;
      dp[f.off_mu + o] = 0.f;
      dp[f.off_var + o] = 0.f;
    }
  }
}

// Several layers' unfolds in one launch: block (o, i) is output channel o of
// layer i.
struct UnfoldList {
  UnfoldItem u[kFoldMax];
};
__global__ void unfold_many_kernel(const __grid_constant__ UnfoldList l, float* __restrict__ dp) {
  const UnfoldItem& u = l.u[blockIdx.y];
  if ((int)blockIdx.x >= u.f.cout) return;
  unfold_body(u.f, u.dWf, u.dw_in_major, u.dbf, dp, blockIdx.x);
}

// x_std[b][c][t] = (x[b][c][t] - mean[c]) / std[c]; one CTA per 1024 samples of
// a row (64-bit index arithmetic per element made 32 x 21 x 8192 take 19 us,
// this takes 8 us).
__global__ void __launch_bounds__(kThreads) standardise_kernel(const float* __restrict__ x, int C, int L, int per_row,
                                                               const float* __restrict__ mean,
                                                               const float* __restrict__ istd, float* __restrict__ y) {
  const int row = blockIdx.x / per_row, t0 = (blockIdx.x - row * per_row) * 4 * kThreads, c = row % C;
  const float m = mean[c], s = istd[c];
  const float* xr = x + (int64_t)row * L;
  float* yr = y + (int64_t)row * L;
  const int t = t0 + 4 * threadIdx.x;
  if (t + 4 <= L && ((((uintptr_t)(xr + t)) | ((uintptr_t)(yr + t))) & 15) == 0) {
    const float4 v = *reinterpret_cast<const float4*>(xr + t);
    *reinterpret_cast<float4*>(yr + t) = make_float4((v.x - m) * s, (v.y - m) * s, (v.z - m) * s, (v.w - m) * s);
  } else {
    for (int i = t; i < min(t + 4, L); ++i) yr[i] = (xr[i] - m) * s;
  }
}

// loss = inv_n * sum of the n partial sums (one CTA).
__global__ void loss_final_kernel(const float* __restrict__ part, int n, float inv_n, float* __restrict__ loss) {
  __shared__ float red[kThreads / 32];
  float s = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
  s = block_sum(s, red);
  if (threadIdx.x == 0) *loss = s * inv_n;
}

// Adam with bias correction (Kingma & Ba, Algorithm 1), FP32 state.
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// The same update with the step count t read from device memory (bias
// corrections 1 - b1^t, 1 - b2^t worked out per thread), after
// adam_count_kernel has incremented it.
__global__ void adam_dev_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                                float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                                const int* __restrict__ step) {
  const float t = (float)*step;
  const float c1 = 1.f - powf(b1, t), c2 = 1.f - powf(b2, t);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}
__global__ void adam_count_kernel(int* step) { *step += 1; }

int grid_for(int64_t n) {
  const int64_t b = (n + kThreads - 1) / kThreads;
  return (int)std::min<int64_t>(std::max<int64_t>(b, 1), 1216);
}

}  // namespace

void launch_fold_many(const FoldArgs* f, int n, cudaStream_t st) {
  GW_CHECK_ARG(n >= 1 && n <= kFoldMax, "fold list size");
  FoldList l{};
  int mx = 1;
  for (int i = 0; i < n; ++i) {
    l.f[i] = f[i];
    mx = std::max(mx, f[i].cout);
  }
  fold_many_kernel<<<dim3(mx, n), kThreads, 0, st>>>(l);
  GW_LAUNCH_CHECK();
}

void launch_unfold_many(const UnfoldItem* u, int n, float* dp, cudaStream_t st) {
  GW_CHECK_ARG(n >= 1 && n <= kFoldMax, "unfold list size");
  UnfoldList l{};
  int mx = 1;
  for (int i = 0; i < n; ++i) {
    l.u[i] = u[i];
    mx = std::max(mx, u[i].f.cout);
  }
  unfold_many_kernel<<<dim3(mx, n), kThreads, 0, st>>>(l, dp);
  GW_LAUNCH_CHECK();
}

void launch_standardise(const float* x, int B, int C, int L, const float* mean, const float* istd, float* y,
                        cudaStream_t st) {
  const int per_row = (L + 4 * kThreads - 1) / (4 * kThreads);
  standardise_kernel<<<(unsigned)((int64_t)B * C * per_row), kThreads, 0, st>>>(x, C, L, per_row, mean, istd, y);
  GW_LAUNCH_CHECK();
}

size_t band_loss_part_floats(int B, int L, int K) { return (size_t)fir_f32_parts(B, L - K + 1); }

void launch_band_loss(const float* strain, const float* y_hat, int B, int L, const float* taps, int K, float* r,
                      float* part, float* loss, cudaStream_t st) {
  const int Lr = L - K + 1;
  FirArgs a = fir_valid_args(strain, L, r, Lr, taps, K, Lr);
  a.x2 = y_hat;
  a.part = part;
  launch_fir_f32(a, B, st);
  loss_final_kernel<<<1, kThreads, 0, st>>>(part, (int)band_loss_part_floats(B, L, K),
                                            1.f / ((float)B * (float)Lr), loss);
  GW_LAUNCH_CHECK();
}

void launch_band_loss_backward(const float* r, int B, int L, const float* taps, int K, const float* dloss,
                               float* dy_hat, cudaStream_t st) {
  const int Lr = L - K + 1;
  // dL/dy_hat[m] = -(2 / N) sum_k g[k] r[m - k]: the FIR's adjoint of r
  FirArgs a = fir_adjoint_args(r, Lr, Lr, dy_hat, L, taps, K, -2.f / ((float)B * (float)Lr));
  a.dscale = dloss;
  launch_fir_f32(a, B, st);
}

void launch_adam_dev(float* p, const float* g, float* m, float* v, int64_t n, int* step, float lr, float b1,
                     float b2, float eps, cudaStream_t st) {
  adam_count_kernel<<<1, 1, 0, st>>>(step);
  GW_LAUNCH_CHECK();
  adam_dev_kernel<<<grid_for(n), kThreads, 0, st>>>(p, g, m, v, n, lr, b1, b2, eps, step);
  GW_LAUNCH_CHECK();
}

void launch_adam(float* p, const float* g, float* m, float* v, int64_t n, int step, float lr, float b1, float b2,
                 float eps, cudaStream_t st) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  adam_kernel<<<grid_for(n), kThreads, 0, st>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
  GW_LAUNCH_CHECK();
}

}  // namespace gw
