// FP32 SIMT kernels of the plain-FP32 path besides the convs (k_conv_f32.cu):
// FIR, pool + head, range of a tensor.
#include <cmath>

#include "gw_internal.h"

namespace gw {

namespace {

constexpr int kThreads = 256;

// FIR over one row:
//   y[r][n] = scale * sum_k h'[k] x[r][n + k + x_off],  x zero outside [0, x_len),
// h' = h (rev = 0) or h reversed (rev = 1).  Valid mode: x_off = 0,
// x_len = lout + ntaps - 1.  Its adjoint (dx[m] = sum_k h[k] dy[m - k]) is
// x_off = -(ntaps - 1), rev = 1.  Optionally x - x2 is filtered, y is
// multiplied by *dscale, and the CTA's sum of y^2 goes to part.
//
// Bound: the FP32 FMA pipe (2049 FMAs per output on 8 bytes).  A thread keeps
// NO consecutive outputs and slides a register window over the taps: per 16
// taps it loads 16 new samples and 16 taps for 16 NO FMAs.  Two windows take
// turns, so that sliding costs no moves: with few outputs a scheduler has one
// warp, and every other instruction shows (a packed-FMA version spends moves on
// its pairs: 35 us where this takes 27 us for 32 rows of 6144 outputs).  Sample
// rows are padded so that the threads' 16-byte loads fall into distinct banks;
// taps and samples are staged by cp.async.  Each output is one FMA chain over
// the taps in order; the last taps run one by one, so that no sample beyond an
// output's own taps takes part.
//
// Measured (GB300, 2049 taps, against 8 outputs per thread staged through
// registers): 512 rows of 2048 outputs 136 -> 83 us (52 TFLOP/s), 32 rows of 6144
// 45 -> 27 us; the training loss's difference and sum of squares (18 us in
// launches of their own) run in the same pass.
constexpr int kFirMaxThreads = 128;
constexpr int kFirTaps = 2048;  // taps per shared-memory block
constexpr int kFirMaxTaps = 25080;

// Floats before sample p of a staged tile: NO per thread, then 4 of padding
// (none needed at NO = 4).
template <int NO>
__host__ __device__ constexpr int fir_at(int p) {
  return NO == 4 ? p : p / NO * (NO + 4) + p % NO;
}

// 4 bytes to shared memory, zero-filled when not valid.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(valid ? 4 : 0)
               : "memory");
}

template <int NO, bool DIFF>
__global__ void __launch_bounds__(kFirMaxThreads) fir_f32_kernel(const __grid_constant__ FirArgs a) {
  static_assert(16 % NO == 0, "a step of 16 samples is whole rows");
  extern __shared__ __align__(16) float smem[];
  __shared__ float red[kFirMaxThreads / 32];
  const int tid = threadIdx.x, nthreads = blockDim.x, tile = nthreads * NO;
  const int r = blockIdx.y, n0 = blockIdx.x * tile;
  const float* xr = a.x + (int64_t)r * a.x_row;
  float acc[NO];
#pragma unroll
  for (int j = 0; j < NO; ++j) acc[j] = 0.f;
  for (int k0 = 0; k0 < a.ntaps; k0 += kFirTaps) {
    const int nk = min(kFirTaps, a.ntaps - k0), npad = (nk + 15) / 16 * 16, span = tile + npad;
    float* hs = smem;         // [npad], zeros beyond the block's taps
    float* xs = smem + npad;  // sample p at fir_at<NO>(p), p < span
    if (k0 > 0) __syncthreads();
    for (int e = tid; e < npad; e += nthreads) {
      const int k = a.rev ? a.ntaps - 1 - k0 - e : k0 + e;
      cp_async4(hs + e, a.h + (e < nk ? k : 0), e < nk);
    }
    const int q0 = n0 + k0 + a.x_off;
    if constexpr (!DIFF) {
#pragma unroll 4
      for (int e = tid; e < span; e += nthreads) {
        const bool ok = (unsigned)(q0 + e) < (unsigned)a.x_len;
        cp_async4(xs + fir_at<NO>(e), xr + (ok ? q0 + e : 0), ok);
      }
    } else {
      const float* x2 = a.x2 + (int64_t)r * a.x_row;
      constexpr int kBatch = 8;  // loads of both inputs in flight before the first use
      for (int e0 = tid; e0 < span; e0 += kBatch * nthreads) {
        float u[kBatch], v[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
          const int q = q0 + e0 + i * nthreads;
          const bool ok = (unsigned)q < (unsigned)a.x_len;
          u[i] = ok ? xr[q] : 0.f;
          v[i] = ok ? x2[q] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i)
          if (e0 + i * nthreads < span) xs[fir_at<NO>(e0 + i * nthreads)] = u[i] - v[i];
      }
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    auto load16 = [](const float* p, float (&d)[16], bool padded) {
#pragma unroll
      for (int i = 0; i < 16; i += 4) {
        const float4 v = *reinterpret_cast<const float4*>(p + (padded ? fir_at<NO>(i) : i));
        d[i] = v.x, d[i + 1] = v.y, d[i + 2] = v.z, d[i + 3] = v.w;
      }
    };
    // 16 taps from k: sample j + k' of the window is prev's last NO, then next
    const float* xp = xs + fir_at<NO>(NO) * (tid + 1);
    auto step = [&](int k, const float (&prev)[16], float (&next)[16]) {
      float hv[16];
      load16(xp, next, true);
      load16(hs + k, hv, false);
      xp += fir_at<NO>(16);
#pragma unroll
      for (int i = 0; i < 16; ++i)
#pragma unroll
        for (int j = 0; j < NO; ++j)
          acc[j] = fmaf(hv[i], i + j < NO ? prev[16 - NO + i + j] : next[i + j - NO], acc[j]);
    };
    float u[16], v[16];
#pragma unroll
    for (int i = 0; i < NO; i += 4) {
      const float4 q = *reinterpret_cast<const float4*>(xp - fir_at<NO>(NO) + i);
      u[16 - NO + i] = q.x, u[16 - NO + i + 1] = q.y, u[16 - NO + i + 2] = q.z, u[16 - NO + i + 3] = q.w;
    }
    int k = 0;
    for (; k + 32 <= nk; k += 32) {
      step(k, u, v);
      step(k + 16, v, u);
    }
    if (k + 16 <= nk) {
      step(k, u, v);
#pragma unroll
      for (int i = 16 - NO; i < 16; ++i) u[i] = v[i];
      k += 16;
    }
    if (k < nk) {
      load16(xp, v, true);
#pragma unroll
      for (int i = 0; i < 15; ++i) {
        if (k + i < nk) {
          const float h = hs[k + i];
#pragma unroll
          for (int j = 0; j < NO; ++j) acc[j] = fmaf(h, i + j < NO ? u[16 - NO + i + j] : v[i + j - NO], acc[j]);
        }
      }
    }
  }
  const float ds = a.dscale ? *a.dscale : 1.f;
  float* y = a.y + (int64_t)r * a.y_row;
  const int n = n0 + tid * NO;
  float sq = 0.f;
#pragma unroll
  for (int j = 0; j < NO; ++j) {
    acc[j] = a.scale * acc[j];
    if (a.dscale) acc[j] *= ds;
    if (n + j < a.lout) sq = fmaf(acc[j], acc[j], sq);
  }
  if (n + NO <= a.lout && ((uintptr_t)(y + n) & 15) == 0) {
#pragma unroll
    for (int j = 0; j < NO; j += 4)
      *reinterpret_cast<float4*>(y + n + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < NO; ++j)
      if (n + j < a.lout) y[n + j] = acc[j];
  }
  if (a.part) {
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((tid & 31) == 0) red[tid >> 5] = sq;
    __syncthreads();
    if (tid == 0) {
      float t = 0.f;
      for (int i = 0; i < nthreads / 32; ++i) t += red[i];
      a.part[blockIdx.y * gridDim.x + blockIdx.x] = t;
    }
  }
}

// Global average pool over time followed by the linear head; one CTA per item.
// Bound: reading the activation once.  Threads walk the item in order
// (coalesced), weight each channel's values as they sum them and reduce only
// once, at the end (one thread per channel, 512 bytes apart from its
// neighbours, took 36 us for 256 items of 256 x 128, this takes 13 us).
__global__ void __launch_bounds__(kThreads) gap_linear_f32_kernel(const float* __restrict__ h, int64_t hb,
                                                                  int64_t hc, int C, int L,
                                                                  const float* __restrict__ w,
                                                                  const float* __restrict__ bias,
                                                                  float* __restrict__ out) {
  __shared__ float red[kThreads / 32];
  const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float part = 0.f;
  const float* hb0 = h + (int64_t)b * hb;
  if (L % 4 == 0 && hc == L && ((uintptr_t)hb0 & 15) == 0) {
    // the item is one run of C L values: eight 16-byte loads in flight
    const unsigned quads = (unsigned)C * (unsigned)L / 4, per_c = (unsigned)L / 4;
#pragma unroll 8
    for (unsigned i = threadIdx.x; i < quads; i += kThreads) {
      const float4 v = reinterpret_cast<const float4*>(hb0)[i];
      part = fmaf((v.x + v.y) + (v.z + v.w), w[i / per_c], part);
    }
  } else {
    for (int c = warp; c < C; c += kThreads / 32) {
      float sum = 0.f;
      for (int t = lane; t < L; t += 32) sum += hb0[(int64_t)c * hc + t];
      part = fmaf(sum, w[c], part);
    }
  }
  part /= (float)L;
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane == 0) red[warp] = part;
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

// Outputs per thread and threads per CTA.  The time of a launch is that of the
// fullest scheduler (four per SM): its warps times the cycles a warp takes per
// tap, and at least the latency of one warp's own chain.  Measured at 2049
// taps: one warp of 16, 8 or 4 outputs per scheduler 27, 16.6 and 14.5 us;
// 32 rows of 8192 outputs 28.9, 26.9 and 33.0 us; 512 rows of 2048 88, 83 and
// 107 us.
static void plan_fir(int rows, int lout, int* no, int* threads) {
  const double slots = 4.0 * current_sm_count();
  const double outputs = (double)rows * lout;
  static const struct {
    int no;
    double alone, each;
  } kChoice[3] = {{16, 17.0, 14.2}, {8, 9.8, 7.6}, {4, 8.3, 5.2}};
  double best = 0;
  for (const auto& c : kChoice) {
    const double cost = std::max(c.alone, std::ceil(outputs / (32.0 * c.no) / slots) * c.each);
    if (best == 0 || cost < best) {
      best = cost;
      *no = c.no;
    }
  }
  // 128 threads share their taps and the overlap of their samples, unless a row
  // fills 64 much better
  const int64_t t64 = 64 * *no, t128 = 2 * t64;
  *threads = 10 * ((lout + t64 - 1) / t64 * t64) < 9 * ((lout + t128 - 1) / t128 * t128) ? 64 : 128;
}

int fir_f32_parts(int rows, int lout) {
  int no, threads;
  plan_fir(rows, lout, &no, &threads);
  return rows * ((lout + threads * no - 1) / (threads * no));
}

template <int NO>
static void launch_fir_tile(const FirArgs& a, int rows, int threads, cudaStream_t st) {
  const int tile = threads * NO, npad = (std::min(kFirTaps, a.ntaps) + 15) / 16 * 16;
  const size_t smem = (size_t)(npad + fir_at<NO>(tile + npad + NO)) * 4;
  auto kernel = a.x2 ? fir_f32_kernel<NO, true> : fir_f32_kernel<NO, false>;
  set_smem_limit_once(kernel, 64 * 1024);
  kernel<<<dim3((a.lout + tile - 1) / tile, rows), threads, smem, st>>>(a);
  GW_LAUNCH_CHECK();
}

void launch_fir_f32(const FirArgs& a, int rows, cudaStream_t st) {
  GW_CHECK_ARG(a.ntaps <= kFirMaxTaps, "FIR too long for the FP32 kernel");
  int no, threads;
  plan_fir(rows, a.lout, &no, &threads);
  if (no == 16)
    launch_fir_tile<16>(a, rows, threads, st);
  else if (no == 8)
    launch_fir_tile<8>(a, rows, threads, st);
  else
    launch_fir_tile<4>(a, rows, threads, st);
}

void launch_gap_linear_f32(const float* h, int64_t hb, int64_t hc, int B, int C, int L, const float* w,
                           const float* b, float* out, cudaStream_t st) {
  gap_linear_f32_kernel<<<B, kThreads, 0, st>>>(h, hb, hc, C, L, w, b, out);
  GW_LAUNCH_CHECK();
}

}  // namespace gw
