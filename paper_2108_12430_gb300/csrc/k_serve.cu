// Batched kernels of the serving loop: one tick processes one snapshot of
// each of up to max_batch streams, each stream with its own stride and state
// (Methods, "Streaming IaaS": the snapshot state stays on the GPU and each
// request brings only the new samples).
//
// Sample timing (per item; the resampler and the alignment are readings):
//   cleaned   c[tau] emitted for tau in [head - delta, head + S - delta);
//   decimated d[m] = sum_j f[j] c[2m + j - (Kf-1)/2]       (c[tau < 0] = 0);
//   whitened  w[n] = sum_j h[j] d[n + j - (Kh-1)/2]        (d[m < 0] = 0);
//   BBHnet input: w[n1 - Lb, n1) of every detector          (w[n < 0] = 0).
#include "gw_serve.h"

namespace gw {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int64_t floordiv64(int64_t a, int64_t b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }
// Ring residue of an absolute sample index (int64, may be negative): one
// 64-bit reduction per thread; the element loops then step through the ring
// in 32 bits with wrap(), which needs 0 <= b < m and 0 <= d < m.
__device__ __forceinline__ uint32_t ring_mod(int64_t a, int64_t m) {
  const int64_t r = a % m;
  return (uint32_t)(r < 0 ? r + m : r);
}
__device__ __forceinline__ uint32_t wrap(uint32_t b, uint32_t d, uint32_t m) {
  const uint32_t q = b + d;
  return q >= m ? q - m : q;
}

// Witness ring update (standardised on write) and strain ring update.
// Blocked BF16 ring: channel group g, ring position q (0 <= q < 2R) is the
// 16-byte row at g * 2R * 8 + (q % P) * (2R / P) * 8 + (q / P) * 8 elements;
// both copies q and q + R are written, so every window is contiguous.
__global__ void serve_push_kernel(const ServeItem* __restrict__ items, ServeGeom g, const float* __restrict__ mean,
                                  const float* __restrict__ istd) {
  // the network kernel after this one may start now: it reads only older
  // samples of the rings until it waits for this kernel to finish
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const ServeItem it = items[blockIdx.y];
  if (!it.active) return;
  const int S = it.S;
  const float* src = it.in;
  const uint32_t R = (uint32_t)g.R, h0 = ring_mod(it.head, g.R);
  if (g.bf16) {
    __nv_bfloat16* ring = reinterpret_cast<__nv_bfloat16*>(it.wring);
    const uint32_t P = (uint32_t)g.P, plane_rows = 2u * R / P;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < g.G * S; e += gridDim.x * blockDim.x) {
      const int grp = e / S, t = e - grp * S;
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = grp * 8 + j;
        v[j] = c < g.C ? src[c * S + t] : 0.f;  // all loads in flight before the first use
      }
      __align__(16) __nv_bfloat16 v8[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = grp * 8 + j;
        v8[j] = __float2bfloat16_rn(c < g.C ? (v[j] - mean[c]) * istd[c] : 0.f);
      }
      const uint32_t q = wrap(h0, (uint32_t)t, R), q2 = q + R;
      uint4* base = reinterpret_cast<uint4*>(ring + (int64_t)grp * 2 * R * 8);
      const uint4 val = *reinterpret_cast<const uint4*>(v8);
      base[(q % P) * plane_rows + q / P] = val;
      base[(q2 % P) * plane_rows + q2 / P] = val;
    }
  } else {
    float* ring = reinterpret_cast<float*>(it.wring);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < g.C * S; e += gridDim.x * blockDim.x) {
      const int c = e / S, t = e - c * S;
      const float v = (src[c * S + t] - mean[c]) * istd[c];
      const uint32_t q = wrap(h0, (uint32_t)t, R);
      ring[(int64_t)c * 2 * R + q] = v;
      ring[(int64_t)c * 2 * R + q + R] = v;
    }
  }
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < S; t += gridDim.x * blockDim.x)
    it.strain[wrap(h0, (uint32_t)t, R)] = src[g.C * S + t];
}

// Subtraction and aggregation of one new window per item (the window ends at
// head + S).  AVERAGE: sums per time in window order, divided by the number
// of windows so far covering the time; LATEST: the newest window alone.
// Bound: the prediction and the aggregation sums, once each (64 windows of
// 32768: 25 MB).  A thread takes 4 consecutive samples (W, every stride and the
// rings' lengths are multiples of 8, so that they are 16 aligned bytes of the
// prediction and of the sums) and only the emitted ones take the 64-bit arithmetic
// (64 items: 16.0 us one sample at a time, 10.6 us so).
__global__ void serve_sub_ola_kernel(const ServeItem* __restrict__ items, ServeGeom g, const float* __restrict__ pred) {
  const ServeItem it = items[blockIdx.y];
  if (!it.active) return;
  const int S = it.S, W = g.W;
  const int64_t head = it.head;
  const float* pr = pred + (int64_t)blockIdx.y * W;
  // window sample e is time tau = head + S - W + e; it is emitted as cleaned
  // sample o = e - (W - S - delta) when 0 <= o < S
  const uint32_t R = (uint32_t)g.R, qb = ring_mod(head + S - W, g.R);
  const int o_shift = W - S - g.delta;
  for (int e = 4 * (blockIdx.x * blockDim.x + threadIdx.x); e < W; e += 4 * gridDim.x * blockDim.x) {
    const bool emits = e + 3 >= o_shift && e < o_shift + S;
    if (g.mode == GW_AGG_LATEST && !emits) continue;
    const float4 p4 = *reinterpret_cast<const float4*>(pr + e);
    float v[4] = {p4.x, p4.y, p4.z, p4.w};
    if (g.mode != GW_AGG_LATEST) {
      // the sums of times before head; a newer time's slot is an old one's
      float4* a4 = reinterpret_cast<float4*>(it.acc + wrap(qb, (uint32_t)e, R));
      const float4 q = *a4;
      const float old[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = (e + i < W - S ? old[i] : 0.f) + v[i];
      *a4 = make_float4(v[0], v[1], v[2], v[3]);
      if (!emits) continue;
    }
    const int64_t k = head / S;
    const uint32_t cb = ring_mod(head - g.delta, g.Rc);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int o = e + i - o_shift;
      if (o < 0 || o >= S) continue;
      const int64_t tau = head + S - W + e + i;
      float value = v[i];
      if (g.mode != GW_AGG_LATEST) {
        const int64_t first = tau >= 0 ? floordiv64(tau, S) : 0;
        value /= (float)(k - first + 1);
      }
      if (g.post) {
        // the post-processing FIR reads the aggregated prediction from its ring
        if (tau >= 0) it.pring[ring_mod(tau, g.Rp)] = value;
        continue;
      }
      const float c = (tau >= 0 ? it.strain[wrap(qb, (uint32_t)(e + i), R)] : 0.f) - value;
      it.out[o] = c;
      if (tau >= 0) it.clean[wrap(cb, (uint32_t)o, (uint32_t)g.Rc)] = c;
    }
  }
}

// Post-processing: cleaned[t] = strain[t] - sum_k h[k] p[t + k - c] for the
// times t = head - delta - c + o, o < S (the prediction at negative times is
// zero: there is no data before the stream start).  One CTA per kServePost
// outputs of an item stages the taps and the prediction segment it reads.
constexpr int kServePost = 256;
__global__ void serve_post_kernel(const ServeItem* __restrict__ items, ServeGeom g, const float* __restrict__ h,
                                  int K) {
  const ServeItem it = items[blockIdx.y];
  if (!it.active) return;
  const int o0 = blockIdx.x * kServePost;
  if (o0 >= it.S) return;
  extern __shared__ float sh[];
  float* hs = sh;      // [K]
  float* ps = sh + K;  // p[t(o0) - c + i], i < kServePost + K - 1
  const int c = g.post_c;
  const int64_t t0 = it.head - g.delta - c + o0;
  for (int k = threadIdx.x; k < K; k += blockDim.x) hs[k] = h[k];
  for (int i = threadIdx.x; i < kServePost + K - 1; i += blockDim.x) {
    const int64_t u = t0 - c + i;
    ps[i] = u >= 0 ? it.pring[ring_mod(u, g.Rp)] : 0.f;
  }
  __syncthreads();
  const int o = o0 + threadIdx.x;
  if (threadIdx.x >= kServePost || o >= it.S) return;
  float q = 0.f;
  for (int k = 0; k < K; ++k) q = fmaf(hs[k], ps[threadIdx.x + k], q);
  const int64_t t = t0 + threadIdx.x;
  const float v = (t >= 0 ? it.strain[ring_mod(t, g.R)] : 0.f) - q;
  it.out[o] = v;
  if (t >= 0) it.clean[ring_mod(t, g.Rc)] = v;
}

// New decimated samples d[m], m in [m0, m1): one per thread, one FMA chain over
// the taps in order.  A block of taps and the samples that the CTA's outputs
// take them with are staged in shared memory: the chain's loads were what it
// waited for (127 taps, 64 items: 8.5 us from the rings, 6.2 us so).
constexpr int kDecOut = 128, kDecTaps = 512;
__global__ void __launch_bounds__(kDecOut) serve_decimate_kernel(const ServeItem* __restrict__ items, ServeGeom g,
                                                                 const float* __restrict__ f, int K) {
  __shared__ float fs[kDecTaps], xs[2 * kDecOut + kDecTaps];
  const ServeItem it = items[blockIdx.y];
  if (!it.active) return;
  const int c = (K - 1) / 2;
  const uint32_t Rc = (uint32_t)g.Rc;
  for (int64_t mb = it.m0 + blockIdx.x * kDecOut; mb < it.m1; mb += gridDim.x * kDecOut) {
    const int n = (int)min((int64_t)kDecOut, it.m1 - mb);
    float a = 0.f;
    for (int j0 = 0; j0 < K; j0 += kDecTaps) {
      const int nk = min(kDecTaps, K - j0), nx = 2 * (n - 1) + nk;
      // the samples before the stream start are zero
      const int64_t x0 = 2 * mb - c + j0;
      const uint32_t q0 = ring_mod(x0, g.Rc);
      for (int i = threadIdx.x; i < nk; i += kDecOut) fs[i] = f[j0 + i];
      for (int i = threadIdx.x; i < nx; i += kDecOut)
        xs[i] = x0 + i >= 0 ? it.clean[(q0 + (uint32_t)i) % Rc] : 0.f;
      __syncthreads();
      if ((int)threadIdx.x < n)
        for (int j = 0; j < nk; ++j) a = fmaf(fs[j], xs[2 * threadIdx.x + j], a);
      __syncthreads();
    }
    if ((int)threadIdx.x < n) it.dec[ring_mod(mb + threadIdx.x, g.Rd)] = a;
  }
}

// New whitened samples w[n], n in [n0, n1): an output's taps go over a warp's
// lanes (lane j mod 32, each lane's in order, then a tree over the lanes).  The
// taps and the decimated segment are staged in shared memory.  Bound: the
// shared-memory loads.  A warp computes kWhitenQ outputs 32 apart, whose samples
// at one step are the next output's at the step before, in the same lane: a
// register window takes one new sample and one tap per kWhitenQ FMAs, and an
// item's outputs go over kWhitenParts CTAs (2049 taps, 64 items of up to 256
// outputs: 32 us with one output per warp and one CTA per item, 13.7 us so).
constexpr int kWhitenQ = 8, kWhitenParts = 4;
__global__ void __launch_bounds__(kThreads) serve_whiten_kernel(const ServeItem* __restrict__ items, ServeGeom g,
                                                                const float* __restrict__ h, int K) {
  extern __shared__ float sh[];
  constexpr int Q = kWhitenQ, kWarps = kThreads / 32;
  static_assert(kWhitenParts * kWarps == 32, "a block of 32 Q outputs: one start per warp");
  const ServeItem it = items[blockIdx.y];
  if (!it.active || it.n1 <= it.n0) return;
  const int c = (K - 1) / 2;
  const int nn = (int)(it.n1 - it.n0), first = blockIdx.x * kWarps;
  if (first >= nn) return;
  float* hs = sh;
  float* ds = sh + K;  // d[n0 - c + i], i < nn + K - 1 (< Rd), then zeros that only discarded outputs read
  for (int j = threadIdx.x; j < K; j += blockDim.x) hs[j] = h[j];
  const uint32_t Rd = (uint32_t)g.Rd, db = ring_mod(it.n0 - c, g.Rd);
  for (int i = threadIdx.x; i < nn + K + 32 * Q; i += blockDim.x)
    ds[i] = i < nn + K - 1 && it.n0 - c + i >= 0 ? it.dec[wrap(db, (uint32_t)i, Rd)] : 0.f;
  __syncthreads();
  const uint32_t Rw = (uint32_t)g.Rw, wb = ring_mod(it.n0, g.Rw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = first + warp; i < nn; i += 32 * Q) {
    const float* x = ds + i + lane;
    float a[Q], d[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) a[q] = 0.f, d[q] = x[32 * q];
    int n = 0;
    for (; 32 * (n + Q) <= K; n += Q) {
#pragma unroll
      for (int m = 0; m < Q; ++m) {
        const float hv = hs[lane + 32 * (n + m)];
#pragma unroll
        for (int q = 0; q < Q; ++q) a[q] = fmaf(hv, d[(q + m) % Q], a[q]);
        d[m] = x[32 * (n + m + Q)];
      }
    }
    for (int j = lane + 32 * n; j < K; j += 32) {
      const float hv = hs[j];
#pragma unroll
      for (int q = 0; q < Q; ++q) a[q] = fmaf(hv, ds[i + j + 32 * q], a[q]);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a[q] += __shfl_xor_sync(0xffffffffu, a[q], o);
      if (lane == 0 && i + 32 * q < nn) it.white[wrap(wb, (uint32_t)(i + 32 * q), Rw)] = a[q];
    }
  }
}

// BBHnet input x[r][d][t] = w_d[n1 - Lb + t] of request r (zero for n < 0
// and for padding requests).
__global__ void serve_gather_kernel(const ServeItem* __restrict__ items, int Bb, int n_det, int Lb, ServeGeom g,
                                    float* __restrict__ x) {
  const int r = blockIdx.y;
  const ServeItem it0 = items[r];
  float* dst = x + (int64_t)r * n_det * Lb;
  const uint32_t Rw = (uint32_t)g.Rw, wb = ring_mod(it0.n1 - Lb, g.Rw);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n_det * Lb; e += gridDim.x * blockDim.x) {
    const int d = e / Lb, t = e - d * Lb;
    float v = 0.f;
    if (it0.active && it0.n1 - Lb + t >= 0) v = items[d * Bb + r].white[wrap(wb, (uint32_t)t, Rw)];
    dst[e] = v;
  }
}

// Scores to the requests' host slots (NaN without a BBHnet), and the tick's
// device status: nonzero when a tensor-core kernel gave up a bounded wait.
__global__ void serve_scores_kernel(const ServeItem* __restrict__ items, int Bb, const float* __restrict__ logits,
                                    const int* e0, const int* e1, int* status) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r == 0) *status = ((e0 && *e0) || (e1 && *e1)) ? 1 : 0;
  if (r >= Bb) return;
  const ServeItem& it = items[r];
  if (it.active && it.score) *it.score = logits ? logits[r] : __int_as_float(0x7fc00000);
}

int grid_x(int64_t work) {
  const int64_t b = (work + kThreads - 1) / kThreads;
  return (int)(b < 1 ? 1 : (b > 64 ? 64 : b));
}

}  // namespace

void launch_serve_push(const ServeItem* items, int n, const ServeGeom& g, int S_max, const float* mean,
                       const float* istd, cudaStream_t st) {
  const int64_t work = (int64_t)(g.bf16 ? g.G : g.C) * S_max;
  serve_push_kernel<<<dim3(grid_x(work), n), kThreads, 0, st>>>(items, g, mean, istd);
  GW_LAUNCH_CHECK();
}

void launch_serve_sub_ola(const ServeItem* items, int n, const ServeGeom& g, const float* pred, cudaStream_t st) {
  GW_CHECK_ARG(g.W % 8 == 0 && g.R % 8 == 0, "window and ring lengths are multiples of 8");
  serve_sub_ola_kernel<<<dim3(grid_x(g.W / 4), n), kThreads, 0, st>>>(items, g, pred);
  GW_LAUNCH_CHECK();
}

void launch_serve_post(const ServeItem* items, int n, const ServeGeom& g, const float* h, int K, int S_max,
                       cudaStream_t st) {
  const size_t smem = (size_t)(2 * K + kServePost) * sizeof(float);
  GW_CHECK_ARG(smem <= 200 * 1024, "post-processing FIR too long for the serving kernel");
  set_smem_limit_once(serve_post_kernel, 200 * 1024);
  serve_post_kernel<<<dim3((S_max + kServePost - 1) / kServePost, n), kServePost, smem, st>>>(items, g, h, K);
  GW_LAUNCH_CHECK();
}

void launch_serve_decimate(const ServeItem* items, int n, const ServeGeom& g, const float* taps, int K, int max_new,
                           cudaStream_t st) {
  serve_decimate_kernel<<<dim3((max_new + kDecOut - 1) / kDecOut, n), kDecOut, 0, st>>>(items, g, taps, K);
  GW_LAUNCH_CHECK();
}

size_t serve_whiten_smem(int K, int max_new) { return (size_t)(2 * K + max_new) * sizeof(float); }

void launch_serve_whiten(const ServeItem* items, int n, const ServeGeom& g, const float* taps, int K, int max_new,
                         cudaStream_t st) {
  GW_CHECK_ARG(serve_whiten_smem(K, max_new) <= 200 * 1024, "whitening FIR too long for the streaming kernel");
  const size_t smem = serve_whiten_smem(K, max_new) + 32 * kWhitenQ * sizeof(float);
  set_smem_limit_once(serve_whiten_kernel, 202 * 1024);
  serve_whiten_kernel<<<dim3(kWhitenParts, n), kThreads, smem, st>>>(items, g, taps, K);
  GW_LAUNCH_CHECK();
}

void launch_serve_gather(const ServeItem* items, int Bb, int n_det, int Lb, const ServeGeom& g, float* x,
                         cudaStream_t st) {
  serve_gather_kernel<<<dim3(grid_x((int64_t)n_det * Lb), Bb), kThreads, 0, st>>>(items, Bb, n_det, Lb, g, x);
  GW_LAUNCH_CHECK();
}

void launch_serve_scores(const ServeItem* items, int Bb, const float* logits, const int* e0, const int* e1,
                         int* status, cudaStream_t st) {
  serve_scores_kernel<<<(Bb + 127) / 128, 128, 0, st>>>(items, Bb, logits, e0, e1, status);
  GW_LAUNCH_CHECK();
}

}  // namespace gw
