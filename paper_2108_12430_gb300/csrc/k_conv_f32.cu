// FP32 conv / transposed conv of the plain-FP32 path (both networks' layer
// shapes, forward and data gradient).
//
// Conv:  y[o,u] = b[o] + sum_{i,k} w[o,i,k] x[i, s u + k - p]
// ConvT: y[o,u] = b[o] + sum_{i,k : s | (u + p - k)} w[o,i,k] x[i, (u + p - k) / s]
// with weights laid out [C_in][K][C_out rounded up to 8] for both.
//
// Bound: the FP32 FMA pipe (TF32 could not meet a 1e-5 relative error), 80.5
// TFLOP/s at 2070 MHz.  A register-only loop reaches 76 packed and 75 scalar on
// the whole chip, but a packed fma.rn.f32x2 does two FMAs per issue slot, so that the
// shared-memory loads, operand moves and staging issue beside the FMAs
// instead of between them.  The pairs are two adjacent output channels: a
// weight pair is one aligned 64-bit value of shared memory, and an input value
// is duplicated once per tap for the CPT / 2 pairs it feeds.
//
// Order of the sums: each output is one FP32 FMA chain over (ci, k), input
// channels in order and taps in order within each, then the bias, whatever the
// tile (a packed and a scalar chain give the same bits).  An item's bits
// therefore do not depend on how many items share its launch: a server's batch
// follows from arrival times, and a stream's results must not.  So no launch
// splits the input channels over threads; one with few outputs gives each thread
// fewer of them instead.
//
// Thread: CPT output channels x PPT positions.  Input rows sit in shared
// memory such that a warp's 16-byte loads walk consecutive addresses: positions
// go in blocks of 4 per thread (a thread's second block is a whole row of
// blocks away), and a stride-2 conv's input row is split into its even and odd
// samples.
//
// Staging: input channels go through two shared-memory stages of CI channels
// with their weights, filled by cp.async (zero-filled outside the input: the
// layer's padding) one chunk ahead of the FMAs.  The small tiles serve launches
// that would leave the chip idle (plan_conv_f32).  A dependent launch stages its
// first weights while the previous layer ends.
//
// Measured (GB300, against scalar FMAs on rows staged through registers, one
// tile shape): 64 windows of 21 x 32768 in one push 1422 -> 794 us (22 -> 40
// TFLOP/s; the 32 -> 64 channel layer 304 -> 156 us), whitening and BBHnet on
// 256 segments 3648 -> 1971 us (its 256 -> 256 layer 947 -> 546 us, 55 TFLOP/s),
// one window of 21 x 4096 184 -> 36 us.
#include <algorithm>

#include "gw_internal.h"
#include "tc_ptx.h"

namespace gw {

namespace {

constexpr int kMaxThreads = 256;

struct ConvTile {
  int CB, np, CI;       // channels, position groups per CTA; input channels per stage
  int lgq;              // log2(CB / 4), or -1 for CB = 1
  int rowp, odd;        // floats per staged input row; offset of its odd samples (stride 2)
  int span;             // samples staged per input row
  int stage_floats;
  int cop;              // weight row length (C_out rounded up to 8)
  int flip, pad;        // transposed conv of stride 1: reversed taps, padding K - 1 - p
  int vec;              // outputs, residual and gy can be accessed 16 bytes at a time
};

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 dup2(float v) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
  return d;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
// `bytes` (0 .. 16) are copied, the rest of the 16 is zero-filled.
__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, int bytes = 16) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ float apply_act(float v, int act) {
  if (act == ACT_TANH) return tanhf(v);
  if (act == ACT_RELU) return fmaxf(v, 0.f);
  return v;
}
__device__ __forceinline__ float act_deriv(float y, int act) {
  return act == ACT_TANH ? 1.f - y * y : (act == ACT_RELU ? (y > 0.f ? 1.f : 0.f) : 1.f);
}

// How a thread's positions lie: NB blocks of BW consecutive ones (a block of
// the transposed stride-2 conv is all of them, and its inputs half as many).
template <int K, int S, bool TR2, int PPT>
struct Geo {
  static constexpr int BW = TR2 ? PPT : (PPT < 4 ? PPT : 4), NB = PPT / BW;
  static constexpr bool SPLIT = S == 2 && !TR2 && K > 1;  // even / odd input rows
  // A stride-1 row is staged from one sample before the first one read, so
  // that (with a padding of 3 mod 4, as every such layer has) it starts 16-byte
  // aligned in memory whenever the tensor's rows do.
  static constexpr int SHIFT = S == 1 && !TR2 && K > 1 ? 1 : 0;
  // inputs a block reads: from one row, or from the even and the odd row
  static constexpr int NX = TR2 ? PPT / 2 + 3 : (SPLIT ? BW + (K - 1) / 2 : BW + K - 1 + SHIFT);
  static constexpr int NXO = SPLIT ? BW + (K - 2) / 2 : 0;
  static constexpr int XSTEP = TR2 ? PPT / 2 : BW;  // input distance between neighbouring threads
};

// N consecutive floats from an address aligned to A floats (A = 2 or 4; reads
// up to the next multiple of A).
template <int N, int A>
__device__ __forceinline__ void load_row(const float* p, float (&v)[(N + 3) / 4 * 4]) {
  if constexpr (A == 4) {
#pragma unroll
    for (int q = 0; q < (N + 3) / 4; ++q) {
      const float4 t = reinterpret_cast<const float4*>(p)[q];
      v[4 * q] = t.x, v[4 * q + 1] = t.y, v[4 * q + 2] = t.z, v[4 * q + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < (N + 1) / 2; ++q) {
      const float2 t = reinterpret_cast<const float2*>(p)[q];
      v[2 * q] = t.x, v[2 * q + 1] = t.y;
    }
  }
}

template <int K, int S, bool TR2, int CPT, int PPT>
__global__ void __launch_bounds__(kMaxThreads, 2)
    conv_f32_kernel(const __grid_constant__ ConvF32Args a, const __grid_constant__ ConvTile t) {
  using G = Geo<K, S, TR2, PPT>;
  constexpr int CP = (CPT + 1) / 2;  // channel pairs (CPT = 1: scalar)
  constexpr int BW = G::BW, NB = G::NB;
  extern __shared__ __align__(16) float smem[];
  const LayerSpec& s = a.s;
  const int tid = threadIdx.x, nthreads = blockDim.x, warp = tid >> 5, lane = tid & 31, nwarps = nthreads >> 5;
  const int cg = tid / t.np, pt = tid - cg * t.np;
  const int TL = t.np * PPT;
  const int t0 = blockIdx.x * TL, co0 = blockIdx.y * t.CB, b = blockIdx.z;
  constexpr int XS = (K == 1) ? S : 1;  // input samples per staged sample
  const int lo = TR2 ? (t0 + t.pad - (K - 1) + 1) / 2 : t0 * S - t.pad - G::SHIFT;

  auto stage_w = [&](int st, int c0) {
    float* ws = smem + st * t.stage_floats + t.CI * t.rowp;
    const int rows = min(t.CI, s.cin - c0) * K;
    const float* src = a.w + (int64_t)c0 * K * t.cop + co0;
    if (t.lgq >= 0) {
      const int lgq = t.lgq, total = rows << lgq;
      for (int e = tid; e < total; e += nthreads) {
        const int r = e >> lgq, q = (e & ((1 << lgq) - 1)) * 4;
        const int sr = t.flip ? r + K - 1 - 2 * (r % K) : r;
        cp_async16(ptx::smem_u32(ws + r * t.CB + q), src + (int64_t)sr * t.cop + q);
      }
    } else {
      for (int r = tid; r < rows; r += nthreads)
        cp_async4(ptx::smem_u32(ws + r), src + (int64_t)(t.flip ? r + K - 1 - 2 * (r % K) : r) * t.cop, true);
    }
  };
  const float* xb = nullptr;
  auto stage_x = [&](int st, int c0) {
    float* xs = smem + st * t.stage_floats;
    const int n = min(t.CI, s.cin - c0);
    for (int ci = warp; ci < n; ci += nwarps) {
      const float* row = xb + (int64_t)(c0 + ci) * a.xc;
      const uint32_t dst = ptx::smem_u32(xs + ci * t.rowp);
      if constexpr (G::SHIFT) {
        if (((uintptr_t)(row + lo) & 15) == 0) {
          for (int j = 4 * lane; j < t.span; j += 128) {
            const int left = lo + j < 0 ? 0 : a.lin - (lo + j);  // lo is a multiple of 4: all or nothing below 0
            cp_async16(dst + 4 * j, row + (left > 0 ? lo + j : 0), left >= 4 ? 16 : (left > 0 ? 4 * left : 0));
          }
          continue;
        }
      }
#pragma unroll 4
      for (int j = lane; j < t.span; j += 32) {
        const int x = lo + j * XS;
        const bool ok = (unsigned)x < (unsigned)a.lin;
        const int d = G::SPLIT ? ((j & 1) ? t.odd : 0) + (j >> 1) : j;
        cp_async4(dst + 4 * d, row + (ok ? x : 0), ok);
      }
    }
  };
  // input standardisation of a landed stage, on the rows the warp copied
  auto standardise = [&](int st, int c0) {
    __syncwarp();
    float* xs = smem + st * t.stage_floats;
    const int n = min(t.CI, s.cin - c0);
    for (int ci = warp; ci < n; ci += nwarps) {
      const float mean = a.in_mean[c0 + ci], istd = a.in_istd[c0 + ci];
      for (int j = lane; j < t.span; j += 32) {
        const int d = ci * t.rowp + (G::SPLIT ? ((j & 1) ? t.odd : 0) + (j >> 1) : j);
        if ((unsigned)(lo + j * XS) < (unsigned)a.lin) xs[d] = (xs[d] - mean) * istd;
      }
    }
  };

  // the weights do not depend on the previous kernel in the stream
  stage_w(0, 0);
  ptx::griddep_wait();
  // A launch of small tiles leaves SMs empty; were its dependent let in here, the
  // next layer's CTAs would crowd on those (BBHnet on eight segments 223 us, 157 us
  // with the trigger after the FMAs).  A full launch's dependent finds no room
  // before its end anyway, and the trigger costs nothing here.
  if (CPT == 8) ptx::griddep_launch_dependents();
  xb = a.item_ptr ? a.item_ptr[b] : a.x + (int64_t)b * a.xb;
  stage_x(0, 0);
  cp_async_commit();

  f32x2 acc[CP][PPT];
  float acc1[CPT == 1 ? PPT : 1];
#pragma unroll
  for (int c = 0; c < CP; ++c)
#pragma unroll
    for (int j = 0; j < PPT; ++j) acc[c][j] = 0ull;
#pragma unroll
  for (int j = 0; j < (CPT == 1 ? PPT : 1); ++j) acc1[j] = 0.f;

  const int n_chunks = (s.cin + t.CI - 1) / t.CI;
  for (int ch = 0; ch < n_chunks; ++ch) {
    const int st = ch & 1, c0 = ch * t.CI;
    cp_async_wait<0>();
    if (a.in_mean) standardise(st, c0);
    __syncthreads();  // this stage has landed, and every thread is done with the other
    if (ch + 1 < n_chunks) {
      stage_w(st ^ 1, c0 + t.CI);
      stage_x(st ^ 1, c0 + t.CI);
      cp_async_commit();
    }
    const float* xs = smem + st * t.stage_floats;
    const float* ws = xs + t.CI * t.rowp + cg * CPT;
    const int n = min(t.CI, s.cin - c0);
    auto channel = [&](int ci) {
      const float* xr = xs + ci * t.rowp + pt * G::XSTEP;
      const float* wr = ws + ci * K * t.CB;
      constexpr int A = G::XSTEP % 4 == 0 ? 4 : 2;
      float xv[NB][(G::NX + 3) / 4 * 4];
      float xo[NB][G::SPLIT ? (G::NXO + 3) / 4 * 4 : 4];
#pragma unroll
      for (int h = 0; h < NB; ++h) {
        load_row<G::NX, A>(xr + h * BW * t.np, xv[h]);
        if constexpr (G::SPLIT) load_row<G::NXO, A>(xr + t.odd + h * BW * t.np, xo[h]);
      }
#pragma unroll
      for (int k = 0; k < K; ++k) {
        f32x2 wv[CP];
        float w1 = 0.f;
        if constexpr (CPT == 1) {
          w1 = wr[k];
        } else if constexpr (CPT == 2) {
          wv[0] = *reinterpret_cast<const f32x2*>(wr + k * t.CB);
        } else {
#pragma unroll
          for (int q = 0; q < CP / 2; ++q) {
            const ulonglong2 v = reinterpret_cast<const ulonglong2*>(wr + k * t.CB)[q];
            wv[2 * q] = v.x;
            wv[2 * q + 1] = v.y;
          }
        }
#pragma unroll
        for (int h = 0; h < NB; ++h)
#pragma unroll
          for (int jj = 0; jj < BW; ++jj) {
            const int j = h * BW + jj;
            float x;
            if constexpr (TR2) {
              // output u = t0 + PPT pt + j takes tap k when j - k + K is even (t0
              // even, K - p even), and reads x[lo + PPT / 2 pt + (j - k + K) / 2 - 1]
              if ((j - k + K) & 1) continue;
              x = xv[h][(j - k + K) / 2 - 1];
            } else if constexpr (G::SPLIT) {
              x = (k & 1) ? xo[h][jj + (k >> 1)] : xv[h][jj + (k >> 1)];
            } else {
              x = xv[h][jj + k + G::SHIFT];
            }
            if constexpr (CPT == 1) {
              acc1[j] = fmaf(w1, x, acc1[j]);
            } else {
              const f32x2 xx = dup2(x);
#pragma unroll
              for (int c = 0; c < CP; ++c) acc[c][j] = fma2(wv[c], xx, acc[c][j]);
            }
          }
      }
    };
    if constexpr (CPT == 8) {
      for (int ci = 0; ci < n; ++ci) channel(ci);
    } else {
      // the next channels' loads run under this one's chain of FMAs (two windows
      // of 21 x 32768: 69.8 us rolled, 60.1 us so)
#pragma unroll 4
      for (int ci = 0; ci < n; ++ci) channel(ci);
    }
  }

  if (CPT < 8) ptx::griddep_launch_dependents();
  float v[CPT][PPT];
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    if constexpr (CPT == 1) {
      v[0][j] = acc1[j];
    } else {
#pragma unroll
      for (int c = 0; c < CP; ++c) unpack2(acc[c][j], v[2 * c][j], v[2 * c + 1][j]);
    }
  }
#pragma unroll
  for (int c = 0; c < CPT; ++c) {
    const int o = co0 + cg * CPT + c;
    if (o >= s.cout) continue;
    const float bias = a.bias[o];
    float* y = a.y + (int64_t)b * a.yb + (int64_t)o * a.yc;
    const float* res = a.res ? a.res + (int64_t)b * a.rb + (int64_t)o * a.rc : nullptr;
    const float* gy = a.gy ? a.gy + (int64_t)b * a.gyb + (int64_t)o * a.gyc : nullptr;
#pragma unroll
    for (int h = 0; h < PPT / 4; ++h) {
      const int j0 = 4 * h, u0 = t0 + (TR2 ? PPT * pt + j0 : h * BW * t.np + BW * pt);
      if (u0 >= a.lout) continue;
      float r[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) r[j] = v[c][j0 + j] + bias;
      if (t.vec) {
        if (res) {
          const float4 q = *reinterpret_cast<const float4*>(res + u0);
          r[0] += q.x, r[1] += q.y, r[2] += q.z, r[3] += q.w;
        }
        if (gy) {
          const float4 q = *reinterpret_cast<const float4*>(gy + u0);
          r[0] *= act_deriv(q.x, a.gact), r[1] *= act_deriv(q.y, a.gact);
          r[2] *= act_deriv(q.z, a.gact), r[3] *= act_deriv(q.w, a.gact);
        }
        *reinterpret_cast<float4*>(y + u0) = make_float4(apply_act(r[0], s.act), apply_act(r[1], s.act),
                                                         apply_act(r[2], s.act), apply_act(r[3], s.act));
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (u0 + j >= a.lout) continue;
          if (res) r[j] += res[u0 + j];
          if (gy) r[j] *= act_deriv(gy[u0 + j], a.gact);
          y[u0 + j] = apply_act(r[j], s.act);
        }
      }
    }
  }
}

constexpr int kMaxSmem = 110 * 1024;  // two CTAs per SM

template <int K, int S, bool TR2, int CPT, int PPT>
ConvTile make_tile(const ConvF32Args& a, int CB, int np) {
  using G = Geo<K, S, TR2, PPT>;
  const LayerSpec& s = a.s;
  ConvTile t{};
  t.CB = CB;
  t.np = np;
  t.cop = conv_f32_cop(s.cout);
  t.flip = s.transposed && s.stride == 1;
  t.pad = t.flip ? K - 1 - s.pad_l : s.pad_l;
  const int TL = np * PPT;
  t.lgq = -1;
  if (CB >= 4)
    for (t.lgq = 0; (4 << t.lgq) < CB; ++t.lgq) {
    }
  // the samples that the tile's outputs read, and the (wider) extent of the
  // last thread's vector loads
  if (TR2) {
    t.span = TL / 2 + 3;
    t.rowp = ((np - 1) * G::XSTEP + (G::NX + 3) / 4 * 4 + 3) / 4 * 4;
  } else if (G::SPLIT) {
    t.span = (TL - 1) * S + K;
    t.odd = ((np * G::NB - 1) * G::BW + (G::NX + 3) / 4 * 4 + 3) / 4 * 4;
    t.rowp = 2 * t.odd;
  } else {
    t.span = TL + K - 1 + G::SHIFT;
    t.rowp = ((np * G::NB - 1) * G::BW + (G::NX + 3) / 4 * 4 + 3) / 4 * 4;
  }
  const int per_ci = t.rowp + K * CB;
  // Channels per stage: a stage's copies are in flight for the FMAs of one stage.
  // Eight channels of an 8-channel tile cover that, a small tile's are over before
  // the copies land (at 8 / 16 / 32 channels: one window of 21 x 4096 40.8 / 38.5 /
  // 37.2 us, BBHnet on one segment 144 / 130 / 124 us; at eight segments, CTAs of 256
  // threads, 32 channels take 212 us for 157 at 16).
  int CI = std::min(s.cin, CPT == 8 ? 8 : (CPT == 2 && np * (CB / CPT) <= 128 ? 32 : 16));
  while (CI > 1 && (size_t)2 * CI * per_ci * 4 > kMaxSmem) --CI;
  const int chunks = (s.cin + CI - 1) / CI;
  t.CI = (s.cin + chunks - 1) / chunks;
  t.stage_floats = (t.CI * per_ci + 3) / 4 * 4;
  auto ok16 = [](const void* p, int64_t b, int64_t c) {
    return p == nullptr || (((uintptr_t)p & 15) == 0 && b % 4 == 0 && c % 4 == 0);
  };
  t.vec = a.lout % 4 == 0 && ok16(a.y, a.yb, a.yc) && ok16(a.res, a.rb, a.rc) && ok16(a.gy, a.gyb, a.gyc);
  return t;
}

template <int K, int S, bool TR2, int CPT, int PPT>
void launch_tile(const ConvF32Args& a, int CB, int np, cudaStream_t st) {
  const ConvTile t = make_tile<K, S, TR2, CPT, PPT>(a, CB, np);
  const int threads = np * (CB / CPT);
  GW_CHECK_ARG(threads >= 32 && threads % 32 == 0 && threads <= kMaxThreads, "FP32 conv tile needs whole warps");
  GW_CHECK_ARG(t.cop % CB == 0, "FP32 conv tile beyond the padded weight row");
  const size_t smem = (size_t)(t.CI < a.s.cin ? 2 : 1) * t.stage_floats * 4;
  auto kernel = conv_f32_kernel<K, S, TR2, CPT, PPT>;
  set_smem_limit_once(kernel, kMaxSmem);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((a.lout + np * PPT - 1) / (np * PPT), (a.s.cout + CB - 1) / CB, a.B);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  GW_CUDA(cudaLaunchKernelEx(&cfg, kernel, a, t));
}

struct Choice {
  int cpt, ppt, CB, np;
};

// The tile of a launch.  A thread's tile (channels x positions) sets how many
// FMAs a loaded value feeds; on full launches 256 -> 256 channels, 256 items of
// 128 positions take 540 us at 8 x 8, 560 us at 8 x 4 and 637 us at 4 x 4, and the
// tiles' `eff` are about in that ratio (2 x 4: by where it overtakes 4 x 4).  A
// launch with few outputs does better with smaller tiles: with fewer than about
// 384 threads per SM the chip idles (32 x 64 x 1024 outputs: 29.6 us at 8 x 8, 26.8
// us at 8 x 4; one window of 4096, 64 -> 32 channels: 27.2 us at 8 x 8, 18.9 us at
// 8 x 4, 15.4 us at 4 x 4, 13.5 us at 2 x 4; two windows of 32768, the same layer:
// 16.2 us at 4 x 4, 18.3 us at 2 x 4; the last two lines at 8 channels per stage).
// The score is that efficiency over the outputs computed, the ones beyond the end
// of a row included.  The batch decides only the tile, never the order of a sum.
Choice plan_conv_f32(const ConvF32Args& a) {
  const LayerSpec& s = a.s;
  const int sms = current_sm_count();
  const bool one = s.cout == 1;
  static const struct {
    int cpt, ppt, threads;
    double eff;
  } kTiles[4] = {{8, 8, 128, 0.86}, {8, 4, 256, 0.80}, {4, 4, 256, 0.70}, {2, 4, 256, 0.45}};
  // channels per CTA: a power of two, at most 64, that divides the padded weight
  // row (a CTA stages its channels of a row unchecked)
  int cmax = 8;
  while (cmax < 64 && conv_f32_cop(s.cout) % (2 * cmax) == 0) cmax *= 2;
  Choice best{};
  double best_score = -1;
  for (int v = 0; v < (one ? 2 : 4); ++v) {
    const int ppt = kTiles[v].ppt, cpt = one ? 1 : kTiles[v].cpt;
    // 2 x 4: 32 channels per CTA, and 16 of half the threads when even that leaves
    // two thirds of the SMs without a CTA (BBHnet, at 8 channels per stage: one
    // segment 163 us at 64 channels, 143 us at 16; eight 235 us at 64, 171 us at 32,
    // 222 us at 16)
    const bool few = cpt == 2 && (double)a.lout * a.B * s.cout * 3 < 256.0 * 8 * sms;
    const int CB = one ? 1 : std::min(cmax, cpt == 2 ? (few ? 16 : 32) : 64);
    double np_eff = 1;
    for (int np = kTiles[v].threads / (few ? 2 : 1) / (CB / cpt); np >= 8; np /= 2, np_eff *= 0.98) {
      const int threads = np * (CB / cpt), TL = np * ppt;
      if (threads < 64) break;
      const double tiles = (double)((a.lout + TL - 1) / TL) * ((s.cout + CB - 1) / CB) * a.B;
      const double useful = (double)a.lout * a.B * s.cout / (tiles * TL * CB);
      // with 8 channels in all, an 8 x 8 tile leaves too few CTAs per row in
      // flight (64 x 8 x 32768 outputs: 126 us, 120 us at 8 x 4)
      const double eff = kTiles[v].eff - (cpt == 8 && ppt == 8 && CB == 8 ? 0.08 : 0.0);
      const double score = useful * eff * np_eff * std::min(1.0, tiles * threads / (384.0 * sms));
      if (score > best_score) {
        best_score = score;
        best = {cpt, ppt, CB, np};
      }
    }
  }
  return best;
}

template <int K, int S, bool TR2>
void launch_shape(const ConvF32Args& a, cudaStream_t st) {
  const Choice c = plan_conv_f32(a);
  if (c.cpt == 8 && c.ppt == 8)
    launch_tile<K, S, TR2, 8, 8>(a, c.CB, c.np, st);
  else if (c.cpt == 8)
    launch_tile<K, S, TR2, 8, 4>(a, c.CB, c.np, st);
  else if (c.cpt == 4)
    launch_tile<K, S, TR2, 4, 4>(a, c.CB, c.np, st);
  else
    launch_tile<K, S, TR2, 2, 4>(a, c.CB, c.np, st);
}

template <int K>
void launch_one_channel(const ConvF32Args& a, cudaStream_t st) {
  const Choice c = plan_conv_f32(a);
  if (c.ppt == 8)
    launch_tile<K, 1, false, 1, 8>(a, c.CB, c.np, st);
  else
    launch_tile<K, 1, false, 1, 4>(a, c.CB, c.np, st);
}

}  // namespace

void launch_conv_f32(const ConvF32Args& a, cudaStream_t st) {
  const LayerSpec& s = a.s;
  const bool tr = s.transposed;
  // the kernel's geometry is built on these paddings (every layer of the two
  // networks and every data gradient of the trainer has them)
  const bool pads = s.k == 1 || (s.k == 7 && s.pad_l == 3) || (s.k == 16 && s.pad_l == 7);
  if (!pads) {
    throw Error(GW_EINVAL, "layer shape has no FP32 conv kernel (DeepClean and BBHnet shapes only)");
  } else if (s.k == 7 && s.stride == 1 && s.cout == 1)
    launch_one_channel<7>(a, st);
  else if (s.k == 7 && s.stride == 1)
    launch_shape<7, 1, false>(a, st);
  else if (s.k == 7 && s.stride == 2 && !tr)
    launch_shape<7, 2, false>(a, st);
  else if (s.k == 7 && s.stride == 2 && tr)
    launch_shape<7, 2, true>(a, st);
  else if (s.k == 16 && s.stride == 1 && !tr)
    launch_shape<16, 1, false>(a, st);
  else if (s.k == 1 && s.stride == 2 && !tr)
    launch_shape<1, 2, false>(a, st);
  else
    throw Error(GW_EINVAL, "layer shape has no FP32 conv kernel (DeepClean and BBHnet shapes only)");
}

}  // namespace gw
