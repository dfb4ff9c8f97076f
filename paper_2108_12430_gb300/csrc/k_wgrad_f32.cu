// FP32 weight and bias gradients of a conv / transposed-conv layer (7 taps,
// stride 1 or 2, padding 3: DeepClean's layers):
//   dW[a][c][k] = sum_{b, t} A[b][a][t] Bm[b][c][s t + k - 3]
// (conv: A = the output gradient, Bm = the layer input; transposed conv: A =
// the layer input, Bm = the output gradient), Bm = 0 outside [0, LB).
//
// Bound: the FP32 FMA pipe, and close behind it the 128 bytes per clock of
// shared-memory loads, so a thread keeps 4 A channels x 1 B channel x 7 taps
// in registers: per position it loads 4 A values and one (stride 1) or two new
// B values for 28 FMAs.  The FMAs are packed over two neighbouring positions
// (even and odd partial sums): an A pair is an aligned 64-bit shared-memory
// value, a B pair at an odd offset costs two moves for the 4 FMAs it feeds.
// That needs neither operand transposed on the way in, so rows are staged by
// cp.async as they lie (a stride-2 operand split into even and odd samples), one
// chunk of positions ahead.
//
// Warp: 8 B channels x 4 runs of kRun positions (lane = run * 8 + channel), for
// one block of 4 A channels; rows are padded so that the 8 channels of a
// 16-byte load fall into distinct banks.  CTA: an `an` x `cn` rectangle of such
// warp tiles, times `tg` groups of runs where the layer has fewer tiles than
// the CTA warps.  CTAs walk the (item, chunk) list with a grid stride and keep
// their sums in registers; runs and groups are added in a fixed order, each
// CTA writes one partial, and one kernel adds the partials of every layer that the
// trainer's buffer holds in CTA order, so gradients are bitwise reproducible.
//
// The bias gradient rides along: conv, the sum of A; transposed conv, the sum
// of Bm over taps 3 .. 3 + s - 1, which visits every output position once
// (LB = s LA).
//
// Measured (GB300, 32 windows of 21 x 8192): all eight layers 806 -> 225 us
// (17 TFLOP/s; 64 x 32 channels 184 -> 46 us) against one A value per
// thread feeding up to 16 outputs; their reductions 381 -> 10 us against one
// thread per column over up to 1024 partials, one launch per layer; the
// bias gradients' own row sums (92 us) are gone; the step 1488 -> 654 us.
#include <algorithm>

#include "gw_train.h"
#include "tc_ptx.h"

namespace gw {

namespace {

constexpr int kK = 7, kPad = 3;
constexpr int kRun = 32;          // consecutive positions of a thread per chunk
constexpr int kRuns = 4;          // runs per warp
constexpr int kWarps = 8;
constexpr int kMaxSmem = 110 * 1024;

struct WgTile {
  int an, cn, tg;     // warp tiles per CTA: A blocks x B blocks x groups of runs
  int ab_tiles;       // CTAs along the A blocks (blockIdx.y = B part * ab_tiles + A part)
  int T;              // positions per chunk: tg * kRuns * kRun
  int ap, bp, odd;    // floats per staged A row, B row; offset of a B row's odd samples
  int span;           // B samples staged per row
  int stage_floats;
  int chunks_per_b, n_chunks;
  int cols;           // partial columns: NA NC 7, then the bias (if any)
};

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float sum2(f32x2 v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return lo + hi;
}
// `bytes` of 4 (or 16) are copied, the rest is zero-filled.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(bytes)
               : "memory");
}
// One row of n samples from position x0 (row valid in [0, len)) to dst, by the
// calling warp; 16 bytes at a time where the row allows it.
__device__ __forceinline__ void stage_row(float* dst, const float* row, int x0, int n, int len, int lane) {
  if (((uintptr_t)(row + x0) & 15) == 0 && (x0 & 3) == 0) {
    for (int j = 4 * lane; j < n; j += 128) {
      const int left = x0 + j < 0 ? 0 : len - (x0 + j);  // x0 + j is a multiple of 4
      cp_async16(dst + j, row + (left > 0 ? x0 + j : 0), left >= 4 ? 16 : (left > 0 ? 4 * left : 0));
    }
  } else {
    for (int j = lane; j < n; j += 32) {
      const bool ok = (unsigned)(x0 + j) < (unsigned)len;
      cp_async4(dst + j, row + (ok ? x0 + j : 0), ok ? 4 : 0);
    }
  }
}

template <int S, int NAT>
__global__ void __launch_bounds__(32 * kWarps, 2)
    wgrad_f32_kernel(const __grid_constant__ WgradArgs w, const __grid_constant__ WgTile g) {
  extern __shared__ __align__(16) float smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwarps = blockDim.x >> 5;
  const int ai = warp % g.an, ci = (warp / g.an) % g.cn, ti = warp / (g.an * g.cn);
  const int a0 = (blockIdx.y % g.ab_tiles) * g.an * NAT, c0 = (blockIdx.y / g.ab_tiles) * g.cn * 8;
  const int cl = ci * 8 + (lane & 7);           // this thread's B channel within the CTA's
  const int run = ti * kRuns + (lane >> 3);     // and its run of positions
  const int rows_a = g.an * NAT, rows_b = g.cn * 8;
  // B row sample 0 is position s t0 - 3 - kShift (stride 1: a multiple of 4)
  constexpr int kShift = S == 1 ? 1 : 0;

  auto stage = [&](int st, int chunk) {
    const int b = chunk / g.chunks_per_b, t0 = (chunk - b * g.chunks_per_b) * g.T;
    float* As = smem + st * g.stage_floats;
    float* Bs = As + rows_a * g.ap;
    for (int r = warp; r < rows_a + rows_b; r += nwarps) {
      if (r < rows_a) {
        const bool ok = a0 + r < w.NA;
        const float* row = w.A + (int64_t)b * w.ab + (int64_t)(ok ? a0 + r : 0) * w.aa;
        stage_row(As + r * g.ap, row, t0, g.T, ok ? w.LA : 0, lane);
      } else {
        const int c = r - rows_a;
        const bool ok = c0 + c < w.NC;
        const float* row = w.Bm + (int64_t)b * w.bb + (int64_t)(ok ? c0 + c : 0) * w.bc;
        const int len = ok ? w.LB : 0;
        float* dst = Bs + c * g.bp;
        if constexpr (S == 1) {
          stage_row(dst, row, t0 - kPad - kShift, g.span, len, lane);
        } else {
#pragma unroll 4
          for (int j = lane; j < g.span; j += 32) {
            const int x = S * t0 - kPad + j;
            const bool in = (unsigned)x < (unsigned)len;
            cp_async4(dst + ((j & 1) ? g.odd : 0) + (j >> 1), row + (in ? x : 0), in ? 4 : 0);
          }
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  f32x2 acc[NAT][kK], bacc[NAT];
#pragma unroll
  for (int a = 0; a < NAT; ++a) {
    bacc[a] = 0ull;
#pragma unroll
    for (int k = 0; k < kK; ++k) acc[a][k] = 0ull;
  }
  // bias 1: one warp row of B blocks sums A; bias 2: one of A blocks sums Bm (in bacc[0])
  const bool bias1 = w.bias == 1 && ci == 0 && c0 == 0, bias2 = w.bias == 2 && ai == 0 && a0 == 0;
  const f32x2 one2 = pack2(1.f, 1.f);

  int chunk = blockIdx.x;
  if (chunk < g.n_chunks) stage(0, chunk);
  for (int st = 0; chunk < g.n_chunks; chunk += gridDim.x, st ^= 1) {
    if (chunk + (int)gridDim.x < g.n_chunks) {
      stage(st ^ 1, chunk + gridDim.x);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const int tb = (chunk % g.chunks_per_b) * g.T + run * kRun;  // first position of this thread's run
    const float* ar = smem + st * g.stage_floats + ai * NAT * g.ap + run * kRun;
    const float* br = smem + st * g.stage_floats + rows_a * g.ap + cl * g.bp + run * kRun;
    // B samples of a block of 8 positions: stride 1, v[j + k + 1]; stride 2,
    // v[j + k / 2] (even k) and o[j + k / 2] (odd k).  The first 8 (4) slots
    // carry over from the block before.
    float v[16], o[12];
    auto load4 = [](const float* p, float* d) {
      const float4 q = *reinterpret_cast<const float4*>(p);
      d[0] = q.x, d[1] = q.y, d[2] = q.z, d[3] = q.w;
    };
    if constexpr (S == 1) {
      load4(br, v + 8), load4(br + 4, v + 12);
    } else {
      load4(br, v + 8), load4(br + g.odd, o + 8);
    }
#pragma unroll
    for (int q = 0; q < kRun / 8; ++q) {
      if constexpr (S == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = v[8 + i];
        load4(br + 8 * q + 8, v + 8), load4(br + 8 * q + 12, v + 12);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = v[8 + i], o[i] = o[8 + i];
        load4(br + 8 * q + 4, v + 4), load4(br + 8 * q + 8, v + 8);
        load4(br + g.odd + 8 * q + 4, o + 4), load4(br + g.odd + 8 * q + 8, o + 8);
      }
      auto bval = [&](int j, int k) { return S == 1 ? v[(j + k + 1) & 15] : ((k & 1) ? o[(j + k / 2) % 12] : v[j + k / 2]); };
      if (tb + 8 * q + 8 <= w.LA) {
#pragma unroll
        for (int jj = 0; jj < 8; jj += 4) {
          ulonglong2 av[NAT];
#pragma unroll
          for (int a = 0; a < NAT; ++a)
            av[a] = *reinterpret_cast<const ulonglong2*>(ar + a * g.ap + 8 * q + jj);
#pragma unroll
          for (int j = 0; j < 4; j += 2) {
#pragma unroll
            for (int k = 0; k < kK; ++k) {
              const f32x2 bv = pack2(bval(jj + j, k), bval(jj + j + 1, k));
#pragma unroll
              for (int a = 0; a < NAT; ++a) acc[a][k] = fma2(j ? av[a].y : av[a].x, bv, acc[a][k]);
            }
            if (bias1) {
#pragma unroll
              for (int a = 0; a < NAT; ++a) bacc[a] = fma2(j ? av[a].y : av[a].x, one2, bacc[a]);
            }
            if (bias2) {
#pragma unroll
              for (int k = kPad; k < kPad + S; ++k)
                bacc[0] = fma2(pack2(bval(jj + j, k), bval(jj + j + 1, k)), one2, bacc[0]);
            }
          }
        }
      } else {
        // the row ends in this block: positions beyond it take no part
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (tb + 8 * q + j >= w.LA) continue;
          f32x2 av[NAT];
#pragma unroll
          for (int a = 0; a < NAT; ++a) av[a] = pack2(ar[a * g.ap + 8 * q + j], 0.f);
#pragma unroll
          for (int k = 0; k < kK; ++k)
#pragma unroll
            for (int a = 0; a < NAT; ++a) acc[a][k] = fma2(av[a], pack2(bval(j, k), 0.f), acc[a][k]);
          if (bias1) {
#pragma unroll
            for (int a = 0; a < NAT; ++a) bacc[a] = fma2(av[a], one2, bacc[a]);
          }
          if (bias2) {
#pragma unroll
            for (int k = kPad; k < kPad + S; ++k) bacc[0] = fma2(pack2(bval(j, k), 0.f), one2, bacc[0]);
          }
        }
      }
    }
    __syncthreads();
  }

  // even + odd positions, then the warp's runs, then the groups of runs
  float r[NAT * (kK + 1)];
#pragma unroll
  for (int a = 0; a < NAT; ++a) {
#pragma unroll
    for (int k = 0; k < kK; ++k) r[a * kK + k] = sum2(acc[a][k]);
    r[NAT * kK + a] = sum2(bacc[a]);
  }
#pragma unroll
  for (int e = 0; e < NAT * (kK + 1); ++e) {
    r[e] += __shfl_xor_sync(0xffffffffu, r[e], 8);
    r[e] += __shfl_xor_sync(0xffffffffu, r[e], 16);
  }
  if (g.tg > 1) {
    const int tiles = g.an * g.cn, tile = warp % tiles;
    float* red = smem;  // [tg - 1][NAT (7 + 1)][tiles * 8]
    if (ti > 0 && lane < 8)
#pragma unroll
      for (int e = 0; e < NAT * (kK + 1); ++e)
        red[((ti - 1) * NAT * (kK + 1) + e) * tiles * 8 + tile * 8 + lane] = r[e];
    __syncthreads();
    if (ti == 0 && lane < 8)
      for (int t = 0; t + 1 < g.tg; ++t)
#pragma unroll
        for (int e = 0; e < NAT * (kK + 1); ++e) r[e] += red[(t * NAT * (kK + 1) + e) * tiles * 8 + tile * 8 + lane];
  }
  const int c = c0 + cl;
  if (ti == 0 && lane < 8) {
    float* out = w.partial + (int64_t)blockIdx.x * g.cols;
#pragma unroll
    for (int a = 0; a < NAT; ++a) {
      const int ag = a0 + ai * NAT + a;
      if (ag >= w.NA) continue;
      if (c < w.NC) {
#pragma unroll
        for (int k = 0; k < kK; ++k) out[((int64_t)ag * w.NC + c) * kK + k] = r[a * kK + k];
      }
      if (bias1 && lane == 0) out[(int64_t)w.NA * w.NC * kK + ag] = r[NAT * kK + a];
    }
    if (bias2 && c < w.NC) out[(int64_t)w.NA * w.NC * kK + c] = r[NAT * kK];
  }
}

// Sums of every layer's partials, in CTA order: a block takes 32 columns of one
// layer (blockIdx.y), warp w the CTAs w, w + 8, ..., and the eight sums are
// added in warp order.
struct ReduceList {
  WgradReduceItem it[kWgradReduceMax];
};
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const __grid_constant__ ReduceList l) {
  __shared__ float red[8][32];
  const WgradReduceItem& it = l.it[blockIdx.y];
  if ((int)blockIdx.x * 32 >= it.cols) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e = blockIdx.x * 32 + lane;
  float acc = 0.f;
  if (e < it.cols) {
    const float* src = it.partial + e;
    int g = warp;
    for (; g + 24 < it.parts; g += 32) {  // four partials in flight
      const float v0 = src[(int64_t)g * it.cols], v1 = src[(int64_t)(g + 8) * it.cols];
      const float v2 = src[(int64_t)(g + 16) * it.cols], v3 = src[(int64_t)(g + 24) * it.cols];
      acc += v0;
      acc += v1;
      acc += v2;
      acc += v3;
    }
    for (; g < it.parts; g += 8) acc += src[(int64_t)g * it.cols];
  }
  red[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && e < it.cols) {
    float t = 0.f;
    for (int i = 0; i < 8; ++i) t += red[i][lane];
    if (e < it.n_w)
      it.out[e] = t;
    else
      it.db[e - it.n_w] = t;
  }
}

WgTile plan(const WgradArgs& w, int B) {
  WgTile g{};
  const int nat = w.NA == 1 ? 1 : 4;
  const int ab = (w.NA + nat - 1) / nat, cb = (w.NC + 7) / 8;
  g.cn = cb <= 3 ? cb : 2;
  g.an = 1;
  while (g.an * 2 * g.cn <= kWarps && g.an < ab) g.an *= 2;
  g.tg = std::max(1, kWarps / (g.an * g.cn));
  g.ab_tiles = (ab + g.an - 1) / g.an;
  g.T = g.tg * kRuns * kRun;
  g.ap = g.T + 4;
  // row lengths: one 16-byte load past the last run's samples, rows of 8
  // channels 4 floats apart modulo 32 banks
  auto row = [](int n) {
    n = (n + 3) / 4 * 4;
    while (n % 32 != 4) n += 4;
    return n;
  };
  if (w.s == 1) {
    g.span = g.T + 8;
    g.bp = row(g.span);
  } else {
    g.span = 2 * g.T + 8;
    g.odd = (g.T + 4 + 3) / 4 * 4;
    g.bp = row(2 * g.odd);
  }
  g.stage_floats = g.an * nat * g.ap + g.cn * 8 * g.bp;
  g.chunks_per_b = (w.LA + g.T - 1) / g.T;
  g.n_chunks = B * g.chunks_per_b;
  g.cols = w.NA * w.NC * kK + (w.bias == 1 ? w.NA : (w.bias == 2 ? w.NC : 0));
  return g;
}

int parts_of(const WgTile& g, const WgradArgs& w) {
  const int cb_tiles = ((w.NC + 7) / 8 + g.cn - 1) / g.cn;
  const int fit = (int)std::min<size_t>(w.partial_cap / g.cols, 1 << 20);
  return std::max(1, std::min({g.n_chunks, 2 * current_sm_count() / (g.ab_tiles * cb_tiles), fit}));
}

}  // namespace

size_t wgrad_f32_partial_floats(const WgradArgs& w, int B) {
  // fewer items can leave fewer chunks but never more partials
  const WgTile g = plan(w, B);
  return (size_t)parts_of(g, w) * g.cols;
}

WgradReduceItem launch_wgrad_f32(const WgradArgs& w, int B, float* out, float* db, cudaStream_t st) {
  GW_CHECK_ARG(w.K == kK && w.p == kPad && (w.s == 1 || w.s == 2),
               "layer shape has no FP32 weight-gradient kernel (DeepClean shapes only)");
  GW_CHECK_ARG(w.bias == 0 || w.bias == 1 || (w.bias == 2 && w.LB == w.s * w.LA), "bias gradient of this layer shape");
  const WgTile g = plan(w, B);
  const int nat = w.NA == 1 ? 1 : 4, parts = parts_of(g, w);
  const int cb_tiles = ((w.NC + 7) / 8 + g.cn - 1) / g.cn;
  const int threads = 32 * g.an * g.cn * g.tg;
  const size_t red = (size_t)(g.tg - 1) * nat * (kK + 1) * g.an * g.cn * 8;
  const size_t smem = std::max<size_t>(2 * (size_t)g.stage_floats, red) * sizeof(float);
  GW_CHECK_ARG(smem <= kMaxSmem, "weight-gradient tile exceeds shared memory");
  const dim3 grid(parts, g.ab_tiles * cb_tiles);
  auto run = [&](auto kernel) {
    set_smem_limit_once(kernel, kMaxSmem);
    kernel<<<grid, threads, smem, st>>>(w, g);
  };
  if (nat == 1)
    w.s == 1 ? run(wgrad_f32_kernel<1, 1>) : run(wgrad_f32_kernel<2, 1>);
  else
    w.s == 1 ? run(wgrad_f32_kernel<1, 4>) : run(wgrad_f32_kernel<2, 4>);
  GW_LAUNCH_CHECK();
  return {w.partial, parts, g.cols, w.NA * w.NC * kK, out, db};
}

void launch_wgrad_reduce(const WgradReduceItem* items, int n, cudaStream_t st) {
  GW_CHECK_ARG(n >= 1 && n <= kWgradReduceMax, "reduction list size");
  ReduceList l{};
  int mx = 1;
  for (int i = 0; i < n; ++i) {
    l.it[i] = items[i];
    mx = std::max(mx, items[i].cols);
  }
  wgrad_reduce_kernel<<<dim3((mx + 31) / 32, n), 256, 0, st>>>(l);
  GW_LAUNCH_CHECK();
}

}  // namespace gw
