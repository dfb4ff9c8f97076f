// Weight gradient of a conv / transposed-conv layer on the tensor cores (BF16
// operands, FP32 accumulation in TMEM), for the training step's backward.
//
// The weight gradient is one contraction over all (item, position) pairs:
//   dW[a][c][k] = sum_{b, t} A[b][a][t] Bm[b][c][s t + k - 3]
// (conv: A = the output gradient, Bm = the layer input; transposed conv: A =
// the layer input, Bm = the output gradient), zero outside [0, LB).  As a
// GEMM, D[a][n] = sum_t A[a][t] B[n][t] with n = k NC + c and
// B[n][t] = Bm[c][s t + k - 3]: M = the A channels in 128 MMA rows, N = 7 NC
// columns, and the reduction runs over positions, which is the dimension the
// tensor core's K steps walk.  A row of ones in A or B gives the bias gradient.
//
// Bound: neither the tensor core nor DRAM but the way of the operands -- each
// chunk of positions makes a global round trip, is rounded to BF16 and
// rearranged, and only then feeds a few MMAs.  So a CTA (one per SM) runs two
// groups of eight warps, each on its own chunks of 64 positions with its own
// two shared-memory stages and its own TMEM accumulator: while one group waits
// for memory or the tensor core, the other stages.  A thread's share of a chunk
// is fixed: for (row a, 8 positions) it loads 8 values and stores one 16-byte
// segment; for (channel c, 8 positions) it loads the 16 (stride 1) or 24
// (stride 2) samples that the seven taps of those positions read and makes all
// seven tap rows from them in registers, so that no operand passes through
// shared memory twice.  The next chunk's loads are in flight meanwhile.  Segments
// of neighbouring positions lie 16 bytes off a multiple of 128 apart (LBO), so
// that a warp's stores (8 position groups x 4 rows) fall into distinct banks.
// Rows and columns beyond the operands' are never written: they reach only
// accumulator rows and columns that are not read.
//
// At the end the two accumulators are added and stored column by column (lanes
// along rows: coalesced) as the CTA's partial; one kernel adds every layer's
// partials in CTA order (deterministic).
//
// Measured (GB300, 32 windows of 21 x 8192, against one group per CTA on chunks
// of 128, tap rows gathered 2 bytes at a time from shared memory and partials
// stored row by row): all eight layers 243 -> 144 us (64 x 32 channels 35.6 ->
// 13.6 us, the first layer 50 -> 30 us), their reductions 55 us in eight launches
// -> 12 us in one; the BF16 training step 572 -> 398 us.
#include <cuda_bf16.h>

#include <algorithm>

#include "gw_internal.h"
#include "gw_train.h"
#include "tc_ptx.h"

namespace gw {

namespace {

using namespace ptx;

constexpr int kK = 7, kPad = 3;
constexpr int kChunk = 64, kSegs = kChunk / 8;   // positions per chunk, 16-byte segments per row
constexpr int kGroups = 2, kGroupWarps = 8, kGroupThreads = 32 * kGroupWarps;
constexpr int kThreads = kGroups * kGroupThreads;
constexpr int kRowsA = 128;                      // MMA M
constexpr int kTasksA = 2;                       // A segments per thread: 64 rows x 8 segments / 256 threads
constexpr uint32_t kSegA = kRowsA * 16 + 16;     // bytes between neighbouring segments of A (LBO)

struct WgTcParams {
  const float* A;
  int64_t ab, aa;  // A[b][a][t] at A + b ab + a aa + t, t < LA
  int NA, LA;
  const float* Bm;
  int64_t bb, bc;  // Bm[b][c][u] at Bm + b bb + c bc + u, u < LB
  int NC, LB;
  int N, Npad;     // N = 7 NC columns n = k NC + c; Npad: the D columns (N, + 1 for bias 1) rounded up to 32
  int bias;        // 1: B row N all ones (D[a][N] = sum_t A[a][t]); 2: A row NA all ones
  int NAr, NAp;    // D rows kept: NA, + 1 for bias 2; rounded up to 8
  int a_vec, b_vec;  // rows 16-byte aligned at every multiple of 4
  int chunks_per_b, n_chunks;
  float* partial;  // [gridDim.x][Npad][NAp]
  int* err;
};

// n floats (a multiple of 4) of a row valid in [0, len), from position x0 (a
// multiple of 4); zeros outside.
template <int N>
__device__ __forceinline__ void load_run(const float* row, int x0, int len, bool vec, float* v) {
  if (vec) {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
      const int x = x0 + i;
      if (x >= 0 && x + 4 <= len) {
        q = *reinterpret_cast<const float4*>(row + x);
      } else if (x >= 0) {
        if (x < len) q.x = row[x];
        if (x + 1 < len) q.y = row[x + 1];
        if (x + 2 < len) q.z = row[x + 2];
      }
      v[i] = q.x, v[i + 1] = q.y, v[i + 2] = q.z, v[i + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = (unsigned)(x0 + i) < (unsigned)len ? row[x0 + i] : 0.f;
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// (high half of a, low half of b)
__device__ __forceinline__ uint32_t straddle(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x5432); }

// Seven tap rows of 8 positions from the samples w: tap k of position e is
// w[S e + k + 1].  store(k, segment) receives each.
template <int S, typename F>
__device__ __forceinline__ void make_taps(const float* w, F store) {
  if constexpr (S == 1) {
    uint32_t even[8];  // (w[2j], w[2j + 1])
#pragma unroll
    for (int j = 0; j < 8; ++j) even[j] = pack_bf16(w[2 * j], w[2 * j + 1]);
    uint32_t odd[7];  // (w[2j + 1], w[2j + 2])
#pragma unroll
    for (int j = 0; j < 7; ++j) odd[j] = straddle(even[j], even[j + 1]);
#pragma unroll
    for (int k = 0; k < kK; ++k) {
      const uint32_t* q = (k & 1) ? even + (k + 1) / 2 : odd + k / 2;
      store(k, make_uint4(q[0], q[1], q[2], q[3]));
    }
  } else {
    // samples of odd index serve the even taps, samples of even index the odd taps
    uint32_t o[6], e[5], o1[5], e1[4];
#pragma unroll
    for (int j = 0; j < 6; ++j) o[j] = pack_bf16(w[4 * j + 1], j < 5 ? w[4 * j + 3] : 0.f);
#pragma unroll
    for (int j = 0; j < 5; ++j) e[j] = pack_bf16(w[4 * j + 2], w[4 * j + 4]);
#pragma unroll
    for (int j = 0; j < 5; ++j) o1[j] = straddle(o[j], o[j + 1]);
#pragma unroll
    for (int j = 0; j < 4; ++j) e1[j] = straddle(e[j], e[j + 1]);
    store(0, make_uint4(o[0], o[1], o[2], o[3]));
    store(1, make_uint4(e[0], e[1], e[2], e[3]));
    store(2, make_uint4(o1[0], o1[1], o1[2], o1[3]));
    store(3, make_uint4(e1[0], e1[1], e1[2], e1[3]));
    store(4, make_uint4(o[1], o[2], o[3], o[4]));
    store(5, make_uint4(e[1], e[2], e[3], e[4]));
    store(6, make_uint4(o1[1], o1[2], o1[3], o1[4]));
  }
}

template <int S>
__global__ void __launch_bounds__(kThreads, 1) wgrad_tc_kernel(const __grid_constant__ WgTcParams p) {
  // B segments per thread: 8 per channel; stride 1 (the network's first layer)
  // takes up to 64 channels, stride 2 up to 32
  constexpr int kTasksB = S == 1 ? 2 : 1, kW = S == 1 ? 16 : 24;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
  const uint32_t seg_b = (uint32_t)p.Npad * 16u + 16u;
  const uint32_t a_bytes = kSegs * kSegA, stage_bytes = (a_bytes + kSegs * seg_b + 127u) & ~127u;
  // per group: [0..1] stage free (its MMAs done), [2..3] stage staged (one arrival per warp), [4] all MMAs done
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + 2 * kGroups * stage_bytes);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(bars + 5 * kGroups);
  uint32_t* tslot = (uint32_t*)(abort_flag + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = tid / kGroupThreads, gt = tid - grp * kGroupThreads;
  uint8_t* stages = smem + grp * 2 * stage_bytes;
  auto bar = [&](int g, int i) { return smem_u32(&bars[5 * g + i]); };

  if (tid == 0) {
    for (int g = 0; g < kGroups; ++g) {
      for (int i = 0; i < 5; ++i) mbar_init(bar(g, i), (i == 2 || i == 3) ? kGroupWarps : 1);
    }
    *abort_flag = 0u;
    fence_barrier_init();
  }
  if (p.bias) {
    // the row of ones (BF16 1.0) in every stage: staging never writes it
    const uint4 ones = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
    if (gt < 2 * kSegs) {
      const int r = p.bias == 1 ? p.N : p.NA, q = gt & (kSegs - 1);
      uint8_t* tile = stages + (gt / kSegs) * stage_bytes + (p.bias == 1 ? a_bytes + q * seg_b : q * kSegA);
      *reinterpret_cast<uint4*>(tile + (r >> 3) * 128 + (r & 7) * 16) = ones;
    }
  }
  fence_proxy_async_smem();
  const uint32_t acc_cols = p.Npad <= 128 ? 128u : 256u;
  if (warp == 0) tmem_alloc(smem_u32(tslot), kGroups * acc_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot + grp * acc_cols;
  // D = F32, A = B = BF16, both K-major, N >> 3 at bit 17, M >> 4 at bit 24
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.Npad >> 3) << 17) |
                         ((uint32_t)(kRowsA >> 4) << 24);

  // this thread's tasks: (row, segment) pairs, segments fastest
  const float* a_row[kTasksA];
  uint32_t a_dst[kTasksA];
  bool a_on[kTasksA];
  const int q = gt & (kSegs - 1);  // the same segment for all of them
#pragma unroll
  for (int i = 0; i < kTasksA; ++i) {
    const int a = (gt >> 3) + i * (kGroupThreads / kSegs);
    a_on[i] = a < p.NA;
    a_row[i] = p.A + (int64_t)(a_on[i] ? a : 0) * p.aa;
    a_dst[i] = (uint32_t)(q * kSegA + (a >> 3) * 128 + (a & 7) * 16);
  }
  const float* b_row[kTasksB];
  int b_c[kTasksB];
#pragma unroll
  for (int i = 0; i < kTasksB; ++i) {
    const int c = (gt >> 3) + i * (kGroupThreads / kSegs);
    b_c[i] = c < p.NC ? c : -1;
    b_row[i] = p.Bm + (int64_t)(c < p.NC ? c : 0) * p.bc;
  }
  float av[kTasksA][8], bv[kTasksB][kW];
  auto load = [&](int chunk) {
    const int b = chunk / p.chunks_per_b, t = (chunk - b * p.chunks_per_b) * kChunk + 8 * q;
#pragma unroll
    for (int i = 0; i < kTasksA; ++i)
      if (a_on[i]) load_run<8>(a_row[i] + (int64_t)b * p.ab, t, p.LA, p.a_vec, av[i]);
#pragma unroll
    for (int i = 0; i < kTasksB; ++i)
      if (b_c[i] >= 0) load_run<kW>(b_row[i] + (int64_t)b * p.bb, S * t - kPad - 1, p.LB, p.b_vec, bv[i]);
  };

  griddep_wait();  // operands come from the previous kernels
  int i = 0;
  const int first = blockIdx.x * kGroups + grp, step = gridDim.x * kGroups;
  if (first < p.n_chunks) load(first);
  for (int chunk = first; chunk < p.n_chunks; chunk += step, ++i) {
    const int st = i & 1;
    // the stage's previous MMAs (chunk i - 2) have read it
    bool ok = true;
    if (i >= 2 && lane == 0) ok = mbar_wait(bar(grp, st), (uint32_t)((i - 2) >> 1) & 1u, abort_flag, p.err, 1);
    if (!__shfl_sync(0xffffffffu, ok ? 1 : 0, 0)) break;
    uint8_t* a_s = stages + st * stage_bytes;
    uint8_t* b_s = a_s + a_bytes + q * seg_b;
#pragma unroll
    for (int x = 0; x < kTasksA; ++x)
      if (a_on[x])
        *reinterpret_cast<uint4*>(a_s + a_dst[x]) =
            make_uint4(pack_bf16(av[x][0], av[x][1]), pack_bf16(av[x][2], av[x][3]), pack_bf16(av[x][4], av[x][5]),
                       pack_bf16(av[x][6], av[x][7]));
#pragma unroll
    for (int x = 0; x < kTasksB; ++x)
      if (b_c[x] >= 0)
        make_taps<S>(bv[x], [&](int k, uint4 seg) {
          const int n = k * p.NC + b_c[x];
          *reinterpret_cast<uint4*>(b_s + (n >> 3) * 128 + (n & 7) * 16) = seg;
        });
    if (chunk + step < p.n_chunks) load(chunk + step);
    fence_proxy_async_smem();  // the stores above are read by the tensor core (async proxy)
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(grp, 2 + st));
    if (gt == 0) {
      // every warp of the group has staged its part of the chunk
      ok = mbar_wait(bar(grp, 2 + st), (uint32_t)(i >> 1) & 1u, abort_flag, p.err, 4);
      if (ok) {
        tc_fence_after();
        const uint32_t a0 = smem_u32(a_s), b0 = a0 + a_bytes;
#pragma unroll
        for (int j = 0; j < kChunk / 16; ++j)
          mma_f16(tmem, make_desc(a0 + 2 * j * kSegA, kSegA, 128), make_desc(b0 + 2 * j * seg_b, seg_b, 128), idesc,
                  (i > 0 || j > 0) ? 1u : 0u);
        mma_commit(bar(grp, st));
      }
    }
    if (!__shfl_sync(0xffffffffu, ok ? 1 : 0, 0)) break;
  }
  __syncthreads();
  // every MMA of this CTA has completed before the accumulators are read
  if (gt == 0) mma_commit(bar(grp, 4));
  for (int g = 0; g < kGroups; ++g) mbar_wait_landed(bar(g, 4), 0u, p.err, 2);
  tc_fence_after();
  // warp w reads TMEM lanes 32 (w % 4) .. and every fourth block of 32 columns
  const int r = (warp & 3) * 32 + lane;  // TMEM lane = MMA row = A channel
  if ((warp & 3) * 32 < p.NAr) {
    float* dst = p.partial + (int64_t)blockIdx.x * p.Npad * p.NAp + r;
    const uint32_t t0 = *tslot + ((uint32_t)((warp & 3) * 32) << 16);
    const bool used0 = blockIdx.x * kGroups < p.n_chunks, used1 = blockIdx.x * kGroups + 1 < p.n_chunks;
    for (int c0 = 32 * (warp >> 2); c0 < p.Npad; c0 += 32 * (kThreads / 128)) {
      float v[32], u[32];
      tmem_ld32(t0 + (uint32_t)c0, v);
      tmem_ld32(t0 + acc_cols + (uint32_t)c0, u);
      if (r < p.NAr) {
#pragma unroll
        for (int x = 0; x < 32; ++x)
          dst[(int64_t)(c0 + x) * p.NAp] = (used0 ? v[x] : 0.f) + (used1 ? u[x] : 0.f);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(*tslot, kGroups * acc_cols);
}

// Sums of every layer's partials, in CTA order: a block takes 32 consecutive
// values of one layer's [Npad][NAp] (blockIdx.y: the layer), warp w the CTAs w,
// w + 8, ..., and the eight sums are added in warp order.  The bias gradient:
// bias 1, db[a] = column N; bias 2, db[c] = the sum of row NA's columns k NC +
// c over taps 3 .. 3 + s - 1 (every output position u = s t + k - 3 of channel c
// is in exactly one such (t, k)).
constexpr int kRedWarps = 8;
struct ReduceList {
  WgradTcReduceItem it[kWgradReduceMax];
};
__global__ void __launch_bounds__(32 * kRedWarps) wgrad_tc_reduce_kernel(const __grid_constant__ ReduceList l) {
  __shared__ float red[kRedWarps][32];
  const WgradTcReduceItem& q = l.it[blockIdx.y];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e = blockIdx.x * 32 + lane, stride = q.Npad * q.NAp;  // index into [Npad][NAp]
  if ((int)blockIdx.x * 32 >= stride) return;
  const int n = e / q.NAp, a = e - n * q.NAp;
  // the values this lane adds (cnt of them, NC columns apart)
  int cnt = 0;
  if (e < stride) {
    if (a < q.NA)
      cnt = (n < q.N || (q.bias == 1 && n == q.N)) ? 1 : 0;
    else if (q.bias == 2 && a == q.NA && n < q.N && n / q.NC == kPad)
      cnt = q.s;
  }
  float acc = 0.f;
  for (int j = 0; j < cnt; ++j) {
    // four CTAs' partials in flight per step
    const float* src = q.partial + e + j * q.NC * q.NAp;
    int g = warp;
    for (; g + 3 * kRedWarps < q.parts; g += 4 * kRedWarps) {
      const float v0 = src[(int64_t)g * stride], v1 = src[(int64_t)(g + kRedWarps) * stride];
      const float v2 = src[(int64_t)(g + 2 * kRedWarps) * stride], v3 = src[(int64_t)(g + 3 * kRedWarps) * stride];
      acc += v0;
      acc += v1;
      acc += v2;
      acc += v3;
    }
    for (; g < q.parts; g += kRedWarps) acc += src[(int64_t)g * stride];
  }
  red[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && cnt > 0) {
    float t = 0.f;
    for (int w = 0; w < kRedWarps; ++w) t += red[w][lane];
    if (a < q.NA && n < q.N) {
      const int k = n / q.NC, c = n - k * q.NC;
      q.out[((int64_t)a * q.NC + c) * kK + k] = t;
    } else if (a < q.NA) {
      q.db[a] = t;
    } else {
      q.db[n - kPad * q.NC] = t;
    }
  }
}

int wgrad_tc_grid(const WgradArgs& w, int B) {
  const int chunks = B * ((w.LA + kChunk - 1) / kChunk);
  return std::max(1, std::min((chunks + kGroups - 1) / kGroups, current_sm_count()));
}
// D's columns (N, + 1 for the ones row of bias 1) rounded up to 32, and rows
// (NA, + 1 for bias 2) rounded up to 8.
int wg_npad(const WgradArgs& w) { return (kK * w.NC + (w.bias == 1 ? 1 : 0) + 31) / 32 * 32; }
int wg_rows(const WgradArgs& w) { return w.NA + (w.bias == 2 ? 1 : 0); }
size_t wg_smem(int npad) {
  const size_t stage = (kSegs * kSegA + kSegs * ((size_t)npad * 16 + 16) + 127) / 128 * 128;
  return 128 + 2 * kGroups * stage + 5 * kGroups * 8 + 16;
}

}  // namespace

bool wgrad_tc_supported(const WgradArgs& w) {
  // bias 2 sums taps 3 .. 3 + s - 1 of every t < LA: each output position u < LB exactly once when LB = s LA
  const bool bias_ok = w.bias == 0 || w.bias == 1 || (w.bias == 2 && w.LB == w.s * w.LA);
  const int channels = (w.s == 1 ? 2 : 1) * kGroupThreads / kSegs;
  return tc_supported() && bias_ok && w.K == kK && w.p == kPad && (w.s == 1 || w.s == 2) && w.NA >= 1 &&
         w.NA <= kTasksA * kGroupThreads / kSegs && w.NC >= 1 && w.NC <= channels && wg_npad(w) <= 256;
}

size_t wgrad_tc_partial_floats(const WgradArgs& w, int B) {
  return (size_t)wgrad_tc_grid(w, B) * wg_npad(w) * ((wg_rows(w) + 7) / 8 * 8);
}

WgradTcReduceItem launch_wgrad_tc(const WgradArgs& w, int B, float* out, float* db, int* err, cudaStream_t st) {
  GW_CHECK_ARG(wgrad_tc_supported(w), "layer shape outside the tensor-core weight-gradient kernel");
  GW_CHECK_ARG(!w.bias || db, "bias gradient requested without an output");
  WgTcParams p{};
  p.A = w.A;
  p.ab = w.ab;
  p.aa = w.aa;
  p.NA = w.NA;
  p.LA = w.LA;
  p.Bm = w.Bm;
  p.bb = w.bb;
  p.bc = w.bc;
  p.NC = w.NC;
  p.LB = w.LB;
  p.N = kK * w.NC;
  p.Npad = wg_npad(w);
  p.bias = w.bias;
  p.NAr = wg_rows(w);
  p.NAp = (p.NAr + 7) / 8 * 8;
  p.a_vec = w.aa % 4 == 0 && w.ab % 4 == 0 && ((uintptr_t)w.A & 15) == 0;
  p.b_vec = w.bc % 4 == 0 && w.bb % 4 == 0 && ((uintptr_t)w.Bm & 15) == 0;
  p.chunks_per_b = (w.LA + kChunk - 1) / kChunk;
  p.n_chunks = B * p.chunks_per_b;
  p.partial = w.partial;
  p.err = err;
  const int grid = wgrad_tc_grid(w, B);
  auto kernel = w.s == 1 ? wgrad_tc_kernel<1> : wgrad_tc_kernel<2>;
  // the limit is set once per device, to the most any layer may ask for
  set_smem_limit_once(kernel, 227 * 1024);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = wg_smem(p.Npad);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  GW_CUDA(cudaLaunchKernelEx(&cfg, kernel, p));
  return {w.partial, grid, w.NA, p.NAp, w.NC, p.N, p.Npad, w.bias, w.s, out, db};
}

void launch_wgrad_tc_reduce(const WgradTcReduceItem* items, int n, cudaStream_t st) {
  GW_CHECK_ARG(n >= 1 && n <= kWgradReduceMax, "reduction list size");
  ReduceList l{};
  int mx = 1;
  for (int i = 0; i < n; ++i) {
    l.it[i] = items[i];
    mx = std::max(mx, items[i].Npad * items[i].NAp);
  }
  wgrad_tc_reduce_kernel<<<dim3((mx + 31) / 32, n), 32 * kRedWarps, 0, st>>>(l);
  GW_LAUNCH_CHECK();
}

}  // namespace gw
