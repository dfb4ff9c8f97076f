// Internal declarations of the training path (train.cu, k_train.cu).
#pragma once

#include <algorithm>

#include "gw_internal.h"

namespace gw {

constexpr float kBnEps = 1e-5f;

// One layer's raw parameters inside the flat parameter vector (offsets in
// floats; the BatchNorm ones only when bn) and its folded device copies.
struct FoldArgs {
  const float* p;             // raw parameters (device)
  int64_t off_w, off_b, off_g, off_be, off_mu, off_var;
  int cin, cout, K, transposed, bn;
  float* wf;                  // folded [C_in][K][conv_f32_cop(C_out)]
  float* wT;                  // folded, transposed [C_out][K][conv_f32_cop(C_in)], or null
  float* bf;                  // folded bias [C_out]
};

// Weight-gradient contraction dW[a][c][k] = sum_{b,t} A[b][a][t] Bv(b, c, s t + k - p)
// (Bv = Bm inside [0, LB), 0 outside) and the bias gradient: 1 = sum_t
// A[a][t] (conv: A is the output gradient), 2 = sum_u Bm[c][u] (transposed
// conv: Bm is the output gradient; needs LB = s LA and p + s <= K), 0 = none.
struct WgradArgs {
  const float* A; int64_t ab, aa; int NA, LA;
  const float* Bm; int64_t bb, bc; int NC, LB;
  int K, s, p;
  int bias;
  float* partial;
  size_t partial_cap;  // FP32 kernel: at most this many floats of partials (but at least one CTA's)
};

// Several layers' folds in one launch (at most kFoldMax).
constexpr int kFoldMax = 16;
void launch_fold_many(const FoldArgs* f, int n, cudaStream_t st);
// Several layers' unfolds in one launch (at most kFoldMax).
struct UnfoldItem {
  FoldArgs f;
  const float* dWf;
  int dw_in_major;  // dWf is [C_in][C_out][K] (transposed conv) instead of [C_out][C_in][K]
  const float* dbf;
};
void launch_unfold_many(const UnfoldItem* u, int n, float* dp, cudaStream_t st);
// FP32 (k_wgrad_f32.cu).  launch_wgrad_f32 writes per-CTA partials
// (w.partial: wgrad_f32_partial_floats) and returns what launch_wgrad_reduce
// needs to add them into out (NA * NC * K floats) and db; several layers go
// into one reduction.
struct WgradReduceItem {
  const float* partial;
  int parts, cols, n_w;  // partials of `cols` floats: n_w weights, then the bias
  float *out, *db;
};
constexpr int kWgradReduceMax = 16;
size_t wgrad_f32_partial_floats(const WgradArgs& w, int B);
WgradReduceItem launch_wgrad_f32(const WgradArgs& w, int B, float* out, float* db, cudaStream_t st);
void launch_wgrad_reduce(const WgradReduceItem* items, int n, cudaStream_t st);
// The same weight gradient on the tensor cores (BF16 operands, FP32
// accumulation; k_wgrad_tc.cu): w.partial must hold wgrad_tc_partial_floats;
// err receives a bounded wait's give-up.  Returns what launch_wgrad_tc_reduce
// needs to add the partials into out (NA * NC * K floats) and, with w.bias, db.
struct WgradTcReduceItem {
  const float* partial;  // [parts][Npad][NAp]
  int parts, NA, NAp, NC, N, Npad, bias, s;
  float *out, *db;
};
bool wgrad_tc_supported(const WgradArgs& w);
size_t wgrad_tc_partial_floats(const WgradArgs& w, int B);
WgradTcReduceItem launch_wgrad_tc(const WgradArgs& w, int B, float* out, float* db, int* err, cudaStream_t st);
void launch_wgrad_tc_reduce(const WgradTcReduceItem* items, int n, cudaStream_t st);
void launch_standardise(const float* x, int B, int C, int L, const float* mean, const float* istd, float* y,
                        cudaStream_t st);
// loss = (1 / (B Lr)) sum r^2 with r = g (*) (strain - y_hat) valid (Lr = L - K + 1);
// r holds B * Lr floats, part band_loss_part_floats.
size_t band_loss_part_floats(int B, int L, int K);
void launch_band_loss(const float* strain, const float* y_hat, int B, int L, const float* taps, int K, float* r,
                      float* part, float* loss, cudaStream_t st);
// dy_hat = dloss * d loss / d y_hat (dloss: device scalar, or null for 1).
void launch_band_loss_backward(const float* r, int B, int L, const float* taps, int K, const float* dloss,
                               float* dy_hat, cudaStream_t st);
void launch_adam(float* p, const float* g, float* m, float* v, int64_t n, int step, float lr, float b1, float b2,
                 float eps, cudaStream_t st);
// Adam with the step count in device memory (incremented by the first of two launches).
void launch_adam_dev(float* p, const float* g, float* m, float* v, int64_t n, int* step, float lr, float b1,
                     float b2, float eps, cudaStream_t st);

}  // namespace gw
