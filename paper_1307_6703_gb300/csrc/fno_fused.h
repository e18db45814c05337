// fno_fused.h -- the network's layers and projection as fused kernels
// (fno_fused.cu).  Internal to the library; not part of the C ABI.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace fno {

constexpr int kWidth = 32;  // channels the fused kernels are written for
constexpr int kFeat = 5;    // input features

// Shape of a pass: B fields of nx x ny; C = kWidth, H hidden (32 or 64), O
// outputs, K2 = 2 modes_x (at most 64).
struct Shape {
  int B, nx, ny, H, O, K2;
};
bool fused_supported(int width, int hidden, int modes_x);
// Tiles of a pass (128 sites of one row each) and, per tile, the FP64 partial
// sums of a kernel's reductions.
long long fused_tiles(const Shape &s);

// Features and lift: x0[b][5][s], and v0 = P x + p as BF16, channel-major
// cm[b][c][s] and site-major sm[b][s][c].
cudaError_t lift(const Shape &s, const float *prm, const float *P, const float *pb, float *x0, __nv_bfloat16 *cm,
                 __nv_bfloat16 *sm, cudaStream_t st);

// One layer: z = W v + w + (G Fxi), v' = gelu(z) (last: z).  v_sm: the input,
// site-major; G[b c][y][j]: rows of the inverse transform; FxiT[x][j].  z is
// kept (FP32) for the backward pass; v' as BF16 in both layouts.
cudaError_t layer_forward(const Shape &s, const __nv_bfloat16 *v_sm, const __nv_bfloat16 *W, const float *w,
                          const __nv_bfloat16 *G, const __nv_bfloat16 *FxiT, bool last, float *z, __nv_bfloat16 *cm,
                          __nv_bfloat16 *sm, int *err, cudaStream_t st);

// Projection: out = Q2 gelu(Q1 v + q1) + q2 (into out and, if set, out_user).
cudaError_t project_forward(const Shape &s, const __nv_bfloat16 *v_sm, const __nv_bfloat16 *Q1, const float *q1,
                            const float *Q2, const float *q2, float *out, float *out_user, int *err, cudaStream_t st);

// Loss and its gradient through the projection: dhp as BF16 [b][h][s]; dz of
// the last layer = Q1^T dhp as BF16 in both layouts, and its sums over groups
// of four sites, quads[b][c][s / 4]; per tile the sums dq1[H], dQ2[O][H],
// dq2[O], loss (part).
int project_back_sums(const Shape &s);
cudaError_t project_backward(const Shape &s, const __nv_bfloat16 *v_sm, const __nv_bfloat16 *Q1, const float *q1,
                             const float *Q2, const __nv_bfloat16 *Q1T, const float *out, const float *target,
                             __nv_bfloat16 *dhp, __nv_bfloat16 *dz_cm, __nv_bfloat16 *dz_sm, float *quads, double *part,
                             int *err, cudaStream_t st);

// Backward through a layer: dv = W^T dz + dA Fx^T.  With zprev (the layer
// below's z): dz' = dv gelu'(zprev) as BF16 in both layouts and its quads.
// Without (the first layer): dv itself, FP32 [b][c][s].
cudaError_t layer_backward(const Shape &s, const __nv_bfloat16 *dz_sm, const __nv_bfloat16 *WT, const __nv_bfloat16 *dA,
                           const __nv_bfloat16 *Fx, const float *zprev, __nv_bfloat16 *cm, __nv_bfloat16 *sm,
                           float *quads, float *dv, int *err, cudaStream_t st);

// Per-tile sums added up in a fixed order into consecutive ranges of outputs
// and, after them, *loss (FP64, divided by `count`).  part2: finish_scratch
// doubles.
struct SumOut {
  float *out;
  int n;
};
long long finish_scratch(int nval);
cudaError_t finish_sums(const double *part, long long tiles, int nval, const SumOut (&o)[3], double *loss, double count,
                        double *part2, cudaStream_t st);

}  // namespace fno
