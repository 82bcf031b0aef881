// Learned-boundary network: sizes, parameter layout and the internal entry
// points of mlp.cu.
#pragma once

#include <cstddef>
#include <cuda_runtime.h>

namespace mlpnet {
constexpr int NI = 324, NH = 64, NO = 6;  // 3x3x3 stencil x 6 fields x 2 steps -> 64 -> 64 -> 6
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NI, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NO * NH, NPARAM = OFF_B3 + NO;
constexpr float R_MIN = 1e-30f;  // smaller stencil RMS counts as a zero stencil
} // namespace mlpnet

// Scratch of the forward / gradient / training calls for minibatches of
// `batch` samples over a set of n samples (the training permutation).
size_t mlp_scratch_bytes(int batch, long long n);
cudaError_t mlp_forward(const float *params, const float *X, long long n, float *Y, cudaStream_t st);
cudaError_t mlp_grad(const float *params, const float *X, const float *T, int n, float *grad, double *loss_host,
                     void *scratch, int batch, cudaStream_t st);
cudaError_t mlp_train(float *params, const float *X, const float *T, long long n, int batch, int epochs, double lr,
                      unsigned long long seed, void *scratch, cudaStream_t st, double *last_epoch_loss);
// The box [lo, hi) of a state (six components at f + c*fstride, rows of
// `pitch`) into dst [6][box cells], and the pairs of `n` of its cells from two
// such copies (S^{n-1}, S^n) and the whole state S^{n+1}.
cudaError_t mlp_record_box(const float *f, long long fstride, int pitch, int ny, const int lo[3], const int hi[3],
                           float *dst, cudaStream_t st);
// ce, ca (nullable): the reference's E coefficients, for the box's own Yee
// step of each recorded cell.
cudaError_t mlp_record(const float *prev, const float *cur, const float *nxt, long long fstride, int pitch, int ny,
                       const int lo[3], const int hi[3], const int *cells, int n, const float *ce, const float *ca,
                       float neg_dt, float *X, float *Y, cudaStream_t st);

// The learned layer's geometry: the six faces of the domain (0..5 = x low, x
// high, y low, ...), each with in-plane axes u, v (the other two, the lower one
// first) of nu x nv cells.  A face computes the cells [u0, u1) x [v0, v1) of
// its plane (each cell of the layer belongs to one face), numbered from
// cell0, u fastest, in pu x pv patches from patch0; `depth` planes (itself
// and the next inward, if there is one) of the six components are kept in a
// snapshot from float `snap`.
struct LearnedFace {
    int nu, nv, depth;
    int u0, u1, v0, v1;
    int pu, pv, patch0;
    long long snap, cell0;
};
struct LearnedGeo {
    int nx, ny, nz, patches;
    LearnedFace face[6];
    long long snap_floats, cells;
};
LearnedGeo learned_geometry(int nx, int ny, int nz);

// Layer update of a simulation step (FP32 fields at f + c*fs, rows of `pitch`):
// a snapshot of the faces' planes; the corrections r f of the layer's cells
// from the snapshots of S^n and S^{n-1} into out [6][cells]; the corrections
// added after the Yee step.  `image`: learned_image_bytes() of weights in the
// kernel's order, made once by learned_layer_configure.
size_t learned_image_bytes();
cudaError_t learned_layer_configure(const float *params, void *image, cudaStream_t st);
cudaError_t learned_snapshot(const LearnedGeo &g, const float *f, long long fs, int pitch, float *snap, cudaStream_t st);
cudaError_t learned_layer_predict(const LearnedGeo &g, const float *params, const void *image, const float *cur,
                                  const float *prev, float *out, int grid, cudaStream_t st);
cudaError_t learned_layer_scatter(const LearnedGeo &g, float *f, long long fs, int pitch, const float *vals,
                                  cudaStream_t st);
