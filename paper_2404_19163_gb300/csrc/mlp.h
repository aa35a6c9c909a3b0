// Learned start proposal: feature and MLP kernels (k_mlp.cu).
#pragma once
#include "common.cuh"

namespace zf {

constexpr int kMlpParams = 5573;  // 16*64 + 64 + 64*64 + 64 + 5*64 + 5

// Y (batch x 5) = the network's outputs.
cudaError_t launch_mlp(const float* P, const float* mean, const float* stdv, const float* X, int batch, float* Y,
                       cudaStream_t s);
int mlp_chunks(int batch);
// grad = the batch's gradient of the training loss and *loss its mean loss; part holds
// mlp_chunks(batch) x kMlpParams floats and lpart mlp_chunks(batch) doubles of scratch.
cudaError_t launch_mlp_backward(const float* P, const float* mean, const float* stdv, const float* X, int batch,
                                const float* tgt, const int* ord, float w, float* part, double* lpart, float* grad,
                                double* loss, cudaStream_t s);
cudaError_t launch_adam(float* P, const float* G, float* M, float* V, int n, int step, float lr, float b1, float b2,
                        float eps, cudaStream_t s);
// rows (3n doubles) and the row statistics st[0..5] (g_hi, g_lo, mean/min diagonal, mean/min row sum)
cudaError_t launch_feat_rows(const double* S, int n, double* rows, double* st, cudaStream_t s);
cudaError_t launch_feat_d0(const double* S, int n, const double* st, double* D0, unsigned long long* amax,
                           cudaStream_t s);
int feat_trace_blocks(int n);
cudaError_t launch_feat_traces(const double* D0, const double* P, int n, double* part, const double* st, float* f,
                               cudaStream_t s);

}  // namespace zf
