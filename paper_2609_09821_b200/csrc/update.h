// Multi-tensor kernels of the update phase: what lies between an update's tensor-core products, one launch each.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/im.h"
#include "ppo_finish.cuh"

namespace im {

constexpr int kMaxNetTensors = 2 * IM_MAX_LAYERS;          // weights, or biases, of an actor and a critic

// One parameter tensor of an Adam step.  wb / wbT (weights only): bf16 [rows][ld_wb] and its transpose [cols][ld_wbT].
struct AdamTensor {
    float *param, *m, *v;
    const float *grad;
    uint16_t *wb, *wbT;
    int rows, cols, ld_wb, ld_wbT;
    float inv_c1, inv_c2;                                  // 1 / (1 - beta^t)
    int first_block;
};
struct AdamMultiArgs {
    AdamTensor t[2 * kMaxNetTensors + 1];
    int first_block[2 * kMaxNetTensors + 1];               // (of t, together)
    int n_tensors, n_blocks;
    im_adam_config cfg;
    float *lr;
    const float *grad_scale;                               // or null: 1
    const float *kl;                                       // or null: the learning rate stays; else it follows *kl (im_adaptive_lr)
    float kl_target, lr_min, lr_max;
    int *done;                                             // zero between launches (needed with kl)
};
void adam_multi_add(AdamMultiArgs &a, float *param, const float *grad, float *m, float *v, int rows, int cols, uint16_t *wb, int ld_wb,
                    uint16_t *wbT, int ld_wbT, int t);
cudaError_t launch_adam_multi(AdamMultiArgs &a, cudaStream_t stream);

// Gradient tensors from what the backward products left: dW = sum of the row slices, db = sum of the partial column
// sums, and, if `partial` is given, the global norm over all of them and `extra`, as the clip factor in scale_out.
struct GradMatrix {
    const uint16_t *in;                                    // [slices][.][ld_in] bf16
    float *out;                                            // dense [rows][cols]
    long long slice_stride;
    int ld_in, slices, rows, cols, first_block;
};
struct GradVector {
    const float *in;                                       // [n_rows][ld]
    float *out;                                            // [cols]
    int n_rows, ld, cols, first_block;
};
struct GradReduceArgs {
    GradMatrix m[kMaxNetTensors];
    GradVector v[kMaxNetTensors];
    int m_first[kMaxNetTensors], v_first[kMaxNetTensors];  // first blocks of m and v, together
    int n_matrices, n_vectors, n_blocks;
    const float *extra;
    int n_extra;
    double *partial;                                       // [n_blocks] or null: no norm
    int *done;                                             // zero between launches
    float max_norm, *scale_out;                            // [2]: clip factor, norm
};
int grad_matrix_blocks(int rows, int cols);
int grad_vector_blocks(int cols);
void grad_reduce_add(GradReduceArgs &a, const uint16_t *in, long long slice_stride, int ld_in, int slices, int rows, int cols, float *out);
void grad_reduce_add(GradReduceArgs &a, const float *in, int n_rows, int ld, int cols, float *out);
cudaError_t launch_grad_reduce(GradReduceArgs &a, cudaStream_t stream);

// Output gradients of up to two nets: bf16 rows padded to ld (64 or 128) columns, and column sums of every 128 rows.
struct OutGrad {
    const float *d_out;                                    // [M][cols]
    uint16_t *dz;                                          // [M][ld]
    float *partial;                                        // [ceil(M / 128)][ld]
    int cols, ld;
};
struct OutGradArgs {
    OutGrad net[2];
    int n_nets, M;
    PpoFinish fin;                                         // the loss's sums, by a block of the same launch (fin.partial null: none)
};
cudaError_t launch_out_grads(const OutGradArgs &a, cudaStream_t stream);

// One shuffled minibatch: observation rows as bf16 (zero padded to ld_h), and the other arrays, gathered by idx.
struct GatherArgs {
    const float *obs, *action, *mean, *logp, *advantage, *value, *returns;
    const int32_t *idx;
    long long ld_obs, n_src;
    int M, D, A, ld_h;
    uint16_t *h, *h2;                                      // h2: a second copy, or null
    float *g_action, *g_mean, *g_logp, *g_advantage, *g_value, *g_returns;
    uint32_t *status;
};
cudaError_t launch_gather_minibatch(const GatherArgs &a, cudaStream_t stream);

// im_f32_to_bf16_padded with an optional second copy.
im_status f32_to_bf16_padded(const float *in, int64_t ld_in, int rows, int cols, uint16_t *out, uint16_t *out2, int ld_out, cudaStream_t st);

}  // namespace im
