// Policy-side declarations shared by the MLP translation units and the API glue.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/im.h"

struct im_policy {
    im_policy_config cfg;
    cudaStream_t stream;
    int nl;
    bool tensor_path;                 // bf16 tcgen05 chain (else fp32 SIMT layers)
    void *d_W[IM_MAX_LAYERS];         // SIMT path: weights as given ([out][in], float or bf16)
    float *d_b[IM_MAX_LAYERS];
    float *d_act[2];                  // SIMT path: fp32 activations, [max_batch][max hidden]
    int act_ld;
    uint32_t *d_status;
    float *d_log_std;                 // [A] per-dimension ln(sigma) once im_policy_set_log_std has been called, else null
    struct im_policy_tc *tc;          // tensor path state (weights padded for the GEMM tiles, bf16 activations, tensor maps)
};

namespace im {
// Hidden layer: C = relu(A W^T + bias).
cudaError_t launch_linear_simt(const float *A, int lda, const void *W, bool w_bf16, const float *bias, float *C,
                               int ldc, int M, int N, int K, cudaStream_t stream);
// Last layer with the Gaussian head: mean [M][N] and, unless action is null, action [M][N] (and logp [M] unless null).
cudaError_t launch_head_simt(const float *A, int lda, const void *W, bool w_bf16, const float *bias, float *mean, float *action,
                             float *logp, int M, int N, int K, float sigma, const float *log_std, uint64_t seed, uint32_t step,
                             uint32_t env_id_base, cudaStream_t stream);

// Tensor-core path (mlp_tc.cu).
im_status tc_policy_create(im_policy *p, const void *const *W, const float *const *b);
void tc_policy_destroy(im_policy *p);
void tc_policy_layer(im_policy *p, int layer, void **W, int32_t *ld, float **bias);
void *tc_policy_input(im_policy *p, int32_t *ld);     // bf16 [max_batch][ld] staging buffer of the first layer
im_status tc_policy_forward(im_policy *p, uint32_t step, int32_t n, const float *obs, int32_t ld_obs,
                            float *mean_out, float *action_out, float *logp_out, im_policy *src = nullptr);
// Whether an actor's and a critic's forward can run layer by layer in common launches (equal widths but for the last).
bool tc_can_pair_nets(const im_policy *a, const im_policy *c, int n);
im_status tc_policy_value_forward(im_policy *a, im_policy *c, uint32_t step, int32_t n, const float *obs, int32_t ld_obs,
                                  float *mean_out, float *action_out, float *logp_out, float *value_out);
// Operands of a tensor-core product; colsum_partial, mask: its backward epilogue (see GemmParams).
struct GemmOperands {
    const void *A;
    int64_t lda;
    const void *B;
    int64_t ldb;
    void *C;
    int64_t ldc;
    const float *bias;
    const void *mask;
    int64_t ld_mask;
    float *colsum_partial;
    uint2 *bits_out;          // forward: one bit per output, whether it is positive ([N / 64][ld_bits] words), or null
    const uint2 *bits_in;     // backward: those bits in the place of `mask`
    int ld_bits;              // (of both nets)
};
// status2: the second product's status word, or null.
im_status tc_gemm(const GemmOperands &x, const GemmOperands *y, int M, int N, int K, bool relu, int ld_partial, uint32_t *status, uint32_t *status2,
                  cudaStream_t stream);
int tc_tn_slices(int Mo, int No, int c_pitch, int R, int max_slices, int n_sm, int nets);
im_status tc_gemm_tn(const GemmOperands &x, const GemmOperands *y, int R, int Mo, int No, int slices, int c_pitch, uint32_t *status,
                     uint32_t *status2, cudaStream_t stream);
im_status tc_gemm_head(const GemmOperands &x, const GemmOperands *y, int M, int N, int N2, int K, uint32_t *status, uint32_t *status2,
                       cudaStream_t stream);
// bounded-wait diagnostics of the tensor-core GEMM kernels and of the bulk-copy PPO loss kernel (current device)
cudaError_t tc_set_wait_debug(unsigned long long limit_ns, int skip_loads);
cudaError_t ppo_set_wait_debug(unsigned long long limit_ns, int skip_loads);
}  // namespace im
