// The sums over the partial rows that the CTAs of the PPO loss leave: d_log_std and the summary.  By one block, of its own after
// im_ppo_loss, or beside the blocks that form the output gradients of an update (update.cu).
#pragma once
#include <cuda_runtime.h>

#include "../../include/im.h"

namespace im {

constexpr int kPpoMaxA = 128;
constexpr int kPpoScalars = 4;               // surrogate, value loss, kl, clip count
constexpr int kPpoPartial = kPpoMaxA + kPpoScalars;
constexpr int kFinishGroups = 32;
constexpr int kFinishBatch = 16;            // partial rows of a group whose loads are in flight together

struct PpoFinish {
    const float *partial;                    // [rows][kPpoPartial], or null: nothing to do
    int rows, A;
    long long M;
    const float *log_std;
    float value_coef, entropy_coef;
    float *d_log_std, *summary;
};

// In fp64: as many interleaved groups of rows as the block has threads for the A + kPpoScalars columns in use, each in order, then
// the groups in order.  One block's time is its chain of loads: 500 rows of A = 28 took 9 to 12 us in four groups of one load at a
// time, 4.8 us with 1024 threads.
template <int THREADS>
__device__ __forceinline__ void ppo_finish(const PpoFinish &F)
{
    __shared__ double s_grp[THREADS];                      // [groups][columns]
    __shared__ double s_tot[kPpoPartial];
    __shared__ double s_H;
    __shared__ float s_ls[kPpoMaxA];
    const int cols = F.A + kPpoScalars, groups = min(THREADS / cols, kFinishGroups);
    const int jj = (int)threadIdx.x % cols, q = (int)threadIdx.x / cols, j = jj < F.A ? jj : kPpoMaxA + jj - F.A;
    if (q < groups) {
        const float *col = F.partial + j;
        double t = 0.0;
        for (int g = q; g < F.rows; g += kFinishBatch * groups) {
            float x[kFinishBatch];                          // loads in flight together, added in order
#pragma unroll
            for (int k = 0; k < kFinishBatch; ++k) x[k] = g + k * groups < F.rows ? __ldcg(col + (size_t)(g + k * groups) * kPpoPartial) : 0.0f;
#pragma unroll
            for (int k = 0; k < kFinishBatch; ++k) t += (double)x[k];
        }
        s_grp[threadIdx.x] = t;
        if (q == groups - 1 && jj < F.A) s_ls[jj] = F.log_std[jj];
    }
    __syncthreads();
    if (q == 0) {
        double t = 0.0;
        for (int k = 0; k < groups; ++k) t += s_grp[k * cols + jj];
        s_tot[j] = t;
        if (jj < F.A) F.d_log_std[jj] = (float)(t - (double)F.entropy_coef);   // the row terms already carry 1/M
    } else if (threadIdx.x == THREADS - 1) {
        double H = 0.0;
        for (int k = 0; k < F.A; ++k) H += (double)s_ls[k] + 0.5 * 2.8378770664093453;   // 1/2 ln(2 pi e)
        s_H = H;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const double M = (double)F.M;
        const double H = s_H;
        const double surr = s_tot[kPpoMaxA + 0] / M, vl = s_tot[kPpoMaxA + 1] / M;
        F.summary[0] = (float)(surr + (double)F.value_coef * vl - (double)F.entropy_coef * H);
        F.summary[1] = (float)surr;
        F.summary[2] = (float)vl;
        F.summary[3] = (float)H;
        F.summary[4] = (float)(s_tot[kPpoMaxA + 2] / M);
        F.summary[5] = (float)(s_tot[kPpoMaxA + 3] / M);
    }
}

// Everything of im_ppo_loss but those sums, which *fin then describes (ppo.cu).
im_status ppo_loss_rows(const im_ppo_config *cfg, int64_t M, int32_t A, const im_ppo_batch *batch, float *d_mean, float *d_log_std,
                        float *d_value, float *summary, void *workspace, void *cuda_stream, PpoFinish *fin);

}  // namespace im
