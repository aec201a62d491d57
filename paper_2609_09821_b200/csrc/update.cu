// Multi-tensor kernels of the update phase (see update.h).
//
// A small minibatch's update is bound by launches: one of 16000 rows of 361-1024-512-28 (and ...-1) took 62 of them, two
// thirds no tensor-core product.  Here each kind of step between the products is one launch over every tensor of both nets
// (22 launches, 14 with the nets' products in common ones), and a thread's loads are issued in batches before anything is
// done with them.  im_ppo_update in a CUDA graph: 231 us; 131072 rows of 577-1024-1024-512-69 2886 us.
#include <cmath>
#include <cuda_bf16.h>

#include "im_internal.h"
#include "update.h"

namespace im {

namespace {

constexpr int kThreads = 256;

// Every kernel here is launched with programmatic stream serialization.
__device__ __forceinline__ void dep_release_wait()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// True in every thread of the block that is the last of the grid to get here; *done is zero again afterwards.
__device__ __forceinline__ bool last_block(int *done, int n_blocks)
{
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1) == n_blocks - 1;
    __syncthreads();
    if (s_last) {
        __threadfence();
        if (threadIdx.x == 0) *done = 0;
    }
    return s_last != 0;
}

// The tensor whose blocks include `block`.  The first blocks lie together: one by one out of the tensors' records they
// cost a constant-cache miss each.
__device__ __forceinline__ int owner(const int *first_block, int n, int block)
{
    int k = 0;
    while (k + 1 < n && block >= first_block[k + 1]) ++k;
    return k;
}

// ---------------------------------------------------------------- Adam
constexpr int kVecElems = 16 * kThreads;                    // elements of a bias tensor per block
constexpr int kAdamBatch = 8;                               // elements of a thread whose loads are in flight together

// N elements `step` apart: all their loads are issued before the first store (the compiler cannot move them there).
template <int N>
__device__ __forceinline__ void adam_update(const im_adam_config &c, const AdamTensor &T, long long i, long long step, const bool (&on)[N],
                                            float lr, float gs, float (&q)[N])
{
    float p[N], g[N], m[N], v[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const long long e = on[k] ? i + k * step : 0;
        p[k] = T.param[e]; g[k] = T.grad[e]; m[k] = T.m[e]; v[k] = T.v[e];
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const float gk = gs * g[k];
        m[k] = fmaf(c.beta1, m[k], (1.0f - c.beta1) * gk);
        v[k] = fmaf(c.beta2, v[k], (1.0f - c.beta2) * gk * gk);
        q[k] = p[k] - lr * (m[k] * T.inv_c1) / (sqrtf(v[k] * T.inv_c2) + c.eps);
        if (on[k]) {
            T.param[i + k * step] = q[k];
            T.m[i + k * step] = m[k];
            T.v[i + k * step] = v[k];
        }
    }
}

// A block takes a 64 x 64 tile of a weight matrix -- rows are read and written as 256-byte runs, the bf16 copy goes out
// the same way and its transpose through shared memory -- or kVecElems elements of a vector.
__global__ void __launch_bounds__(kThreads) adam_multi_kernel(const __grid_constant__ AdamMultiArgs P)
{
    __shared__ __align__(16) __nv_bfloat16 tile[64][66];    // 33-word rows: a column walk spreads over the banks
    dep_release_wait();
    const AdamTensor T = P.t[owner(P.first_block, P.n_tensors, blockIdx.x)];
    const int blk = (int)blockIdx.x - T.first_block;
    const float lr = *P.lr, gs = P.grad_scale ? *P.grad_scale : 1.0f;
    if (!T.wb) {
        const int n = T.rows * T.cols, i0 = blk * kVecElems + threadIdx.x;
        for (int k0 = 0; k0 < kVecElems / kThreads && i0 + k0 * kThreads < n; k0 += kAdamBatch) {
            bool on[kAdamBatch];
            float q[kAdamBatch];
#pragma unroll
            for (int k = 0; k < kAdamBatch; ++k) on[k] = i0 + (k0 + k) * kThreads < n;
            adam_update<kAdamBatch>(P.cfg, T, i0 + k0 * kThreads, kThreads, on, lr, gs, q);
        }
    } else {
        const int tiles_c = (T.cols + 63) >> 6, r0 = (blk / tiles_c) << 6, c0 = (blk % tiles_c) << 6;
        const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
        const bool in_c = c0 + tx < T.cols;
        __nv_bfloat16 *wb = reinterpret_cast<__nv_bfloat16 *>(T.wb);
#pragma unroll 1
        for (int i = ty; i < 64; i += 4 * kAdamBatch) {
            bool on[kAdamBatch];
            float q[kAdamBatch];
#pragma unroll
            for (int k = 0; k < kAdamBatch; ++k) on[k] = in_c && r0 + i + 4 * k < T.rows;
            adam_update<kAdamBatch>(P.cfg, T, (long long)(r0 + i) * T.cols + c0 + tx, 4ll * T.cols, on, lr, gs, q);
#pragma unroll
            for (int k = 0; k < kAdamBatch; ++k) {
                const __nv_bfloat16 h = __float2bfloat16_rn(on[k] ? q[k] : 0.0f);
                if (on[k]) wb[(long long)(r0 + i + 4 * k) * T.ld_wb + c0 + tx] = h;
                tile[i + 4 * k][tx] = h;
            }
        }
        __syncthreads();
        __nv_bfloat16 *wbT = reinterpret_cast<__nv_bfloat16 *>(T.wbT);
        for (int q = threadIdx.x; q < 512; q += kThreads) {
            const int j = q >> 3, ch = (q & 7) << 3;         // output row c0 + j, elements r0 + ch .. + 7 (padding rows: zeros)
            if (c0 + j >= T.cols) continue;
            __align__(16) __nv_bfloat16 e[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) e[k] = tile[ch + k][j];
            *reinterpret_cast<uint4 *>(wbT + (long long)(c0 + j) * T.ld_wbT + r0 + ch) = *reinterpret_cast<const uint4 *>(e);
        }
    }
    if (P.kl && last_block(P.done, P.n_blocks) && threadIdx.x == 0) {       // every block has read the old learning rate
        const float k = *P.kl;
        float x = lr;
        if (k > 2.0f * P.kl_target) x = fmaxf(x / 1.5f, P.lr_min);
        else if (k > 0.0f && k < 0.5f * P.kl_target) x = fminf(x * 1.5f, P.lr_max);
        *P.lr = x;
    }
}

// ---------------------------------------------------------------- gradient tensors and their norm
constexpr int kBatch = 8;                                   // slices whose loads are in flight together
constexpr int kVecCols = 32;                                // columns of a vector per block

__device__ __forceinline__ double block_sum(double x)
{
    __shared__ double s[kThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = x;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) t += s[w];
    __syncthreads();
    return t;
}

// Bound by the latency of its loads: 16-byte words, eight slices in flight (scalar 8-byte words, at most four in flight and
// less at the ends took 42.8 us for the 47 MB of partial products of 361-1024-512-28 and ...-1; now 16.0).
// Sums of squares are taken in fp64 per thread and block, blocks added in a fixed order by the last one: the result does
// not depend on scheduling.
__global__ void __launch_bounds__(kThreads) grad_reduce_kernel(const __grid_constant__ GradReduceArgs P)
{
    dep_release_wait();
    const int block = P.n_blocks - 1 - (int)blockIdx.x;      // (the vectors' long columns first: they would be the tail)
    double sq = 0.0;
    const int first_vector = P.n_vectors > 0 ? P.v_first[0] : P.n_blocks;
    if (block < first_vector) {
        // dW: the row slices' partial products added in order, eight columns a thread
        __shared__ __align__(16) float s_out[kThreads][8];
        const GradMatrix G = P.m[owner(P.m_first, P.n_matrices, block)];
        const int gpr = (G.cols + 7) >> 3, i = (block - G.first_block) * kThreads + (int)threadIdx.x;
        const bool on = i < G.rows * gpr;
        const int r = on ? i / gpr : 0, c = on ? (i - r * gpr) << 3 : 0;
        const uint4 *src = reinterpret_cast<const uint4 *>(G.in + (long long)r * G.ld_in + c);
        const long long stride = G.slice_stride >> 3;
        float a[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
        for (int s = 0; s < G.slices; s += kBatch) {
            uint4 w[kBatch];
#pragma unroll
            for (int k = 0; k < kBatch; ++k) w[k] = s + k < G.slices ? __ldcg(src + (s + k) * stride) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                const uint32_t x[4] = {w[k].x, w[k].y, w[k].z, w[k].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&x[j]));
                    a[2 * j] += f.x;
                    a[2 * j + 1] += f.y;
                }
            }
        }
        const int n = on ? min(G.cols - c, 8) : 0;            // columns of this thread
        const long long o = (long long)r * G.cols + c;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j < n) sq = fma((double)a[j], (double)a[j], sq);
        if ((G.cols & 7) == 0) {
            if (on) {
                *reinterpret_cast<float4 *>(G.out + o) = make_float4(a[0], a[1], a[2], a[3]);
                *reinterpret_cast<float4 *>(G.out + o + 4) = make_float4(a[4], a[5], a[6], a[7]);
            }
        } else {
            // rows that do not start on 32-byte boundaries: the warp's 32 x 8 values leave in the order of memory
            const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
            *reinterpret_cast<float4 *>(s_out[threadIdx.x]) = make_float4(a[0], a[1], a[2], a[3]);
            *reinterpret_cast<float4 *>(s_out[threadIdx.x] + 4) = make_float4(a[4], a[5], a[6], a[7]);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int from = 4 * k + (lane >> 3);
                const long long of = __shfl_sync(0xffffffffu, o, from);
                const int nf = __shfl_sync(0xffffffffu, n, from);
                if ((lane & 7) < nf) G.out[of + (lane & 7)] = s_out[w0 + from][lane & 7];
            }
        }
    } else if (P.n_vectors > 0 && block < P.n_blocks - (P.n_extra > 0 ? 1 : 0)) {
        // db: 32 columns, 32 groups of rows; eight rows are added in fp32 as a tree, everything beyond in fp64 (a fp32 chain
        // would grow with the batch; all of it in fp64 costs a conversion a row, 30 -> 42 us for 4096 rows of 64 columns)
        __shared__ double s_col[32][kVecCols + 1];
        const GradVector G = P.v[owner(P.v_first, P.n_vectors, block)];
        const int cg = threadIdx.x & 7, rg = threadIdx.x >> 3, c = (block - G.first_block) * kVecCols + 4 * cg;
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        if (c < G.ld) {
#pragma unroll 1
            for (int r = rg; r < G.n_rows; r += 8 * 32) {
                float4 x[8];                                  // loads in flight together
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    x[k] = r + 32 * k < G.n_rows ? __ldcg(reinterpret_cast<const float4 *>(G.in + (long long)(r + 32 * k) * G.ld + c))
                                                 : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int k = 4; k > 0; k >>= 1)
#pragma unroll
                    for (int i = 0; i < k; ++i) {
                        x[i].x += x[i + k].x; x[i].y += x[i + k].y; x[i].z += x[i + k].z; x[i].w += x[i + k].w;
                    }
                a[0] += (double)x[0].x; a[1] += (double)x[0].y; a[2] += (double)x[0].z; a[3] += (double)x[0].w;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) s_col[rg][4 * cg + j] = a[j];
        __syncthreads();
        if (threadIdx.x < kVecCols) {
            double t = 0.0;
#pragma unroll 8
            for (int g = 0; g < 32; ++g) t += s_col[g][threadIdx.x];
            const int col = (block - G.first_block) * kVecCols + threadIdx.x;
            if (col < G.cols) {
                const float x = (float)t;
                G.out[col] = x;
                sq = (double)x * (double)x;
            }
        }
    } else {
        for (int i = threadIdx.x; i < P.n_extra; i += kThreads) sq = fma((double)P.extra[i], (double)P.extra[i], sq);
    }
    if (!P.partial) return;
    sq = block_sum(sq);
    if (threadIdx.x == 0) P.partial[block] = sq;
    if (!last_block(P.done, P.n_blocks)) return;
    double t = 0.0;
    for (int i = threadIdx.x; i < P.n_blocks; i += kThreads) t += __ldcg(P.partial + i);
    t = block_sum(t);
    if (threadIdx.x == 0) {
        const double s = (double)P.max_norm / (sqrt(t) + 1e-6);
        P.scale_out[0] = (float)(s < 1.0 ? s : 1.0);
        P.scale_out[1] = (float)sqrt(t);
    }
}

// ---------------------------------------------------------------- output gradients
constexpr int kOutRows = 128;
constexpr int kOutBatch = 16;

// 128 rows of a net to a block; the first block has the loss's sums, which the gradient reduction reads.  The products in between wait
// for this grid, sums and all, so that what is saved is a launch (us per update with one of its own, of 1024 threads / here, 256: 4096
// rows of 361-1024-512-28 and -1 111.8 / 109.0, 131072 1310 / 1303; 131072 rows, 888 partial sums, of 577-1024-512-69 1538 / 1529, -80
// 1551 / 1545).
__global__ void __launch_bounds__(kThreads) out_grads_kernel(const __grid_constant__ OutGradArgs P)
{
    __shared__ float s_sum[8][128];
    dep_release_wait();
    if (P.fin.partial && blockIdx.x == 0) { ppo_finish<kThreads>(P.fin); return; }
    const int block = (int)blockIdx.x - (P.fin.partial ? 1 : 0), row_block = block / P.n_nets;
    const OutGrad &G = P.net[block - row_block * P.n_nets];
    const int lanes = G.ld >> 1, groups = kThreads / lanes;       // a thread owns two columns of every `groups`-th row
    const int c = 2 * ((int)threadIdx.x % lanes), g = (int)threadIdx.x / lanes;
    const int r0 = row_block * kOutRows, r1 = min(r0 + kOutRows, P.M);
    __nv_bfloat16 *dz = reinterpret_cast<__nv_bfloat16 *>(G.dz);
    float s0 = 0.0f, s1 = 0.0f;
#pragma unroll 1
    for (int r = r0 + g; r < r1; r += kOutBatch * groups) {
        float a[kOutBatch], b[kOutBatch];                         // loads in flight together
#pragma unroll
        for (int k = 0; k < kOutBatch; ++k) {
            const bool on = r + k * groups < r1;
            const float *src = G.d_out + (long long)(r + k * groups) * G.cols + c;
            a[k] = on && c < G.cols ? __ldcg(src) : 0.0f;
            b[k] = on && c + 1 < G.cols ? __ldcg(src + 1) : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < kOutBatch; ++k) {
            if (r + k * groups < r1) *reinterpret_cast<__nv_bfloat162 *>(dz + (long long)(r + k * groups) * G.ld + c) = __floats2bfloat162_rn(a[k], b[k]);
            s0 += a[k];
            s1 += b[k];
        }
    }
    s_sum[g][c] = s0;
    s_sum[g][c + 1] = s1;
    __syncthreads();
    if ((int)threadIdx.x < G.ld) {
        float t = 0.0f;
        for (int k = 0; k < groups; ++k) t += s_sum[k][threadIdx.x];
        G.partial[(long long)row_block * G.ld + threadIdx.x] = t;
    }
}

// ---------------------------------------------------------------- shuffled minibatch
constexpr int kRowBatch = 4;

// A warp gathers a row; VEC: observation rows start on 16-byte boundaries.
template <bool VEC>
__global__ void __launch_bounds__(kThreads) gather_minibatch_kernel(const __grid_constant__ GatherArgs P)
{
    dep_release_wait();
    const int lane = threadIdx.x & 31, warps = (gridDim.x * kThreads) >> 5;
    for (int i = (blockIdx.x * kThreads + threadIdx.x) >> 5; i < P.M; i += warps) {
        long long src = P.idx[i];
        if (src < 0 || src >= P.n_src) {                          // a bad index is clamped and reported, never followed
            if (lane == 0) atomicOr(P.status, IM_DEV_BAD_STATE);
            src = src < 0 ? 0 : P.n_src - 1;
        }
        const float *row = P.obs + src * P.ld_obs;
        uint16_t *h = P.h + (long long)i * P.ld_h, *h2 = P.h2 ? P.h2 + (long long)i * P.ld_h : nullptr;
#pragma unroll 1
        for (int c0 = 4 * lane; c0 < P.ld_h; c0 += 128 * kRowBatch) {
            float v[kRowBatch][4];                                // loads in flight together
#pragma unroll
            for (int q = 0; q < kRowBatch; ++q) {
                const int c = c0 + 128 * q;
                if (VEC && c + 4 <= P.D) {
                    const float4 x = __ldcg(reinterpret_cast<const float4 *>(row + c));
                    v[q][0] = x.x; v[q][1] = x.y; v[q][2] = x.z; v[q][3] = x.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[q][j] = c + j < P.D ? __ldcg(row + c + j) : 0.0f;
                }
            }
#pragma unroll
            for (int q = 0; q < kRowBatch; ++q) {
                const int c = c0 + 128 * q;
                const __nv_bfloat162 lo = __floats2bfloat162_rn(v[q][0], v[q][1]), hi = __floats2bfloat162_rn(v[q][2], v[q][3]);
                const uint2 w = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
                if (c < P.ld_h) *reinterpret_cast<uint2 *>(h + c) = w;
                if (h2 && c < P.ld_h) *reinterpret_cast<uint2 *>(h2 + c) = w;
            }
        }
        const long long o = (long long)i * P.A, s = src * P.A;
        const float *from = lane == 0 ? P.logp : lane == 1 ? P.advantage : lane == 2 ? P.value : P.returns;
        float *to = lane == 0 ? P.g_logp : lane == 1 ? P.g_advantage : lane == 2 ? P.g_value : P.g_returns;
        const float scalar = lane < 4 ? __ldcg(from + src) : 0.0f;
#pragma unroll 1
        for (int k0 = lane; k0 < P.A; k0 += 32 * kRowBatch) {
            float a[kRowBatch], m[kRowBatch];
#pragma unroll
            for (int q = 0; q < kRowBatch; ++q) {
                const bool on = k0 + 32 * q < P.A;
                a[q] = on ? __ldcg(P.action + s + k0 + 32 * q) : 0.0f;
                m[q] = on ? __ldcg(P.mean + s + k0 + 32 * q) : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < kRowBatch; ++q) {
                if (k0 + 32 * q >= P.A) break;
                P.g_action[o + k0 + 32 * q] = a[q];
                P.g_mean[o + k0 + 32 * q] = m[q];
            }
        }
        if (lane < 4) to[i] = scalar;
    }
}

}  // namespace

void adam_multi_add(AdamMultiArgs &a, float *param, const float *grad, float *m, float *v, int rows, int cols, uint16_t *wb, int ld_wb,
                    uint16_t *wbT, int ld_wbT, int t)
{
    a.first_block[a.n_tensors] = a.n_blocks;
    AdamTensor &T = a.t[a.n_tensors++];
    T.param = param; T.grad = grad; T.m = m; T.v = v; T.wb = wb; T.wbT = wbT;
    T.rows = rows; T.cols = cols; T.ld_wb = ld_wb; T.ld_wbT = ld_wbT;
    T.inv_c1 = (float)(1.0 / (1.0 - std::pow((double)a.cfg.beta1, (double)t)));
    T.inv_c2 = (float)(1.0 / (1.0 - std::pow((double)a.cfg.beta2, (double)t)));
    T.first_block = a.n_blocks;
    a.n_blocks += wb ? ((rows + 63) / 64) * ((cols + 63) / 64) : (rows * cols + kVecElems - 1) / kVecElems;
}

cudaError_t launch_adam_multi(AdamMultiArgs &a, cudaStream_t stream)
{
    const cudaError_t e = launch_pdl(adam_multi_kernel, dim3((unsigned)a.n_blocks), dim3(kThreads), 0, stream, 0, a);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return e;
}

int grad_matrix_blocks(int rows, int cols) { return (int)(((long long)rows * ((cols + 7) / 8) + kThreads - 1) / kThreads); }
int grad_vector_blocks(int cols) { return (cols + kVecCols - 1) / kVecCols; }

// (all matrices are added before the first vector)
void grad_reduce_add(GradReduceArgs &a, const uint16_t *in, long long slice_stride, int ld_in, int slices, int rows, int cols, float *out)
{
    a.m_first[a.n_matrices] = a.n_blocks;
    a.m[a.n_matrices++] = {in, out, slice_stride, ld_in, slices, rows, cols, a.n_blocks};
    a.n_blocks += grad_matrix_blocks(rows, cols);
}
void grad_reduce_add(GradReduceArgs &a, const float *in, int n_rows, int ld, int cols, float *out)
{
    a.v_first[a.n_vectors] = a.n_blocks;
    a.v[a.n_vectors++] = {in, out, n_rows, ld, cols, a.n_blocks};
    a.n_blocks += grad_vector_blocks(cols);
}

cudaError_t launch_grad_reduce(GradReduceArgs &a, cudaStream_t stream)
{
    if (a.n_extra > 0) a.n_blocks += 1;
    const cudaError_t e = launch_pdl(grad_reduce_kernel, dim3((unsigned)a.n_blocks), dim3(kThreads), 0, stream, 0, a);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return e;
}

cudaError_t launch_out_grads(const OutGradArgs &a, cudaStream_t stream)
{
    const cudaError_t e = launch_pdl(out_grads_kernel, dim3((unsigned)((a.M + kOutRows - 1) / kOutRows * a.n_nets + (a.fin.partial ? 1 : 0))), dim3(kThreads), 0,
                                     stream, 0, a);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return e;
}

cudaError_t launch_gather_minibatch(const GatherArgs &a, cudaStream_t stream)
{
    const bool vec = (reinterpret_cast<uintptr_t>(a.obs) & 15u) == 0 && (a.ld_obs & 3) == 0;
    const int most = device_sm_count() * 16, blocks = (a.M + 7) / 8 < most ? (a.M + 7) / 8 : most;
    const cudaError_t e = launch_pdl(vec ? gather_minibatch_kernel<true> : gather_minibatch_kernel<false>, dim3((unsigned)blocks), dim3(kThreads), 0,
                                     stream, 0, a);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return e;
}

}  // namespace im
