// fp32 SIMT policy layers and the Gaussian head of the fp32 policy.
//
//   C[m][n] = relu(sum_k A[m][k] W[n][k] + b[n])      fp32 products and sums; W is float or bf16
//
// Used for fp32 policies (a few to a few thousand rows) and as a cross-check of the tensor-core path.
//
// At 64 rows a layer is 24-67 M multiply-adds and 1.5-2 MB of weights: about 2 us of either, so latency and issue
// slots are what bound it.  Both operands lie with the contraction index contiguous, and the tile kernel keeps them
// that way: rows of a k-chunk are copied into shared memory by cp.async, one or two chunks ahead (16-byte copies
// where the rows allow them; a thread's copies are a pointer step apart), padded by four floats so that the 16-byte
// reads of eight consecutive rows hit distinct banks.  The warps of a CTA share one output tile and split every
// chunk's k range between them; their partial tiles are added in warp order at the end (bit-reproducible).  Small
// tiles spread a 64-row layer over the SMs.  Measured (361-1024-512-28, one forward with its noise, CUDA graph):
// 64 rows 17 us, 300 rows 35 us, 2048 rows 128 us against
// 265 us at 64 rows for one 64 x 64 tile per CTA with 16-wide k-steps loaded element by element between barriers
// and a noise kernel of one thread per row.
#include <cuda_bf16.h>

#include <type_traits>

#include "im_internal.h"
#include "im_device.cuh"
#include "mlp.h"

namespace im {

namespace {

// Tile of a CTA: BM x BN outputs, BK-wide k-chunks.  WM x WN warps cover the tile, KW such groups split
// the chunk's k range.  A warp's lanes form an 8 x 4 grid over its (BM / WM) x (BN / WN) part, rows and columns
// interleaved (lane row + 8 i, lane column + 4 j) so that one 16-byte read serves 8 (or 4) distinct rows.
template <int THREADS, int BM_, int BN_, int BK_, int WM_, int WN_, int STAGES>
struct Tile {
    static constexpr int BM = BM_, BN = BN_, BK = BK_, WM = WM_, WN = WN_, kStages = STAGES, kThreads = THREADS;
    static constexpr int KW = kThreads / 32 / (WM * WN);
    static constexpr int TM = BM / WM / 8, TN = BN / WN / 4;
    static constexpr int kUnroll = TM * TN > 16 ? 1 : 2;                // k-steps whose operands are in registers at once
    static constexpr int kMinBlocks = kThreads == 512 ? 1 : 2;          // (two 16 x 16 CTAs per SM need 64 registers: 23.6 us against 21.0 at 64 rows)
    static constexpr int LD = BK + 4;                                   // floats between two rows of a chunk
    static constexpr int kStageFloats = (BM + BN) * LD;
    // Partial tiles (reuse the stages' space), their rows four floats longer than the tile's: a warp's 8 x 4 lanes then write to 32
    // banks.  Unpadded rows put its eight rows into the same four banks, or into eight (forwards of 361-1024-512-28 on 64 / 300 /
    // 2048 rows 18.0 / 41.4 / 141 us; padded 17.2 / 37.4 / 128)
    static constexpr int kRedLd = BN + 4;
    static constexpr int kRedFloats = KW * BM * kRedLd;
    static constexpr size_t kSmem = sizeof(float) * (kStages * kStageFloats > kRedFloats ? kStages * kStageFloats : kRedFloats);
    static_assert(BK % (4 * KW) == 0 && TM >= 1 && TN >= 1, "k range of a warp is whole 16-byte words");
};

__device__ __forceinline__ void cp_async(uint32_t dst, const void *src, int bytes_valid, bool wide)
{
    if (wide) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes_valid) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes_valid) : "memory");
}

enum Source { kNarrow, kWide, kBf16 };       // float rows by 4-byte or 16-byte copies (base and stride multiples of 16 bytes), bf16 rows

// The copies of one operand that a thread makes per k-chunk: column k of the chunk (fixed), rows r, r + step, ...
// Rows past the matrix and columns past K arrive as zeros.
template <int ROWS, int BK, int LD, int THREADS, Source SRC>
struct RowLoader {
    static constexpr int V = SRC == kWide ? 4 : 1, PER_ROW = BK / V, STEP = THREADS / PER_ROW, COUNT = ROWS / STEP;
    static_assert(THREADS % PER_ROW == 0 && ROWS % STEP == 0 && COUNT <= 32, "every thread makes the same number of copies");
    const uint8_t *p;            // first row's element
    size_t row_step;             // bytes between two of the thread's rows
    uint32_t dst, live;          // destination in stage 0, bit i: row i exists
    int left;                    // columns from this thread's on, in the current chunk

    __device__ __forceinline__ RowLoader(const void *src, int ld, int r0, int rows, int K, uint32_t smem)
    {
        constexpr int ESZ = SRC == kBf16 ? 2 : 4;
        const int r = threadIdx.x / PER_ROW, k = (threadIdx.x % PER_ROW) * V;
        live = 0;
#pragma unroll
        for (int i = 0; i < COUNT; ++i) live |= (r0 + r + i * STEP < rows ? 1u : 0u) << i;
        p = static_cast<const uint8_t *>(src) + ((size_t)(live & 1u ? r0 + r : 0) * ld + k) * ESZ;
        row_step = (size_t)STEP * ld * ESZ;
        dst = smem + 4u * (uint32_t)(r * LD + k);
        left = K - k;
    }
    __device__ __forceinline__ void issue(uint32_t stage_bytes)
    {
        const int bytes = left >= V ? 4 * V : (left > 0 ? 4 * left : 0);
        const uint8_t *q = p;
#pragma unroll
        for (int i = 0; i < COUNT; ++i, q += row_step) {
            const int n = (live >> i) & 1u ? bytes : 0;
            const uint32_t d = dst + stage_bytes + 4u * (uint32_t)(i * STEP * LD);
            if (SRC == kBf16) {                          // converted on the way, visible after the next barrier
                const float x = n ? __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(q)) : 0.0f;
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(d), "f"(x) : "memory");
            } else {
                cp_async(d, q, n, SRC == kWide);
            }
        }
        p += BK * (SRC == kBf16 ? 2 : 4);
        left -= BK;
    }
};

__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

struct LayerArgs {
    const float *A;
    const void *W;
    const float *bias;
    float *C;
    int lda, ldc, M, N, K;
};

// One BM x BN tile at (m0, n0): leaves its sums in shared memory as KW partial tiles [KW][BM][kRedLd] and meets.
template <class T, Source SA, Source SW>
__device__ __forceinline__ void tile_product(const LayerArgs &L, int m0, int n0, float *smem)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kw = warp / (T::WM * T::WN), wm = (warp / T::WN) % T::WM, wn = warp % T::WN;
    const int lm = lane >> 2, ln = lane & 3;
    const int n_chunks = (L.K + T::BK - 1) / T::BK;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
    RowLoader<T::BM, T::BK, T::LD, T::kThreads, SA> load_a(L.A, L.lda, m0, L.M, L.K, base);
    RowLoader<T::BN, T::BK, T::LD, T::kThreads, SW> load_w(L.W, L.K, n0, L.N, L.K, base + 4u * T::BM * T::LD);
    auto stage_ptr = [&](int s) { return smem + s * T::kStageFloats; };
    auto issue = [&](int c) {
        if (c < n_chunks) {
            const uint32_t off = 4u * (uint32_t)((c % T::kStages) * T::kStageFloats);
            load_a.issue(off);
            load_w.issue(off);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int c = 0; c < T::kStages - 1; ++c) issue(c);
    float acc[T::TM][T::TN] = {};
    for (int c = 0; c < n_chunks; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(T::kStages - 2) : "memory");
        __syncthreads();                     // chunk c is there for everybody, and nobody reads chunk c - 1 any more
        issue(c + T::kStages - 1);
        const float *a = stage_ptr(c % T::kStages) + (wm * (T::BM / T::WM) + lm) * T::LD + kw * (T::BK / T::KW);
        const float *w = stage_ptr(c % T::kStages) + (T::BM + wn * (T::BN / T::WN) + ln) * T::LD + kw * (T::BK / T::KW);
#pragma unroll(T::kUnroll)
        for (int k = 0; k < T::BK / T::KW; k += 4) {
            float4 wv[T::TN];
#pragma unroll
            for (int j = 0; j < T::TN; ++j) wv[j] = lds4(w + 4 * j * T::LD + k);
#pragma unroll
            for (int i = 0; i < T::TM; ++i) {
                const float4 av = lds4(a + 8 * i * T::LD + k);
#pragma unroll
                for (int j = 0; j < T::TN; ++j) {
                    acc[i][j] = fmaf(av.x, wv[j].x, acc[i][j]);
                    acc[i][j] = fmaf(av.y, wv[j].y, acc[i][j]);
                    acc[i][j] = fmaf(av.z, wv[j].z, acc[i][j]);
                    acc[i][j] = fmaf(av.w, wv[j].w, acc[i][j]);
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float *red = smem + kw * (T::BM * T::kRedLd);
#pragma unroll
    for (int i = 0; i < T::TM; ++i)
#pragma unroll
        for (int j = 0; j < T::TN; ++j)
            red[(wm * (T::BM / T::WM) + lm + 8 * i) * T::kRedLd + wn * (T::BN / T::WN) + ln + 4 * j] = acc[i][j];
    __syncthreads();
}
template <class T>
__device__ __forceinline__ float tile_sum(const float *smem, int i)
{
    const float *p = smem + i / T::BN * T::kRedLd + i % T::BN;
    float s = p[0];
#pragma unroll
    for (int q = 1; q < T::KW; ++q) s += p[q * (T::BM * T::kRedLd)];
    return s;
}

template <class T, Source SA, Source SW>
__global__ void __launch_bounds__(T::kThreads, T::kMinBlocks) linear_simt_kernel(const LayerArgs L)
{
    extern __shared__ __align__(16) float smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");       // the rows come from the kernel before, the weights may
    const int m0 = blockIdx.y * T::BM, n0 = blockIdx.x * T::BN;
    tile_product<T, SA, SW>(L, m0, n0, smem);
    for (int i = threadIdx.x; i < T::BM * T::BN; i += T::kThreads) {
        const int m = m0 + i / T::BN, n = n0 + i % T::BN;
        if (m >= L.M || n >= L.N) continue;
        L.C[(size_t)m * L.ldc + n] = fmaxf(tile_sum<T>(smem, i) + L.bias[n], 0.0f);
    }
}

// Last layer: mean = A W^T + b, action = mean + sigma z with z from Philox counter (env id, step, 1, block) and
// Box-Muller (block i feeds outputs 4 i .. 4 i + 3), logp = -0.5 sum z^2 - A ln sigma - (A/2) ln 2 pi.  A cluster
// takes 16 whole rows, each of its CTAs every n-th 32 columns, so that a row's noise and log-probability need no
// second pass: the CTAs' sums of z^2 meet in the first CTA's shared memory and are added in rank order.
struct HeadArgs {
    float *action, *logp;        // action null: the mean only
    float sigma;
    const float *log_std;        // [N] per-column ln(sigma), or null
    uint32_t seed_lo, seed_hi, step, env_id_base;
};
using HeadTile = Tile<512, 16, 32, 256, 1, 1, 2>;

constexpr int kHeadMaxCluster = 8;

template <Source SA, Source SW>
__global__ void __launch_bounds__(HeadTile::kThreads, HeadTile::kMinBlocks) head_simt_kernel(const LayerArgs L, const HeadArgs H)
{
    using T = HeadTile;
    extern __shared__ __align__(16) float smem[];
    __shared__ float s_zz[T::BM][T::BN / 4], s_rank_zz[kHeadMaxCluster][T::BM];
    uint32_t rank, n_ranks;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n_ranks));
    if (n_ranks > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");       // (waited for before the remote store)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int m0 = (int)(blockIdx.x / n_ranks) * T::BM;
    float zz_row = 0.0f, sum_log = 0.0f;                     // thread r < 16: row r
    if (H.logp && threadIdx.x < T::BM) {
        sum_log = (float)L.N * logf(H.sigma);
        if (H.log_std) {
            sum_log = 0.0f;
            for (int i = 0; i < L.N; ++i) sum_log += H.log_std[i];
        }
    }
    for (int n0 = (int)rank * T::BN; n0 < L.N; n0 += (int)n_ranks * T::BN) {
        tile_product<T, SA, SW>(L, m0, n0, smem);
        if (threadIdx.x < T::BM * (T::BN / 4)) {
            const int r = threadIdx.x / (T::BN / 4), q = threadIdx.x % (T::BN / 4);
            const int row = m0 + r, col = n0 + 4 * q;
            float z[4] = {0.0f, 0.0f, 0.0f, 0.0f}, zz = 0.0f;
            if (row < L.M && col < L.N) {
                if (H.action) {
                    const uint4 x = philox4x32_10(make_uint4(H.env_id_base + (uint32_t)row, H.step, IM_STREAM_ACTION, (uint32_t)(col >> 2)),
                                                  make_uint2(H.seed_lo, H.seed_hi));
                    box_muller(x.x, x.y, z[0], z[1]);
                    box_muller(x.z, x.w, z[2], z[3]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (col + i >= L.N) break;
                    const float mu = tile_sum<T>(smem, r * T::BN + 4 * q + i) + L.bias[col + i];
                    L.C[(size_t)row * L.ldc + col + i] = mu;
                    if (H.action) {
                        const float sg = H.log_std ? expf(H.log_std[col + i]) : H.sigma;
                        H.action[(size_t)row * L.N + col + i] = mu + sg * z[i];
                        zz += z[i] * z[i];
                    }
                }
            }
            s_zz[r][q] = zz;
        }
        __syncthreads();                                     // before the next columns reuse the tile's space
        if (threadIdx.x < T::BM)
            for (int q = 0; q < T::BN / 4; ++q) zz_row += s_zz[threadIdx.x][q];
    }
    if (n_ranks > 1) {
        asm volatile("barrier.cluster.wait;" ::: "memory");                // every CTA of the cluster has started
        if (threadIdx.x < T::BM) {
            uint32_t dst;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(&s_rank_zz[rank][threadIdx.x])), "r"(0));
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(zz_row) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        if (rank != 0) return;
        if (threadIdx.x < T::BM) {
            zz_row = 0.0f;
            for (uint32_t r = 0; r < n_ranks; ++r) zz_row += s_rank_zz[r][threadIdx.x];
        }
    }
    if (H.logp && threadIdx.x < T::BM && m0 + (int)threadIdx.x < L.M)
        H.logp[m0 + threadIdx.x] = -0.5f * zz_row - sum_log - 0.5f * (float)L.N * 1.8378770664093453f;
}

bool rows_wide(const void *p, int ld) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && (ld & 3) == 0; }

// Calls f with the sources of A and W as compile-time values.
template <class F>
cudaError_t with_sources(const LayerArgs &L, bool w_bf16, F f)
{
    const bool wa = rows_wide(L.A, L.lda), ww = rows_wide(L.W, L.K);
#define IM_SRC(A, W) f(std::integral_constant<Source, A>(), std::integral_constant<Source, W>())
    if (w_bf16) return wa ? IM_SRC(kWide, kBf16) : IM_SRC(kNarrow, kBf16);
    if (ww) return wa ? IM_SRC(kWide, kWide) : IM_SRC(kNarrow, kWide);
    return wa ? IM_SRC(kWide, kNarrow) : IM_SRC(kNarrow, kNarrow);
#undef IM_SRC
}

template <class T>
cudaError_t launch_tile(const LayerArgs &L, bool w_bf16, cudaStream_t stream)
{
    return with_sources(L, w_bf16, [&](auto sa, auto sw) {
        static DeviceOnce once;
        const auto kernel = linear_simt_kernel<T, decltype(sa)::value, decltype(sw)::value>;
        const cudaError_t e = once.run([&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::kSmem); });
        if (e != cudaSuccess) return e;
        const dim3 grid((L.N + T::BN - 1) / T::BN, (L.M + T::BM - 1) / T::BM);
        return launch_pdl(kernel, grid, dim3(T::kThreads), T::kSmem, stream, 0, L);
    });
}

}  // namespace

cudaError_t launch_linear_simt(const float *A, int lda, const void *W, bool w_bf16, const float *bias, float *C,
                               int ldc, int M, int N, int K, cudaStream_t stream)
{
    const LayerArgs L = {A, W, bias, C, lda, ldc, M, N, K};
    const auto tiles = [&](int bm, int bn) { return (long long)((M + bm - 1) / bm) * ((N + bn - 1) / bn); };
    cudaError_t e;
    // The smallest tile whose CTAs, one per SM with sixteen warps, hold the layer in one wave: a wave's time grows with the
    // tile, a second wave costs more (1024 x 361, us with its head: 64 rows 18.5 as two waves of 16 x 16, 15.0 as one of
    // 32 x 16; 128 rows 19.2 with 32 x 16, 18.2 with 32 x 32.  512 x 1024: 128 rows 19.0 with 16 x 16, 15.6 with 32 x 16; 200
    // rows 23.3 with 32 x 16, 21.6 with 32 x 32).  Whole forwards of 361-1024-512-28 on 129 / 192 / 300 / 416 rows with 32 x 48
    // 31.0 / 30.7 / 41.5 / 42.2 us, 34.0 / 33.8 / 46.6 / 47.1 without it (361-2048-1024-28, 192 rows: 59 and 69; 361-512-256-28, 640
    // rows: 33.3 and 36.2; all of these before the partial tiles were padded).  Beyond that two 32 x 32 CTAs per SM while they are
    // one wave; then 64 x 48 while that is (300 / 700 rows: 37.4 / 65.5 us without, 34.8 / 62.9 with; where one wave of 32 x 32
    // does, at 200 rows, 30.0 and 32.4), 32 x 32 up to four per SM (512 rows: 52 us against 107 with 64 x 64; one wave of 64 x 64
    // with sixteen warps 51 against 45.6), and 64 x 64 (2048 rows, before the padding too: 142 us against 156)
    const int n_sm = device_sm_count();
    if (tiles(16, 16) <= n_sm) e = launch_tile<Tile<512, 16, 16, 256, 1, 1, 3>>(L, w_bf16, stream);
    else if (tiles(32, 16) <= n_sm) e = launch_tile<Tile<512, 32, 16, 128, 1, 1, 3>>(L, w_bf16, stream);
    else if (tiles(32, 32) <= n_sm) e = launch_tile<Tile<512, 32, 32, 128, 1, 1, 3>>(L, w_bf16, stream);
    else if (tiles(32, 48) <= n_sm) e = launch_tile<Tile<512, 32, 48, 128, 1, 1, 3>>(L, w_bf16, stream);
    else if (tiles(32, 32) > 2 * n_sm && tiles(64, 48) <= n_sm) e = launch_tile<Tile<512, 64, 48, 128, 1, 2, 3>>(L, w_bf16, stream);
    else if (tiles(32, 32) <= 4 * n_sm) e = launch_tile<Tile<256, 32, 32, 128, 1, 1, 3>>(L, w_bf16, stream);
    else e = launch_tile<Tile<256, 64, 64, 64, 1, 2, 3>>(L, w_bf16, stream);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_head_simt(const float *A, int lda, const void *W, bool w_bf16, const float *bias, float *mean, float *action,
                             float *logp, int M, int N, int K, float sigma, const float *log_std, uint64_t seed, uint32_t step,
                             uint32_t env_id_base, cudaStream_t stream)
{
    const LayerArgs L = {A, W, bias, mean, lda, N, M, N, K};
    const HeadArgs H = {action, logp, sigma, log_std, (uint32_t)seed, (uint32_t)(seed >> 32), step, env_id_base};
    const int col_tiles = (N + HeadTile::BN - 1) / HeadTile::BN, ranks = col_tiles < kHeadMaxCluster ? col_tiles : kHeadMaxCluster;
    const cudaError_t e = with_sources(L, w_bf16, [&](auto sa, auto sw) {
        static DeviceOnce once;
        const auto kernel = head_simt_kernel<decltype(sa)::value, decltype(sw)::value>;
        const cudaError_t r = once.run([&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)HeadTile::kSmem); });
        if (r != cudaSuccess) return r;
        return launch_pdl(kernel, dim3((M + HeadTile::BM - 1) / HeadTile::BM * ranks), dim3(HeadTile::kThreads), HeadTile::kSmem, stream, ranks, L, H);
    });
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace im
