// Tensor-core policy chain for sm_100a: one persistent, warp-specialised GEMM
// kernel per layer, C[M][N] = act(A[M][K] W[N][K]^T + b), bf16 operands, fp32
// accumulation in tensor memory.
//
//   warp 0      TMA producer: A and W tiles (128B-swizzled, K-major) into a ring of smem stages
//   warp 1      MMA issuer: tcgen05.mma 128 x BLOCK_N x 16 into one of two TMEM accumulators
//   warps 2..   epilogue (four or eight warps; sixteen of the last layer): tcgen05.ld the finished
//               accumulator, add bias, then either ReLU + bf16 store (hidden layers) or the Gaussian
//               head (last layer: mean, Philox/Box-Muller noise, action, log-probability), while the
//               MMA warp works on the next tile
//
// Hidden activations stay bf16 and L2-resident between layers.  Every wait on
// an mbarrier is bounded: when the limit runs out the kernel raises
// IM_DEV_WAIT_TIMEOUT in the status word, stops issuing work, and leaves
// through the common exit that frees its tensor memory.
#include <cmath>
#include <cstring>
#include <type_traits>
#include <cuda.h>
#include <cuda_bf16.h>

#include <new>
#include <vector>

#include "im_internal.h"
#include "im_device.cuh"
#include "mlp.h"

namespace im {

namespace {

constexpr int BLOCK_M = 128;
constexpr int BLOCK_K = 64;               // 64 bf16 = 128 bytes = one swizzle row
constexpr int UMMA_K = 16;
// Epilogues of the hidden-layer kernels: bias and floor; the same and the outputs' signs as bits; backward with the ReLU mask as
// boxes of the forward activations; backward with the mask as bits.  A box costs as much L2 traffic as the output, which these
// products are bound by: a minibatch update with boxes / bits, actor and critic, 16000 rows of 361-1024-512-28 258 / 250 us,
// 131072 rows of 577-1024-1024-512-69 3435 / 3315; on 64-column tiles the two are even (361-320-192-33, 16000 rows 133.3 / 131.1,
// 131072 rows 652 / 658).  (The bits are an epilogue of their own: tested for at run time they cost the policy's products 1 %.)
constexpr int kFwd = 0, kFwdBits = 1, kBwdBoxes = 2, kBwdBits = 3;
constexpr __host__ __device__ bool is_bwd(int epi) { return epi >= kBwdBoxes; }

// Epilogue warps of the hidden-layer kernels: two per tensor-memory lane quadrant, which share the tile's 64-column chunks
// and have one staging slab each (four warps with two slabs against it, in a chain of launches: 8192 x 1024 x 384 10.4 ->
// 9.1 us, 4096 x 2048 x 384 11.2 -> 9.3, 16384 x 1024 x 384 15.9 -> 14.9).  64-column tiles have one chunk and keep four
// warps, as do the backward epilogue of the single-CTA kernel and the M/N-major products, which have neither bias nor floor
// (384 x 2048 over 16 slices of 256 rows: 11.0 us with eight, 10.5 with four).
constexpr __host__ __device__ int hidden_epi_warps(int block_n, bool mn, int epi) { return mn || is_bwd(epi) || block_n == 64 ? 4 : 8; }
constexpr __host__ __device__ int hidden_threads(int block_n, bool mn, int epi) { return 64 + 32 * hidden_epi_warps(block_n, mn, epi); }
// Limit of every bounded wait below (2 s unless im_debug_set_wait changed it), and the diagnostic switch that makes the
// TMA producers issue nothing, so that a test can watch a wait run out with no copy or MMA in flight.
__device__ unsigned long long g_wait_limit_ns = 2000000000ull;
__device__ int g_skip_loads = 0;

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait: false when the limit ran out or another role already gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (int spin = 0;; ++spin) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((spin & 255) == 255) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > g_wait_limit_ns) { *abort_flag = 1; return false; }
        }
    }
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Programmatic dependent launch: a kernel launched with the stream-serialization attribute may start while its
// predecessor in the stream is still running; dep_wait() returns once that predecessor has completed and its
// writes are visible, dep_release() lets the successor's blocks be scheduled as SMs free up.  Both are no-ops
// for a plain launch.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem], single-CTA, bf16 inputs, fp32 accumulate.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrives on the mbarrier once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 32 lanes x 16 consecutive columns of fp32: thread i gets row (lane base + i).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 columns, issue only; pair with tmem_ld_wait() before the values are used.
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, float *v)
{
    uint32_t *r = reinterpret_cast<uint32_t *>(v);
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
}
// 64 columns of 16 lanes, issue only: thread t gets columns 8 j + 2 (t % 4) + {0, 1} of lane t / 4 in v[4 j], v[4 j + 1] and of lane
// t / 4 + 8 in v[4 j + 2], v[4 j + 3].
__device__ __forceinline__ void tmem_ld_16x64_issue(uint32_t taddr, float *v)
{
    uint32_t *r = reinterpret_cast<uint32_t *>(v);
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x8.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major tile of 128-byte rows, 128B swizzle,
// 8-row groups 1024 bytes apart (the layout a SWIZZLE_128B tensor-map load produces).
__device__ __forceinline__ uint64_t smem_desc_k_major_sw128(uint32_t smem_addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);          // start address, 16-byte units
    d |= (uint64_t)0 << 16;                                // leading byte offset: unused for swizzled K-major
    d |= (uint64_t)(1024u >> 4) << 32;                     // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;                                // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                                // SWIZZLE_128B
    return d;
}
// Operand stored with its M (or N) index contiguous: rows of the shared-memory tile are contraction
// (K) steps, each row holding 64 consecutive M/N elements (128 bytes, 128B-swizzled).  Eight K rows
// form a 1024-byte group (stride byte offset); the next block of 64 M/N elements starts
// `mn_block_bytes` further (leading byte offset).
__device__ __forceinline__ uint64_t smem_desc_mn_major_sw128(uint32_t smem_addr, uint32_t mn_block_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((mn_block_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// Instruction descriptor: D fp32, A and B bf16, both K-major, M x N tile.
__host__ __device__ constexpr uint32_t instr_desc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// ... the same with both operands M/N-major (bits 15 and 16).
__host__ __device__ constexpr uint32_t instr_desc_bf16_mn(int M, int N) { return instr_desc_bf16(M, N) | (1u << 15) | (1u << 16); }

struct GemmParams {
    int M;             // rows in use (envs)
    int N;             // valid output columns
    int K_blocks;      // K / 64 (K is padded with zeros)
    int n_tiles_n;     // N tiles of BLOCK_N
    int stages;        // depth of the operand ring in shared memory
    int bufs;          // head: staging buffers
    const float *bias; // [n_tiles_n * BLOCK_N], zero padded
    float act_floor;   // hidden-layer epilogue: out = max(acc + bias, act_floor); 0 is ReLU, -inf no activation
    int n_batches;     // M/N-major products: slices of the contraction, each with its own output; else 1
    int c_batch_rows;  // rows of C between two slices
    // M/N-major products: the contraction's kb_total k-blocks are shared out over the batches ("slices") as evenly as
    // whole k-blocks allow, slice b taking [b kb_total / n_batches, (b + 1) kb_total / n_batches)
    int kb_total;
    // Backward-pass epilogue (kBwdBoxes, kBwdBits): output (r, c) is zeroed where mask[r][c] <= 0 (the ReLU of the
    // forward pass), and the column sums of the masked fp32 values over each 32-row block r / 32 go to
    // colsum_partial[(r / 32) * ld_partial + c] (M a multiple of 32).  Either may be null.
    const __nv_bfloat16 *mask;
    float *colsum_partial;
    int ld_partial;
    // The same mask as one bit per output (sign_bits): the epilogue kFwdBits of the forward product leaves it, kBwdBits of the
    // backward product reads it.  The words of row r and columns 64 c .. 64 c + 63 lie at c * ld_bits + r.
    uint2 *bits_out, *bits_out2;
    const uint2 *bits_in, *bits_in2;
    int ld_bits;
    // Two nets' products of equal sizes in one launch (DUAL instantiations): the first half of the tiles is the first net's,
    // the second half the second's, which has operand, output and mask maps of its own; its head is a value head (no
    // sampling) and may have fewer columns.
    const float *bias2;
    float *colsum_partial2;
    int N2;
    float *mean2;
    // Gaussian head
    float *mean, *action, *logp;
    float sigma;
    const float *log_std;   // [N] per-column ln(sigma), or null: the scalar sigma for every column
    uint32_t seed_lo, seed_hi, step, env_id_base;
    uint32_t *status, *status2;      // status2: of the second net, or null
};

// A wait ran out in this launch: reported to every net that has a part in it.
__device__ __forceinline__ void report_timeout(const GemmParams &P)
{
    atomicOr(P.status, IM_DEV_WAIT_TIMEOUT);
    if (P.status2) atomicOr(P.status2, IM_DEV_WAIT_TIMEOUT);
}

constexpr int kEpiSlabBytes = 32 * 128;    // one epilogue warp's 32 rows x 64 bf16 staging slab

constexpr size_t kSmemLimit = 232448;       // opt-in shared memory per block on this architecture (227 KB)

// KD: k-blocks per stage.  One trip of the producer and of the MMA issuer round the ring costs about 290 cycles besides the
// MMAs (barrier waits, commit; measured without loads and with one MMA per trip), which narrow tiles do not cover with one
// k-block (four 128 x 64 x 16 MMAs: 260 cycles).  Two per stage, in a chain of launches: 1024 x 512 x 1024 7.9 -> 6.8 us,
// 1024 x 1024 x 384 5.1 -> 4.7; a forward of 361-1024-512-28 on 64 rows 17.7 -> 15.6, on 4096 rows 22.3 -> 20.7.
template <int BLOCK_N, int KD = 1>
struct SmemPlan {
    static constexpr int kDepth = KD;
    static constexpr int kABytes = BLOCK_M * BLOCK_K * 2;                    // one k-block
    static constexpr int kBBytes = BLOCK_N * BLOCK_K * 2;
    static constexpr int kBBytesPadded = (kBBytes + 1023) / 1024 * 1024;     // keep every tile 1024-byte aligned
    static constexpr int kStageBytes = KD * (kABytes + kBBytesPadded);      // KD blocks of A, then KD of W
    static constexpr int kBOffset = KD * kABytes;
    static constexpr int kAccStride = BLOCK_N <= 128 ? 128 : 256;           // TMEM columns between the two accumulators
    static constexpr int kTmemCols = 2 * kAccStride;
    static constexpr int kBarBytes = 256;
    static constexpr int kMaxStages = 8;
    // hidden layers: eight staging slabs for the TMA stores, shared out over the epilogue warps (kBwdBoxes: two per warp and two
    // more for the ReLU mask boxes)
    static constexpr __host__ __device__ int hidden_epi_bytes(int epi = kFwd) { return (epi == kBwdBoxes ? 4 * 4 : 8) * kEpiSlabBytes; }
    // head: [2 accumulators][mean, action][128 rows][A] floats laid out as in global memory,
    // partial sums of z^2 [2][4][128], band counters [2][4]
    // (+ bias, per-column sigma and the second net's bias of the tile's columns, 3 x 128 floats)
    // (one buffer where no CTA has a second tile)
    __host__ __device__ static constexpr int head_epi_bytes(int A, int bufs)
    {
        return (bufs * 2 * 128 * A * 4 + 2 * 4 * 128 * 4 + 64 + 3 * 128 * 4 + 1023) / 1024 * 1024;
    }
    __host__ __device__ static constexpr int stages_for(int epi_bytes)
    {
        const int room = (int)kSmemLimit - 1024 - kBarBytes - epi_bytes;
        const int s = room / kStageBytes;
        return s > kMaxStages ? kMaxStages : s;
    }
    __host__ __device__ static constexpr size_t bytes(int stages, int epi_bytes) { return 1024 + (size_t)stages * kStageBytes + epi_bytes + kBarBytes; }
};

// k-blocks of a tile of batch b: first and count.
template <bool MN>
__device__ __forceinline__ void slice_k_blocks(const GemmParams &P, int b, int &kb0, int &n_kb)
{
    if (!MN) { kb0 = 0; n_kb = P.K_blocks; return; }
    // floor(b kb_total / n) in 32 bits: 64-bit divisions cost a short slice a tenth of its time (there is a remainder only for
    // the trainer's slices, 64 at most)
    const uint32_t n = (uint32_t)P.n_batches, q = (uint32_t)P.kb_total / n, r = (uint32_t)P.kb_total % n, u = (uint32_t)b;
    kb0 = (int)(u * q + (r ? u * r / n : 0u));
    n_kb = (int)((u + 1u) * q + (r ? (u + 1u) * r / n : 0u)) - kb0;
}

// Which output tile the number `tile` stands for: net, slice, row and column of tiles.
struct TileAt {
    bool second;
    int slice, m, n;
};
template <bool MN, bool DUAL>
__device__ __forceinline__ TileAt tile_at(const GemmParams &P, int tile, int tiles_per_slice)
{
    const int net_tiles = MN ? tiles_per_slice * P.n_batches : tiles_per_slice;
    const bool second = DUAL && tile >= net_tiles;
    if (second) tile -= net_tiles;
    const int slice = MN ? tile / tiles_per_slice : 0, t = tile - slice * tiles_per_slice, m = t / P.n_tiles_n;
    return {second, slice, m, t - m * P.n_tiles_n};
}

struct Pipe {
    int stages;
    uint8_t *tiles;
    uint64_t *full, *empty, *acc_full, *acc_empty;
    uint32_t *tmem_slot;
    volatile int *abort_flag;
    uint64_t *mask_bar;      // [4 epilogue warps][2]
    uint8_t *epi;
};

template <class Plan>
__device__ __forceinline__ Pipe carve_pipe(uint8_t *smem_raw, int stages, int epi_bytes)
{
    Pipe p;
    p.stages = stages;
    p.tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    p.epi = p.tiles + (size_t)stages * Plan::kStageBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(p.epi + epi_bytes);
    p.full = bars;
    p.empty = bars + Plan::kMaxStages;
    p.acc_full = bars + 2 * Plan::kMaxStages;
    p.acc_empty = bars + 2 * Plan::kMaxStages + 2;
    p.tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * Plan::kMaxStages + 4);
    p.abort_flag = reinterpret_cast<volatile int *>(p.tmem_slot + 1);
    p.mask_bar = bars + 2 * Plan::kMaxStages + 5;
    return p;
}

template <class Plan>
__device__ __forceinline__ void pipe_init(const Pipe &p, int epi_arrivals)
{
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(&p.full[s], 1); mbar_init(&p.empty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&p.acc_full[a], 1); mbar_init(&p.acc_empty[a], epi_arrivals); }
        for (int i = 0; i < 8; ++i) mbar_init(&p.mask_bar[i], 1);
        *p.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if ((threadIdx.x >> 5) == 1) tmem_alloc(p.tmem_slot, Plan::kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}

// Common exit: everyone meets, the allocating warp frees tensor memory.
template <class Plan>
__device__ __forceinline__ void pipe_exit(const Pipe &p, uint32_t tmem_base, const GemmParams &P)
{
    if (*p.abort_flag && (threadIdx.x & 31) == 0) {
        // a wait ran out: give copies and MMAs that are still in flight time to land (bounded)
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) { }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *p.abort_flag) report_timeout(P);
    if ((threadIdx.x >> 5) == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, Plan::kTmemCols);
    }
}

// TMA producer (one thread): A and W tiles of every k-block of every tile of this CTA.
template <class Plan, int BLOCK_N, bool MN = false, bool DUAL = false>
__device__ __forceinline__ void producer_role(const Pipe &p, const CUtensorMap *map_a, const CUtensorMap *map_b,
                                              const GemmParams &P, int n_tiles, int tiles_per_slice,
                                              const CUtensorMap *map_a2 = nullptr, const CUtensorMap *map_b2 = nullptr)
{
    int stage = 0;
    uint32_t phase = 0;
    if (g_skip_loads) return;                        // diagnostic: the consumers' first wait runs out
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const TileAt at = tile_at<MN, DUAL>(P, tile, tiles_per_slice);
        const CUtensorMap *ma = at.second ? map_a2 : map_a, *mb = at.second ? map_b2 : map_b;
        if (MN) {
            // operands are [contraction rows][M or N columns]: a K block is 64 rows, fetched as boxes of 64 columns;
            // batch b is a range of the k-blocks of both operands
            int kb0, n_kb;
            slice_k_blocks<true>(P, at.slice, kb0, n_kb);
            const int mm = at.m * BLOCK_M, nn = at.n * BLOCK_N, r0 = kb0 * BLOCK_K;
            for (int kb = 0; kb < n_kb; ++kb) {
                if (!mbar_wait(&p.empty[stage], phase ^ 1u, p.abort_flag)) return;
                uint8_t *sa = p.tiles + (size_t)stage * Plan::kStageBytes;
                mbar_arrive_expect_tx(&p.full[stage], Plan::kABytes + Plan::kBBytes);
#pragma unroll
                for (int i = 0; i < BLOCK_M / 64; ++i)
                    tma_load_2d(sa + i * 8192, ma, &p.full[stage], mm + 64 * i, r0 + kb * BLOCK_K);
#pragma unroll
                for (int i = 0; i < BLOCK_N / 64; ++i)
                    tma_load_2d(sa + Plan::kABytes + i * 8192, mb, &p.full[stage], nn + 64 * i, r0 + kb * BLOCK_K);
                if (++stage == p.stages) { stage = 0; phase ^= 1u; }
            }
            continue;
        }
        const int m0 = at.m * BLOCK_M, n0 = at.n * BLOCK_N;
        for (int kb = 0; kb < P.K_blocks; kb += Plan::kDepth) {
            if (!mbar_wait(&p.empty[stage], phase ^ 1u, p.abort_flag)) return;
            uint8_t *sa = p.tiles + (size_t)stage * Plan::kStageBytes;
            mbar_arrive_expect_tx(&p.full[stage], Plan::kDepth * (Plan::kABytes + Plan::kBBytes));
#pragma unroll
            for (int d = 0; d < Plan::kDepth; ++d) {                // (a block past K arrives as zeros)
                tma_load_2d(sa + d * Plan::kABytes, ma, &p.full[stage], (kb + d) * BLOCK_K, m0);
                tma_load_2d(sa + Plan::kBOffset + d * Plan::kBBytesPadded, mb, &p.full[stage], (kb + d) * BLOCK_K, n0);
            }
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
    }
}

// MMA issuer (one thread).
template <class Plan, int BLOCK_N, bool MN = false, bool DUAL = false>
__device__ __forceinline__ void mma_role(const Pipe &p, uint32_t tmem_base, const GemmParams &P, int n_tiles, int tiles_per_slice)
{
    constexpr uint32_t idesc = MN ? instr_desc_bf16_mn(BLOCK_M, BLOCK_N) : instr_desc_bf16(BLOCK_M, BLOCK_N);
    int stage = 0, acc = 0;
    uint32_t phase = 0, acc_phase = 0;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        if (!mbar_wait(&p.acc_empty[acc], acc_phase ^ 1u, p.abort_flag)) return;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * Plan::kAccStride);
        int kb0, n_kb;
        slice_k_blocks<MN>(P, MN ? tile_at<MN, DUAL>(P, tile, tiles_per_slice).slice : 0, kb0, n_kb);
        for (int kb = 0; kb < n_kb; kb += Plan::kDepth) {
            if (!mbar_wait(&p.full[stage], phase, p.abort_flag)) return;
            tc_fence_after();
            const uint32_t sa = smem_u32(p.tiles + (size_t)stage * Plan::kStageBytes);
            if (MN) {
                const uint64_t da = smem_desc_mn_major_sw128(sa, 8192u), db = smem_desc_mn_major_sw128(sa + Plan::kABytes, 8192u);
#pragma unroll
                for (int k = 0; k < BLOCK_K / UMMA_K; ++k) {
                    // advancing K by 16 rows = two 1024-byte groups: +128 in 16-byte units
                    umma_bf16(d_tmem, da + (uint64_t)(128 * k), db + (uint64_t)(128 * k), idesc, (kb | k) != 0 ? 1u : 0u);
                }
            } else {
#pragma unroll
                for (int d = 0; d < Plan::kDepth; ++d) {
                    const uint64_t da = smem_desc_k_major_sw128(sa + d * Plan::kABytes);
                    const uint64_t db = smem_desc_k_major_sw128(sa + Plan::kBOffset + d * Plan::kBBytesPadded);
#pragma unroll
                    for (int k = 0; k < BLOCK_K / UMMA_K; ++k) {
                        // advancing K by 16 bf16 = 32 bytes inside the swizzled row: +2 in 16-byte units
                        umma_bf16(d_tmem, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, (kb | d | k) != 0 ? 1u : 0u);
                    }
                }
            }
            umma_commit(&p.empty[stage]);            // smem stage is free once these MMAs have read it
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
        umma_commit(&p.acc_full[acc]);               // accumulator complete
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
}

// Warp reduce-scatter step: every lane holds 2 C values; afterwards C sums over the lane pair (lane, lane ^ offset),
// the lower lane keeping the first C columns and the upper lane the second C.
template <int C>
__device__ __forceinline__ void reduce_scatter_step(float *v, int lane, int offset)
{
    const bool up = (lane & offset) != 0;
#pragma unroll
    for (int i = 0; i < C; ++i) {
        const float keep = up ? v[i + C] : v[i], send = up ? v[i] : v[i + C];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, offset);
    }
}

// ReLU mask of the backward epilogue: each epilogue warp keeps two 32-row x 64-column boxes of the forward
// activations in shared memory (128B-swizzled, like the output slabs), fetched by TMA one chunk ahead.
__device__ __forceinline__ void mask_issue(const CUtensorMap *map_m, uint8_t *slab, uint64_t *bar, int col0, int row0)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // the warp's earlier reads of this slab come first
    mbar_arrive_expect_tx(bar, kEpiSlabBytes);
    tma_load_2d(slab, map_m, bar, col0, row0);
}
__device__ __forceinline__ void mask_read(const uint8_t *slab, int lane, uint4 (&mk)[8])
{
    const uint32_t row = smem_u32(slab) + (uint32_t)lane * 128u;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(mk[c].x), "=r"(mk[c].y), "=r"(mk[c].z), "=r"(mk[c].w)
                     : "r"(row + (uint32_t)((c ^ (lane & 7)) << 4)) : "memory");
}
__device__ __forceinline__ void mask_all_positive(uint4 (&mk)[8])
{
#pragma unroll
    for (int c = 0; c < 8; ++c) mk[c] = make_uint4(0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u);
}

// Which of 64 packed outputs are positive: columns 2 i and 2 i + 1 in bits i and 16 + i, of x for i < 16, of y for the rest.
// The outputs have passed a ReLU, so that none has its sign bit set and a bf16 is positive when it is not zero.
__device__ __forceinline__ uint2 sign_bits(const uint32_t (&pk)[32])
{
    uint2 r = make_uint2(0u, 0u);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        r.x |= ((pk[i] + 0x7fff7fffu) >> (15 - i)) & (0x00010001u << i);
        r.y |= ((pk[i + 16] + 0x7fff7fffu) >> (15 - i)) & (0x00010001u << i);
    }
    return r;
}
// ... of this thread's rows of the band from row0, in the layout of bits_chunk, and the 64 columns from col0 (past the last row: none).
struct BandBits {
    uint2 w[4];
};
__device__ __forceinline__ BandBits load_bits(const GemmParams &P, bool second, int row0, int col0, int lane)
{
    const uint2 *src = (second ? P.bits_in2 : P.bits_in) + (size_t)(col0 >> 6) * P.ld_bits + row0 + (lane >> 2);
    BandBits b;
#pragma unroll
    for (int i = 0; i < 4; ++i) b.w[i] = row0 + (lane >> 2) + 8 * i < P.M ? __ldcg(src + 8 * i) : make_uint2(0u, 0u);
    return b;
}
__device__ __forceinline__ void store_bits(const GemmParams &P, bool second, int row, int col0, const uint32_t (&pk)[32])
{
    const uint2 b = sign_bits(pk);
    if (row < P.M) (second ? P.bits_out2 : P.bits_out)[(size_t)(col0 >> 6) * P.ld_bits + row] = b;
}

// One epilogue chunk of the hidden-layer kernels: 64 accumulator columns of this thread's row -> bias, floor,
// (backward: ReLU mask of the forward activations, column sums over the warp's 32 rows) -> 32 packed bf16 pairs.
template <int EPI>
__device__ __forceinline__ void hidden_chunk(const GemmParams &P, uint32_t t_addr, int row, int col0, int lane,
                                             const uint4 (&mk)[8], uint32_t (&pk)[32], const float *bias, float *colsum)
{
    float v[64];
    tmem_ld32_issue(t_addr, v);
    tmem_ld32_issue(t_addr + 32u, v + 32);
    tmem_ld_wait();
    const float fl = P.act_floor;          // 0: ReLU; -inf: linear output
    if (bias) {
        const float4 *b4 = reinterpret_cast<const float4 *>(bias + col0);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float4 b = b4[i];
            v[4 * i] = fmaxf(v[4 * i] + b.x, fl);
            v[4 * i + 1] = fmaxf(v[4 * i + 1] + b.y, fl);
            v[4 * i + 2] = fmaxf(v[4 * i + 2] + b.z, fl);
            v[4 * i + 3] = fmaxf(v[4 * i + 3] + b.w, fl);
        }
    } else if (fl > -INFINITY) {
#pragma unroll
        for (int i = 0; i < 64; ++i) v[i] = fmaxf(v[i], fl);
    }
    if (EPI == kBwdBoxes) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint32_t w[4] = {mk[c].x, mk[c].y, mk[c].z, mk[c].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // a bf16 is positive when its 16 bits read as a signed integer are
                if ((int)(short)(w[j] & 0xffffu) <= 0) v[8 * c + 2 * j] = 0.0f;
                if ((int)(short)(w[j] >> 16) <= 0) v[8 * c + 2 * j + 1] = 0.0f;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        pk[i] = *reinterpret_cast<const uint32_t *>(&h);
    }
    if (is_bwd(EPI)) {
        if (colsum) {
            reduce_scatter_step<32>(v, lane, 16);
            reduce_scatter_step<16>(v, lane, 8);
            reduce_scatter_step<8>(v, lane, 4);
            reduce_scatter_step<4>(v, lane, 2);
            reduce_scatter_step<2>(v, lane, 1);
            const int row0 = row - lane;                 // lane now holds columns 2 lane, 2 lane + 1 of the 64
            if (row0 < P.M)
                *reinterpret_cast<float2 *>(colsum + (long long)(row0 >> 5) * P.ld_partial + col0 + 2 * lane) =
                    make_float2(v[0], v[1]);
        }
    }
}

// The chunk of the kBwdBits epilogue, from tensor memory to the slab.  A thread has columns 8 j + 2 q + {0, 1} (q = lane % 4) of the
// rows g, g + 8, g + 16, g + 24 (g = lane / 4) of the 32-row band, so that a column's sum needs three exchanges between lanes
// instead of five, and the packed pairs are the fragments that stmatrix takes.  The sums are added in the same order as above: rows
// 16, then 8, 4, 2, 1 apart.  `free` makes sure that the slab may be written.  This epilogue is the longer part of a product with a
// short contraction, and its instructions what bounds it (a row to a thread, as in hidden_chunk: 250 of 430 were the column sums).
// Updates with a row to a thread / this: 8 minibatches of 16000 rows (361-1024-512-28 and -1) 2015 / 1978 us, 131072 rows
// (577-1024-1024-512-69 and -1) 3296 / 3259.
template <typename Free>
__device__ __forceinline__ void bits_chunk(const GemmParams &P, uint32_t t_addr, int row0, int col0, int lane, const BandBits &bits, uint8_t *slab,
                                           float *colsum, Free free)
{
    float v[64];
    tmem_ld_16x64_issue(t_addr, v);
    tmem_ld_16x64_issue(t_addr + (16u << 16), v + 32);
    tmem_ld_wait();
    const int q = lane & 3;
    uint32_t w[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) { w[i][0] = bits.w[i].x >> q; w[i][1] = bits.w[i].y >> q; }
#pragma unroll
    for (int k = 0; k < 64; ++k) {                       // k = 32 h + 4 j + 2 s + c: row 16 h + 8 s + g
        const int j = (k >> 2) & 7, i = 2 * (k >> 5) + ((k >> 1) & 1), c = k & 1;
        if (!(w[i][j >> 2] & (1u << (4 * (j & 3) + 16 * c)))) v[k] = 0.0f;
    }
    uint32_t pk[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
        pk[k] = *reinterpret_cast<const uint32_t *>(&h);
    }
    if (colsum) {
        float sum[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int o = 4 * (k >> 1) + (k & 1);
            sum[k] = (v[o] + v[o + 32]) + (v[o + 2] + v[o + 34]);
        }
        reduce_scatter_step<8>(sum, lane, 16);
        reduce_scatter_step<4>(sum, lane, 8);
        reduce_scatter_step<2>(sum, lane, 4);
        const int j = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
        if (row0 < P.M)
            *reinterpret_cast<float2 *>(colsum + (long long)(row0 >> 5) * P.ld_partial + col0 + 8 * j + 2 * q) = make_float2(sum[0], sum[1]);
    }
    free();
    // 8 x 8 matrices: lane L gives the address of row L % 8 of matrix L / 8 (128B-swizzled rows of 128 bytes)
    const uint32_t at = smem_u32(slab) + (uint32_t)(lane & 7) * 128u + (uint32_t)(((lane >> 3) ^ (lane & 7)) << 4);
#pragma unroll
    for (int i = 0; i < 4; ++i) {                        // rows 8 i ..
#pragma unroll
        for (int jj = 0; jj < 2; ++jj) {
            const uint32_t *f = pk + 16 * (i >> 1) + 8 * jj + (i & 1);
            asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"((at ^ (64u * jj)) + 1024u * i), "r"(f[0]),
                         "r"(f[2]), "r"(f[4]), "r"(f[6]) : "memory");
        }
    }
}

// ------------------------------------------------------------------ hidden layers
// C = relu(A W^T + b) as bf16.  Each epilogue warp owns 32 rows of the tile: it
// reads 64 accumulator columns at a time, applies bias and ReLU, packs to bf16
// into a 128B-swizzled slab in shared memory and hands the slab to a TMA store.
constexpr __host__ __device__ int hidden_depth(int block_n, bool mn, int epi) { return block_n < 256 && !mn && !is_bwd(epi) ? 2 : 1; }

// Kernel parameters of the second net of a DUAL launch (its ReLU mask comes as bits only).
struct NoMaps {};
struct DualMaps {
    CUtensorMap a, b, c;
};
template <bool DUAL>
using SecondNet = std::conditional_t<DUAL, DualMaps, NoMaps>;

template <int BLOCK_N, bool MN = false, int EPI = kFwd, bool DUAL = false>
__global__ void __launch_bounds__(hidden_threads(BLOCK_N, MN, EPI), 1) linear_tc_hidden_kernel(const __grid_constant__ CUtensorMap map_a,
                                                                       const __grid_constant__ CUtensorMap map_b,
                                                                       const __grid_constant__ CUtensorMap map_c,
                                                                       const __grid_constant__ CUtensorMap map_m,
                                                                       const GemmParams P,
                                                                       const __grid_constant__ SecondNet<DUAL> second)
{
    using Plan = SmemPlan<BLOCK_N, hidden_depth(BLOCK_N, MN, EPI)>;
    extern __shared__ uint8_t smem_raw[];
    const Pipe p = carve_pipe<Plan>(smem_raw, P.stages, Plan::hidden_epi_bytes(EPI));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles_per_slice = ((P.M + BLOCK_M - 1) / BLOCK_M) * P.n_tiles_n;
    const int n_tiles = tiles_per_slice * (MN ? P.n_batches : 1) * (DUAL ? 2 : 1);
    const CUtensorMap *map_c2 = &map_c;
    if constexpr (DUAL) map_c2 = &second.c;
    pipe_init<Plan>(p, hidden_epi_warps(BLOCK_N, MN, EPI));
    const uint32_t tmem_base = *p.tmem_slot;
    dep_release();
    dep_wait();                       // nothing before this line touches global memory

    if (warp == 0) {
        if (lane == 0) {
            if constexpr (DUAL) producer_role<Plan, BLOCK_N, MN, true>(p, &map_a, &map_b, P, n_tiles, tiles_per_slice, &second.a, &second.b);
            else producer_role<Plan, BLOCK_N, MN>(p, &map_a, &map_b, P, n_tiles, tiles_per_slice);
        }
    } else if (warp == 1) {
        if (lane == 0) mma_role<Plan, BLOCK_N, MN, DUAL>(p, tmem_base, P, n_tiles, tiles_per_slice);
    } else {
        const int quad = warp & 3;                    // TMEM lanes 32*quad .. 32*quad+31 belong to this warp
        constexpr bool kFour = hidden_epi_warps(BLOCK_N, MN, EPI) == 4;
        constexpr int kSlabs = kFour ? 2 : 1, kStep = kFour ? 64 : 128;
        const int half = kFour ? 0 : (warp - 2) >> 2;                            // first chunk of this warp
        uint8_t *slabs = p.epi + (size_t)(warp - 2) * kSlabs * kEpiSlabBytes;  // two are used alternately
        int which = 0;
        int acc = 0;
        uint32_t acc_phase = 0;
        // kBwdBoxes: the mask box of a chunk is fetched one chunk ahead (across tile boundaries), so its latency
        // hides behind the previous chunk and the wait for the accumulator
        const bool masked = EPI == kBwdBoxes && P.mask != nullptr;
        uint8_t *mslabs = p.epi + (size_t)(4 + warp - 2) * 2 * kEpiSlabBytes;
        uint64_t *mbar = p.mask_bar + (warp - 2) * 2;
        uint32_t ci = 0;                               // chunks consumed by this warp
        bool bail = false;
        uint4 mk[8];
        if (masked && (int)blockIdx.x < n_tiles && lane == 0) {
            const TileAt at = tile_at<MN, DUAL>(P, blockIdx.x, tiles_per_slice);
            mask_issue(&map_m, mslabs, &mbar[0], at.n * BLOCK_N, at.m * BLOCK_M + quad * 32);
        }
        for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
            const TileAt at = tile_at<MN, DUAL>(P, tile, tiles_per_slice);
            const int m0 = at.slice * P.c_batch_rows + at.m * BLOCK_M, n0 = at.n * BLOCK_N;
            BandBits bits_next = {};                                       // (the next chunk's)
            if (EPI == kBwdBits) bits_next = load_bits(P, at.second, m0 + quad * 32, n0, lane);
            bool ready = mbar_wait(&p.acc_full[acc], acc_phase, p.abort_flag);
            if (is_bwd(EPI)) ready = __all_sync(0xffffffffu, ready);           // the column sums shuffle across the whole warp
            if (!ready) break;
            tc_fence_after();
            const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * Plan::kAccStride);
#pragma unroll 1
            for (int c0 = 64 * half; c0 < BLOCK_N; c0 += kStep) {
                uint8_t *slab = slabs + which * kEpiSlabBytes;
                // the last store from this slab must have finished reading shared memory
                const auto slab_free = [&] {
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kSlabs - 1) : "memory");
                    __syncwarp();
                };
                if constexpr (EPI == kBwdBits) {
                    const BandBits bits = bits_next;
                    if (c0 + 64 < BLOCK_N) bits_next = load_bits(P, at.second, m0 + quad * 32, n0 + c0 + 64, lane);
                    bits_chunk(P, t_row + (uint32_t)c0, m0 + quad * 32, n0 + c0, lane, bits, slab, at.second ? P.colsum_partial2 : P.colsum_partial, slab_free);
                } else {
                    uint32_t pk[32];
                    if (EPI == kBwdBoxes) {
                        if (masked) {
                            if (lane == 0) {
                                uint8_t *nslab = mslabs + ((ci + 1u) & 1u) * kEpiSlabBytes;
                                if (c0 + 64 < BLOCK_N) mask_issue(&map_m, nslab, &mbar[(ci + 1u) & 1u], n0 + c0 + 64, m0 + quad * 32);
                                else if (tile + (int)gridDim.x < n_tiles) {
                                    const TileAt next = tile_at<MN, DUAL>(P, tile + (int)gridDim.x, tiles_per_slice);
                                    mask_issue(&map_m, nslab, &mbar[(ci + 1u) & 1u], next.n * BLOCK_N,
                                               next.m * BLOCK_M + quad * 32);
                                }
                            }
                            if (!__all_sync(0xffffffffu, mbar_wait(&mbar[ci & 1u], (ci >> 1) & 1u, p.abort_flag))) { bail = true; break; }
                            mask_read(mslabs + (ci & 1u) * kEpiSlabBytes, lane, mk);
                            ++ci;
                        } else mask_all_positive(mk);
                    }
                    hidden_chunk<EPI>(P, t_row + (uint32_t)c0, m0 + quad * 32 + lane, n0 + c0, lane, mk, pk, at.second ? P.bias2 : P.bias,
                                      at.second ? P.colsum_partial2 : P.colsum_partial);
                    if (EPI == kFwdBits) store_bits(P, at.second, m0 + quad * 32 + lane, n0 + c0, pk);
                    slab_free();
                    const uint32_t slab_row = smem_u32(slab) + (uint32_t)lane * 128u;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const uint32_t dst = slab_row + (uint32_t)((c ^ (lane & 7)) << 4);      // 128B swizzle
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(pk[4 * c]), "r"(pk[4 * c + 1]),
                                     "r"(pk[4 * c + 2]), "r"(pk[4 * c + 3]) : "memory");
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                 ::"l"(at.second ? map_c2 : &map_c), "r"(smem_u32(slab)), "r"(n0 + c0), "r"(m0 + quad * 32) : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                if (kSlabs == 2) which ^= 1;
            }
            if (bail) break;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&p.acc_empty[acc]);
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // stores complete before smem goes away
    }
    pipe_exit<Plan>(p, tmem_base, P);
}

// ------------------------------------------------------------------ hidden layers, CTA pairs
// The single-CTA kernel above is limited by shared-memory bandwidth: per 64-deep k-block the
// tensor core reads A (16 KB) and W (32 KB) while TMA writes as much.  Here two CTAs of a cluster
// (one TPC) compute a 256 x 256 tile together with tcgen05.mma.cta_group::2: each holds its own 128
// rows of A and HALF of the W tile (128 of the 256 output columns' rows), the tensor cores exchange
// the W halves between the two SMs, and each CTA accumulates its 128 rows x 256 columns in its own
// tensor memory.  Per SM that is 32 KB per k-block instead of 48 KB, and a six-deep ring.
//   rank 0 ("leader"): its MMA thread issues for the pair; its full[] barriers collect the
//     transaction bytes of BOTH CTAs' TMA loads; its acc_empty[] barriers collect both epilogues.
//   both ranks: own TMA producer (own A rows, own W half), own epilogue (own accumulator rows),
//     own empty[] / acc_full[] barriers, which the leader's commits reach by multicast.
// No load is multicast; the only multicast is the commit's mbarrier arrive.
constexpr int kPairStages = 6;
constexpr int kPairStageBytes = 2 * BLOCK_M * BLOCK_K * 2;             // A 128x64 + W half 128x64, bf16
constexpr int kPairTmemCols = 512;                                     // two 256-column accumulators
// The backward instantiation (ReLU mask and column sums in the epilogue) runs eight epilogue warps, two per
// tensor-memory lane quadrant, each owning one half of the tile's columns; every warp cycles through a ring of
// three 4 KB slabs, each of which first receives a chunk's mask box and is then overwritten with the chunk's
// output for the TMA store.  The ring takes the room of two operand stages.
// With the mask as bits the slabs only hold output, one per warp.
constexpr int kPairEpiWarpsBwd = 8;
constexpr int kPairRing = 3;
constexpr __host__ __device__ int pair_epi_warps(int epi) { return is_bwd(epi) ? kPairEpiWarpsBwd : 4; }
constexpr __host__ __device__ int pair_threads(int bwd) { return 64 + 32 * pair_epi_warps(bwd); }
constexpr __host__ __device__ int pair_stages(int bwd) { return bwd == kBwdBoxes ? kPairStages - 2 : kPairStages; }
constexpr __host__ __device__ int pair_epi_bytes(int bwd)
{
    return bwd == kBwdBoxes ? kPairEpiWarpsBwd * kPairRing * kEpiSlabBytes : 8 * kEpiSlabBytes;
}
constexpr size_t pair_smem_bytes(int bwd) { return 1024 + (size_t)pair_stages(bwd) * kPairStageBytes + pair_epi_bytes(bwd) + 512; }
static_assert(pair_smem_bytes(kBwdBoxes) <= kSmemLimit && pair_smem_bytes(kFwd) <= kSmemLimit, "shared memory plan of the pair kernel");
static_assert((2 * kPairStages + 5 + kPairEpiWarpsBwd * kPairRing) * 8 <= 512, "barrier area of the pair kernel");

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Address of the same shared-memory offset in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t smem_addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Tensor memory of a CTA pair: one warp of EACH CTA issues the allocation, both get the same base.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t *dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// TMA load into this CTA's shared memory whose completion is signalled on a barrier that may live
// in the peer CTA (cluster address).
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, uint32_t bar_cluster_addr, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(bar_cluster_addr), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrives, once the pair's MMAs so far have completed, on the barrier at this offset in both CTAs.
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar)
{
    const uint16_t both = 3;
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"(both) : "memory");
}

// MN: both operands are stored [contraction rows][M or N columns] (the transposed product of two row-major
// matrices, as in the single-CTA kernel's MN instantiation), possibly over several row slices ("batches").
template <int EPI = kFwd, bool MN = false, bool DUAL = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(pair_threads(EPI), 1)
linear_tc_hidden_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                             const __grid_constant__ CUtensorMap map_c, const __grid_constant__ CUtensorMap map_m,
                             const GemmParams P, const __grid_constant__ SecondNet<DUAL> second)
{
    constexpr int kStages = pair_stages(EPI);
    constexpr int kEpi = pair_epi_warps(EPI);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *epi = tiles + (size_t)kStages * kPairStageBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(epi + pair_epi_bytes(EPI));
    uint64_t *mask_bar = bars + 2 * kPairStages + 5;
    uint64_t *full = bars, *empty = bars + kPairStages, *acc_full = bars + 2 * kPairStages,
             *acc_empty = bars + 2 * kPairStages + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kPairStages + 4);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const int tiles_m = (P.M + 2 * BLOCK_M - 1) / (2 * BLOCK_M);
    const int tiles_per_slice = tiles_m * P.n_tiles_n;               // 256 x 256 tiles
    const int n_tiles = tiles_per_slice * (MN ? P.n_batches : 1) * (DUAL ? 2 : 1);
    const CUtensorMap *map_a2 = &map_a, *map_b2 = &map_b, *map_c2 = &map_c;
    if constexpr (DUAL) { map_a2 = &second.a; map_b2 = &second.b; map_c2 = &second.c; }

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        if (EPI == kBwdBoxes)
            for (int i = 0; i < kPairEpiWarpsBwd * kPairRing; ++i) mbar_init(&mask_bar[i], 1);
        for (int a = 0; a < 2; ++a) { mbar_init(&acc_full[a], 1); mbar_init(&acc_empty[a], 2 * kEpi); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, kPairTmemCols);         // one warp of each CTA, collectively
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                              // both CTAs' barriers exist before anyone signals them
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    dep_release();
    dep_wait();                       // nothing before this line touches global memory
    if (threadIdx.x == 0 && rank == 1) {
        // the pair's MMAs address the accumulator at the same tensor-memory address in both CTAs
        uint32_t leader_base;
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(leader_base) : "r"(map_to_rank(smem_u32(tmem_slot), 0)) : "memory");
        if (leader_base != tmem_base) *abort_flag = 1;
    }
    __syncthreads();

    if (warp == 0) {
        // ---------------- TMA producer (both ranks): own A rows and own half of W, signalled to the leader
        if (lane == 0 && !*abort_flag) {
            int stage = 0;
            uint32_t phase = 0;
            for (int tile = pair; tile < n_tiles; tile += n_pairs) {
                const TileAt at = tile_at<MN, DUAL>(P, tile, tiles_per_slice);
                const CUtensorMap *ma = at.second ? map_a2 : &map_a, *mb = at.second ? map_b2 : &map_b;
                const int m0 = at.m * 2 * BLOCK_M + (int)rank * BLOCK_M;
                const int n0 = at.n * 256 + (int)rank * 128;
                bool ok = true;
                int kb0, n_kb;
                slice_k_blocks<MN>(P, at.slice, kb0, n_kb);
                for (int kb = 0; kb < n_kb; ++kb) {
                    if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag)) { ok = false; break; }
                    uint8_t *sa = tiles + (size_t)stage * kPairStageBytes;
                    const uint32_t leader_full = map_to_rank(smem_u32(&full[stage]), 0);
                    if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * kPairStageBytes);
                    if (MN) {
                        // a K block is 64 rows of the slice; this CTA's 128 M columns and its 128 N columns as 64-column boxes
                        const int r = (kb0 + kb) * BLOCK_K;
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            tma_load_2d_pair(sa + i * 8192, ma, leader_full, m0 + 64 * i, r);
                            tma_load_2d_pair(sa + BLOCK_M * BLOCK_K * 2 + i * 8192, mb, leader_full, n0 + 64 * i, r);
                        }
                    } else {
                        tma_load_2d_pair(sa, ma, leader_full, kb * BLOCK_K, m0);
                        tma_load_2d_pair(sa + BLOCK_M * BLOCK_K * 2, mb, leader_full, kb * BLOCK_K, n0);
                    }
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader only)
        if (lane == 0 && rank == 0 && !*abort_flag) {
            constexpr uint32_t idesc = MN ? instr_desc_bf16_mn(2 * BLOCK_M, 256) : instr_desc_bf16(2 * BLOCK_M, 256);
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int tile = pair; tile < n_tiles && ok; tile += n_pairs) {
                if (!mbar_wait(&acc_empty[acc], acc_phase ^ 1u, abort_flag)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * 256);
                int kb0, n_kb;
                slice_k_blocks<MN>(P, MN ? tile_at<MN, DUAL>(P, tile, tiles_per_slice).slice : 0, kb0, n_kb);
                for (int kb = 0; kb < n_kb; ++kb) {
                    if (!mbar_wait(&full[stage], phase, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(tiles + (size_t)stage * kPairStageBytes);
                    if (MN) {
                        const uint64_t da = smem_desc_mn_major_sw128(sa, 8192u), db = smem_desc_mn_major_sw128(sa + BLOCK_M * BLOCK_K * 2, 8192u);
#pragma unroll
                        for (int k = 0; k < BLOCK_K / UMMA_K; ++k)
                            umma_bf16_pair(d_tmem, da + (uint64_t)(128 * k), db + (uint64_t)(128 * k), idesc, (kb | k) != 0 ? 1u : 0u);
                    } else {
                        const uint64_t da = smem_desc_k_major_sw128(sa), db = smem_desc_k_major_sw128(sa + BLOCK_M * BLOCK_K * 2);
#pragma unroll
                        for (int k = 0; k < BLOCK_K / UMMA_K; ++k)
                            umma_bf16_pair(d_tmem, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, (kb | k) != 0 ? 1u : 0u);
                    }
                    umma_commit_pair(&empty[stage]);          // both CTAs' stages are free once these MMAs have read them
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                umma_commit_pair(&acc_full[acc]);             // both CTAs' accumulators complete
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
    } else {
        // ---------------- epilogue warps (both ranks): own 128 rows x 256 columns
        const int quad = warp & 3;                     // tensor-memory lanes 32 quad .. 32 quad + 31
        int acc = 0;
        uint32_t acc_phase = 0;
        if constexpr (!is_bwd(EPI)) {
            uint8_t *slabs = epi + (size_t)(warp - 2) * 2 * kEpiSlabBytes;
            int which = 0;
            uint4 mk[8];                                // unused without the backward epilogue
            if (!*abort_flag)
            for (int tile = pair; tile < n_tiles; tile += n_pairs) {
                const TileAt at = tile_at<MN, DUAL>(P, tile, tiles_per_slice);
                const int m0 = at.slice * P.c_batch_rows + at.m * 2 * BLOCK_M + (int)rank * BLOCK_M;
                const int n0 = at.n * 256;
                if (!mbar_wait(&acc_full[acc], acc_phase, abort_flag)) break;
                tc_fence_after();
                const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * 256);
#pragma unroll 1
                for (int c0 = 0; c0 < 256; c0 += 64) {
                    uint32_t pk[32];
                    hidden_chunk<kFwd>(P, t_row + (uint32_t)c0, m0 + quad * 32 + lane, n0 + c0, lane, mk, pk,
                                       at.second ? P.bias2 : P.bias, nullptr);
                    if (EPI == kFwdBits) store_bits(P, at.second, m0 + quad * 32 + lane, n0 + c0, pk);
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    __syncwarp();
                    uint8_t *slab = slabs + which * kEpiSlabBytes;
                    const uint32_t slab_row = smem_u32(slab) + (uint32_t)lane * 128u;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const uint32_t dst = slab_row + (uint32_t)((c ^ (lane & 7)) << 4);      // 128B swizzle
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(pk[4 * c]), "r"(pk[4 * c + 1]),
                                     "r"(pk[4 * c + 2]), "r"(pk[4 * c + 3]) : "memory");
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"(at.second ? map_c2 : &map_c), "r"(smem_u32(slab)), "r"(n0 + c0), "r"(m0 + quad * 32) : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                    which ^= 1;
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&acc_empty[acc]), 0));   // the leader's barrier
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        } else if constexpr (EPI == kBwdBits) {
            // warp 2 + e: quadrant (2 + e) & 3, column chunks 2 (e / 4) and 2 (e / 4) + 1 of every tile, through one slab; the
            // mask's words are asked for before the accumulator is waited for
            const int ew = warp - 2, half = ew >> 2;
            uint8_t *slab = epi + (size_t)ew * kEpiSlabBytes;
            if (!*abort_flag)
            for (int tile = pair; tile < n_tiles; tile += n_pairs) {
                const TileAt at = tile_at<MN, DUAL>(P, tile, tiles_per_slice);
                const int row0 = at.m * 2 * BLOCK_M + (int)rank * BLOCK_M + quad * 32, n0 = at.n * 256 + 128 * half;
                BandBits bits = load_bits(P, at.second, row0, n0, lane);
                const BandBits bits1 = load_bits(P, at.second, row0, n0 + 64, lane);
                // (the column sums shuffle across the whole warp: every lane takes the same decision)
                if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], acc_phase, abort_flag))) break;
                tc_fence_after();
                const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * 256 + 128 * half);
#pragma unroll 1
                for (int c0 = 0; c0 < 128; c0 += 64) {
                    bits_chunk(P, t_row + (uint32_t)c0, row0, n0 + c0, lane, bits, slab, at.second ? P.colsum_partial2 : P.colsum_partial, [&] {
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        __syncwarp();
                    });
                    bits = bits1;
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"(at.second ? map_c2 : &map_c), "r"(smem_u32(slab)), "r"(n0 + c0), "r"(row0) : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&acc_empty[acc]), 0));   // the leader's barrier
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        } else {
            // warp 2 + e: quadrant (2 + e) & 3, column chunks 2 (e / 4) and 2 (e / 4) + 1 of every tile.  Chunk j of
            // the warp's sequence uses slab j % 3: mask box in (requested one chunk ahead), output out.
            const int ew = warp - 2, half = ew >> 2;
            uint8_t *ring = epi + (size_t)ew * kPairRing * kEpiSlabBytes;
            uint64_t *mbar = mask_bar + ew * kPairRing;
            const bool masked = P.mask != nullptr;
            uint32_t ci = 0;
            bool bail = false;
            uint4 mk[8];
            auto issue_mask = [&](uint32_t j) {
                const int t2 = pair + (int)(j >> 1) * n_pairs;
                if (t2 >= n_tiles) return;
                const TileAt at = tile_at<MN, DUAL>(P, t2, tiles_per_slice);
                mask_issue(&map_m, ring + (j % kPairRing) * kEpiSlabBytes, &mbar[j % kPairRing],
                           at.n * 256 + (2 * half + (int)(j & 1u)) * 64, at.m * 2 * BLOCK_M + (int)rank * BLOCK_M + quad * 32);
            };
            if (masked && lane == 0 && !*abort_flag) issue_mask(0u);
            if (!*abort_flag)
            for (int tile = pair; tile < n_tiles; tile += n_pairs) {
                const TileAt at = tile_at<MN, DUAL>(P, tile, tiles_per_slice);
                const int m0 = at.m * 2 * BLOCK_M + (int)rank * BLOCK_M;
                const int n0 = at.n * 256;
                // (the column sums shuffle across the whole warp: every lane takes the same decision)
                if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], acc_phase, abort_flag))) break;
                tc_fence_after();
                const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * 256);
#pragma unroll 1
                for (int j = 0; j < 2; ++j) {
                    const int c0 = (2 * half + j) * 64;
                    if (lane == 0) {
                        // slab (ci + 1) % 3 last held chunk ci - 2: its store must have read it before the next box lands
                        asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                        if (masked) issue_mask(ci + 1u);
                    }
                    __syncwarp();
                    uint8_t *slab = ring + (ci % kPairRing) * kEpiSlabBytes;
                    if (masked) {
                        if (!__all_sync(0xffffffffu, mbar_wait(&mbar[ci % kPairRing], (ci / kPairRing) & 1u, abort_flag))) { bail = true; break; }
                        mask_read(slab, lane, mk);
                    } else mask_all_positive(mk);
                    uint32_t pk[32];
                    hidden_chunk<kBwdBoxes>(P, t_row + (uint32_t)c0, m0 + quad * 32 + lane, n0 + c0, lane, mk, pk,
                                            at.second ? P.bias2 : P.bias, at.second ? P.colsum_partial2 : P.colsum_partial);
                    // each lane overwrites the 128 bytes it read its own mask words from
                    const uint32_t slab_row = smem_u32(slab) + (uint32_t)lane * 128u;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const uint32_t dst = slab_row + (uint32_t)((c ^ (lane & 7)) << 4);      // 128B swizzle
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(pk[4 * c]), "r"(pk[4 * c + 1]),
                                     "r"(pk[4 * c + 2]), "r"(pk[4 * c + 3]) : "memory");
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"(at.second ? map_c2 : &map_c), "r"(smem_u32(slab)), "r"(n0 + c0), "r"(m0 + quad * 32) : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                    ++ci;
                }
                if (bail) break;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&acc_empty[acc]), 0));   // the leader's barrier
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    // ---------------- common exit: both CTAs meet (the peer's shared memory and barriers stay alive
    // until the leader is done with them), then each frees its tensor memory
    if (*abort_flag && lane == 0) {
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) { }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (threadIdx.x == 0 && *abort_flag) report_timeout(P);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kPairTmemCols);
    }
}

// ------------------------------------------------------------------ Gaussian head (last layer)
// mean = A W^T + b; action = mean + sigma z with z from Philox counter (env, step, 1, block)
// and Box-Muller; logp = -0.5 sum z^2 - A ln sigma - (A/2) ln 2 pi.  The GEMM is tiny, the
// noise is not: sixteen epilogue warps share the tile, four per group of 16 columns, and draw a
// tile's noise while its operands are on their way (the first tile's even before the previous
// kernel has finished: it depends on nothing in memory).  A finished 32-row band leaves as one
// bulk copy per output.  Against noise drawn after the accumulator and a warp copying the band: a rollout
// step (policy and env) of 4096 envs x 28 actions 46.6 -> 45.2 us, of 16384 envs 74.2 -> 73.1 us.
constexpr int kHeadEpiWarps = 16;
constexpr int kHeadThreads = 64 + 32 * kHeadEpiWarps;
constexpr __host__ __device__ int head_depth(int block_n) { return block_n <= 32 ? 2 : 1; }      // (wider: too few stages beside the staging)

// Standard normals of one row for the columns [c0, c0 + 16) and [c0 + 64, c0 + 80) below A.
template <int CHUNKS>
__device__ __forceinline__ float head_noise(const GemmParams &P, int row, int c0, int A, float (&z)[16 * CHUNKS])
{
    float zz = 0.0f;
#pragma unroll
    for (int g = 0; g < 4 * CHUNKS; ++g) {
        const int col = c0 + (g >> 2) * 64 + 4 * (g & 3);
        if (col < A) {
            const uint4 x = philox4x32_10(make_uint4(P.env_id_base + (uint32_t)row, P.step, IM_STREAM_ACTION, (uint32_t)(col >> 2)),
                                          make_uint2(P.seed_lo, P.seed_hi));
            box_muller(x.x, x.y, z[4 * g], z[4 * g + 1]);
            box_muller(x.z, x.w, z[4 * g + 2], z[4 * g + 3]);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (col + i < A) zz += z[4 * g + i] * z[4 * g + i];
        }
    }
    return zz;
}

template <int BLOCK_N, bool DUAL = false>
__global__ void __launch_bounds__(kHeadThreads, 1) linear_tc_head_kernel(const __grid_constant__ CUtensorMap map_a,
                                                                         const __grid_constant__ CUtensorMap map_b,
                                                                         const GemmParams P,
                                                                         const __grid_constant__ SecondNet<DUAL> second)
{
    using Plan = SmemPlan<BLOCK_N, head_depth(BLOCK_N)>;
    extern __shared__ uint8_t smem_raw[];
    const int A = P.N, bufs = P.bufs;
    const Pipe p = carve_pipe<Plan>(smem_raw, P.stages, Plan::head_epi_bytes(A, bufs));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int net_tiles = (P.M + BLOCK_M - 1) / BLOCK_M;           // one N tile holds the whole action row
    const int n_tiles = DUAL ? 2 * net_tiles : net_tiles;
    const int out_floats = 128 * A;                                // (A is the wider of two nets)
    // staging: per accumulator buffer the tile's mean and action rows laid out exactly as in global
    // memory ([128][A], dense), so a 32-row band leaves as one contiguous copy
    float *out_tiles = reinterpret_cast<float *>(p.epi);                            // [bufs][2][128 * A]
    float *zz_part = out_tiles + bufs * 2 * out_floats;                                // [2][4][128]
    int *band_count = reinterpret_cast<int *>(zz_part + 2 * 4 * 128);               // [2][4]
    float *s_bias = reinterpret_cast<float *>(band_count + 16);                     // [128]: bias of the tile's columns
    float *s_sigma = s_bias + 128;                                                  // [128]: standard deviation per column
    float *s_bias2 = s_sigma + 128;                                                 // [128]: bias of the second net
    if (threadIdx.x < 8) band_count[threadIdx.x] = 0;
    pipe_init<Plan>(p, kHeadEpiWarps);
    const uint32_t tmem_base = *p.tmem_slot;

    if (warp == 0) {
        dep_wait();                   // nothing before this line touches global memory
        if (lane == 0) {
            if constexpr (DUAL) producer_role<Plan, BLOCK_N, false, true>(p, &map_a, &map_b, P, n_tiles, net_tiles, &second.a, &second.b);
            else producer_role<Plan, BLOCK_N>(p, &map_a, &map_b, P, n_tiles, net_tiles);
        }
    } else if (warp == 1) {
        dep_wait();
        if (lane == 0) mma_role<Plan, BLOCK_N>(p, tmem_base, P, n_tiles, net_tiles);
    } else {
        const int quad = warp & 3;                                  // 32-row band of the tile (TMEM lane quadrant)
        const int group = (warp - 2) >> 2;                          // 16-column groups group, group+4, ...
        const int row_in_tile = quad * 32 + lane;
        constexpr int kGroups = (BLOCK_N / 16) < 4 ? (BLOCK_N / 16) : 4;
        constexpr int kChunks = (BLOCK_N + 63) / 64;
        const bool sample_1 = P.action != nullptr;                   // a value head reads only the mean
        float z[16 * kChunks], zz = 0.0f;
#pragma unroll
        for (int i = 0; i < 16 * kChunks; ++i) z[i] = 0.0f;
        if (sample_1 && group < kGroups && (!DUAL || (int)blockIdx.x < net_tiles))
            zz = head_noise<kChunks>(P, (int)blockIdx.x * BLOCK_M + row_in_tile, 16 * group, A, z);
        dep_wait();
        // the epilogue reads bias and sigma from shared memory as 16-byte words instead of one global load per output
        if ((int)threadIdx.x - 64 < BLOCK_N) {
            const int cidx = (int)threadIdx.x - 64;
            s_bias[cidx] = P.bias[cidx];
            if (DUAL) s_bias2[cidx] = cidx < P.N2 ? P.bias2[cidx] : 0.0f;
            s_sigma[cidx] = cidx < A ? (P.log_std ? expf(P.log_std[cidx]) : P.sigma) : 0.0f;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kHeadEpiWarps) : "memory");
        float logp_const = 0.0f;
        if (sample_1) {
            float sum_log = (float)A * logf(P.sigma);
            if (P.log_std) {                                         // same order in every thread
                sum_log = 0.0f;
                for (int i = 0; i < A; ++i) sum_log += P.log_std[i];
            }
            logp_const = -sum_log - 0.5f * (float)A * 1.8378770664093453f;
        }
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
            const bool net2 = DUAL && tile >= net_tiles;
            const int m0 = (net2 ? tile - net_tiles : tile) * BLOCK_M, A = net2 ? P.N2 : P.N;
            const bool sample = sample_1 && !net2;
            const float *bias = net2 ? s_bias2 : s_bias;
            if (!mbar_wait(&p.acc_full[acc], acc_phase, p.abort_flag)) break;
            tc_fence_after();
            const int row = m0 + row_in_tile;
            const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * Plan::kAccStride);
            float *s_mean = out_tiles + (size_t)acc * 2 * out_floats;
            float *s_act = s_mean + out_floats;
            if (group < kGroups) {
#pragma unroll
                for (int ch = 0; ch < kChunks; ++ch) {
                    const int c0 = 16 * group + 64 * ch;
                    if (c0 >= A) break;
                    float v[16];
                    tmem_ld16(t_row + (uint32_t)c0, v);
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const int col = c0 + 4 * g;
                        if (col >= A) break;
                        const float4 b4 = *reinterpret_cast<const float4 *>(bias + col);
                        const float4 s4 = *reinterpret_cast<const float4 *>(s_sigma + col);
                        const float bb[4] = {b4.x, b4.y, b4.z, b4.w}, ss[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            if (col + i < A) {
                                const float mu = v[4 * g + i] + bb[i];
                                s_mean[row_in_tile * A + col + i] = mu;
                                if (sample) s_act[row_in_tile * A + col + i] = mu + ss[i] * z[16 * ch + 4 * g + i];
                            }
                        }
                    }
                }
                zz_part[(acc * 4 + group) * 128 + row_in_tile] = zz;
            }
            tc_fence_before();
            // The last of the column-group warps to finish a 32-row band sums that band's partial z^2
            // in group order (so the result does not depend on which warp that is) and sends the
            // band's mean and action rows out.  The accumulator buffer, and with it this staging buffer,
            // is released only when they have been read.
            if (group < kGroups) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // the copy engine reads what was written above
                __threadfence_block();
                __syncwarp();
                int prev = 0;
                if (lane == 0) prev = atomicAdd(&band_count[acc * 4 + quad], 1);
                prev = __shfl_sync(0xffffffffu, prev, 0);
                if (prev == kGroups - 1) {
                    __threadfence_block();
                    if (lane == 0) band_count[acc * 4 + quad] = 0;
                    const int band_row0 = m0 + quad * 32;
                    int rows_valid = P.M - band_row0;
                    rows_valid = rows_valid > 32 ? 32 : rows_valid;
                    if (rows_valid > 0) {
                        const int count = rows_valid * A;                       // floats, contiguous in global
                        const float *src_m = s_mean + quad * 32 * A, *src_a = s_act + quad * 32 * A;
                        float *dst_m = (net2 ? P.mean2 : P.mean) + (size_t)band_row0 * A;
                        float *dst_a = sample ? P.action + (size_t)band_row0 * A : nullptr;
                        // both sides start on a 16-byte boundary: band offsets are multiples of 32 rows
                        const int bulk = count & ~3;
                        if (lane == 0 && bulk > 0) {
                            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst_m), "r"(smem_u32(src_m)), "r"(4 * bulk) : "memory");
                            if (sample)
                                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst_a), "r"(smem_u32(src_a)), "r"(4 * bulk) : "memory");
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        }
                        for (int i = bulk + lane; i < count; i += 32) {         // ragged last band: at most three floats
                            dst_m[i] = src_m[i];
                            if (sample) dst_a[i] = src_a[i];
                        }
                        if (P.logp && !net2 && lane < rows_valid) {
                            float sum = 0.0f;
#pragma unroll
                            for (int g = 0; g < kGroups; ++g) sum += zz_part[(acc * 4 + g) * 128 + row_in_tile];
                            P.logp[row] = -0.5f * sum + logp_const;
                        }
                    }
                }
                // the next tile's noise, while this band leaves and the tile's operands arrive
                if (sample && tile + (int)gridDim.x < net_tiles)
                    zz = head_noise<kChunks>(P, (tile + (int)gridDim.x) * BLOCK_M + row_in_tile, 16 * group, A, z);
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&p.acc_empty[acc]);
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    pipe_exit<Plan>(p, tmem_base, P);
    // Released late: the env step usually comes next, several CTAs to an SM, and an earlier start would pack them onto
    // the SMs that this grid leaves idle
    dep_release();
}

// fp32 observations -> bf16 rows of a padded buffer; columns beyond `cols` are written as zero.
__global__ void obs_to_bf16_kernel(const float *obs, int ld_obs, int cols, __nv_bfloat16 *__restrict__ out,
                                   int ld_out, int n, int early)
{
    if (early) dep_release();
    dep_wait();
    // (in 32 bits: beside the observations that they come from and the hidden layers' buffers, the device's memory holds fewer
    // than 2^32 of these 16-byte chunks)
    const uint32_t chunks = (uint32_t)ld_out / 8u, total = (uint32_t)n * chunks;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int r = (int)(i / chunks), c = (int)(i - (uint32_t)r * chunks) * 8;
        float v[8];
        if (c + 8 <= cols) {
            const float4 a = __ldcg(reinterpret_cast<const float4 *>(obs + (size_t)r * ld_obs + c));
            const float4 b = __ldcg(reinterpret_cast<const float4 *>(obs + (size_t)r * ld_obs + c + 4));
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = (c + k < cols) ? __ldcg(obs + (size_t)r * ld_obs + c + k) : 0.0f;
        }
        uint32_t pk[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
            pk[k] = *reinterpret_cast<const uint32_t *>(&h);
        }
        *reinterpret_cast<uint4 *>(out + (size_t)r * ld_out + c) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// 2-D bf16 tensor map over a row-major [rows][ld] array; box = 64 columns x box_rows, 128B swizzle.
bool make_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {ld * 2};
    const cuuint32_t box[2] = {BLOCK_K, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Columns of a tile: the whole action row for the last layer; else the narrowest of 64, 128, 256 whose tiles still fit
// the SMs in one wave (a lone tile's time is its operand loads and its epilogue, both shorter when it is narrow:
// 1024 x 1024 x 384 in a chain of launches 4.62 us with 64 columns, 5.39 with 128, 6.54 with 256; 2048 rows 6.21 / 5.45 /
// 6.64), and the widest that divides N once there are several waves (4096 rows 9.37 / 7.24 / 6.89, 8192 rows 14.1 / 10.7 / 9.3).
int pick_block_n(int rows, int N, bool last, int n_sm)       // rows: 128-row tiles
{
    if (last) return (N + 15) / 16 * 16;
    int widest = 64;
    for (int bn = 64; bn <= 256 && N % bn == 0; bn *= 2) {
        if (rows * (N / bn) <= n_sm) return bn;
        widest = bn;
    }
    return widest;
}

}  // namespace

struct TcLayer {
    int N, K, Kpad, block_n, n_tiles_n;      // block_n: the widest tile the layer may take
    __nv_bfloat16 *d_W;      // [n_tiles_n * block_n][Kpad], zero padded
    float *d_bias;           // [n_tiles_n * block_n]
    CUtensorMap map_a, map_b, map_c;    // map_c: the hidden-activation buffer this layer stores to
    CUtensorMap map_b2;                 // W in 128-row boxes: one CTA's half of a 256-column tile, or a 128-column tile
    CUtensorMap map_b1;                 // W in 64-row boxes: a 64-column tile
    CUtensorMap map_head[5];            // last layer: W in boxes of 16, 32, .. 80 rows (rows past the layer's read as zeros)
    const CUtensorMap &map_b_head(int block_n) const { return map_head[block_n / 16 - 1]; }
    CUtensorMap map_m;                  // backward epilogue: the forward activations behind the ReLU mask (boxes like map_c)
};

}  // namespace im

struct im_policy_tc {
    std::vector<im::TcLayer> layers;
    __nv_bfloat16 *d_in;          // [max_batch][Kpad0] bf16 observations
    __nv_bfloat16 *d_hidden[2];   // [max_batch][max hidden]
    int ld_in, ld_hidden;
    int n_sm;
};

namespace im {

namespace {

// L2: the second net's layer of a launch for two (DUAL), else null.
template <int BLOCK_N, bool MN, int EPI, bool DUAL>
cudaError_t launch_hidden(const TcLayer &L, const TcLayer *L2, const GemmParams &gp_in, int n_sm, cudaStream_t stream)
{
    using Plan = SmemPlan<BLOCK_N, hidden_depth(BLOCK_N, MN, EPI)>;
    const auto kernel = linear_tc_hidden_kernel<BLOCK_N, MN, EPI, DUAL>;
    static DeviceOnce once;                      // the attribute is per device
    const cudaError_t e = once.run([&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit); });
    if (e != cudaSuccess) return e;
    GemmParams gp = gp_in;
    gp.stages = Plan::stages_for(Plan::hidden_epi_bytes(EPI));
    const size_t smem = Plan::bytes(gp.stages, Plan::hidden_epi_bytes(EPI));
    const int tiles = ((gp.M + BLOCK_M - 1) / BLOCK_M) * gp.n_tiles_n * gp.n_batches * (DUAL ? 2 : 1);
    const int grid = tiles < n_sm ? tiles : n_sm;
    SecondNet<DUAL> second;
    if constexpr (DUAL) second = {L2->map_a, L2->map_b, L2->map_c};
    const cudaError_t le = launch_pdl(kernel, dim3(grid), dim3(hidden_threads(BLOCK_N, MN, EPI)), smem, stream, 0, L.map_a, L.map_b, L.map_c,
                                      L.map_m, gp, second);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return le != cudaSuccess ? le : cudaGetLastError();
}

// The same products on CTA pairs (256-column tiles).
template <int EPI, bool MN, bool DUAL>
cudaError_t launch_hidden_pair(const TcLayer &L, const TcLayer *L2, const GemmParams &gp, int n_sm, cudaStream_t stream)
{
    const auto kernel = linear_tc_hidden_pair_kernel<EPI, MN, DUAL>;
    static DeviceOnce once;                      // the attribute is per device
    const cudaError_t e = once.run([&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pair_smem_bytes(EPI)); });
    if (e != cudaSuccess) return e;
    const int tiles = ((gp.M + 2 * BLOCK_M - 1) / (2 * BLOCK_M)) * gp.n_tiles_n * gp.n_batches * (DUAL ? 2 : 1);
    const int pairs = tiles < n_sm / 2 ? tiles : n_sm / 2;
    SecondNet<DUAL> second;
    if constexpr (DUAL) second = {L2->map_a, MN ? L2->map_b : L2->map_b2, L2->map_c};
    const cudaError_t le = launch_pdl(kernel, dim3(2 * pairs), dim3(pair_threads(EPI)), pair_smem_bytes(EPI), stream, 0, L.map_a,
                                      MN ? L.map_b : L.map_b2, L.map_c, L.map_m, gp, second);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return le != cudaSuccess ? le : cudaGetLastError();
}

template <int BLOCK_N, bool DUAL>
cudaError_t launch_head(const TcLayer &L, const GemmParams &gp_in, int n_sm, const SecondNet<DUAL> &second, cudaStream_t stream)
{
    using Plan = SmemPlan<BLOCK_N, head_depth(BLOCK_N)>;
    const auto kernel = linear_tc_head_kernel<BLOCK_N, DUAL>;
    static DeviceOnce once;                      // the attribute is per device
    const cudaError_t e = once.run([&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit); });
    if (e != cudaSuccess) return e;
    GemmParams gp = gp_in;
    const int tiles = (gp.M + BLOCK_M - 1) / BLOCK_M * (DUAL ? 2 : 1);
    gp.bufs = tiles <= n_sm ? 1 : 2;
    const int epi = Plan::head_epi_bytes(gp.N, gp.bufs);
    gp.stages = Plan::stages_for(epi);
    if (gp.stages < 2) return cudaErrorInvalidValue;
    const size_t smem = Plan::bytes(gp.stages, epi);
    const int grid = tiles < n_sm ? tiles : n_sm;
    const cudaError_t le = launch_pdl(kernel, dim3(grid), dim3(kHeadThreads), smem, stream, 0, L.map_a, L.map_b, gp, second);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return le != cudaSuccess ? le : cudaGetLastError();
}

template <bool DUAL>
cudaError_t dispatch_head(const TcLayer &L, const GemmParams &gp, int n_sm, const SecondNet<DUAL> &second, cudaStream_t stream)
{
    switch (L.block_n) {
    case 16: return launch_head<16, DUAL>(L, gp, n_sm, second, stream);
    case 32: return launch_head<32, DUAL>(L, gp, n_sm, second, stream);
    case 48: return launch_head<48, DUAL>(L, gp, n_sm, second, stream);
    case 64: return launch_head<64, DUAL>(L, gp, n_sm, second, stream);
    case 80: return launch_head<80, DUAL>(L, gp, n_sm, second, stream);
    default: return cudaErrorInvalidValue;
    }
}

template <int EPI, bool DUAL>
cudaError_t dispatch_width(const TcLayer &L, const TcLayer *L2, const GemmParams &gp, int n_sm, bool pairs, cudaStream_t stream)
{
    if (pairs) return launch_hidden_pair<EPI, false, DUAL>(L, L2, gp, n_sm, stream);
    switch (L.block_n) {
    case 256: return launch_hidden<256, false, EPI, DUAL>(L, L2, gp, n_sm, stream);
    case 128: return launch_hidden<128, false, EPI, DUAL>(L, L2, gp, n_sm, stream);
    default: return launch_hidden<64, false, EPI, DUAL>(L, L2, gp, n_sm, stream);
    }
}

// A hidden layer's product, of one net or (DUAL) of two at once.
template <bool DUAL>
cudaError_t dispatch_hidden(const TcLayer &L, const TcLayer *L2, const GemmParams &gp, int n_sm, bool force_pairs, cudaStream_t stream)
{
    // CTA pairs pay off when the main loop is long enough to amortise the cluster set-up and there
    // are at least two waves of 256 x 256 tiles; otherwise the single-CTA kernel's finer tiles
    // balance the machine better (measured: 16384 x 1024 x 384 is 8 % faster single, 16384 x 1024 x 2048
    // 7 % faster paired).  The tiles of both nets count.  Actor and critic, conversion included, with and without
    // pairs: 577-1024-1024-512 on 8000 / 9001 / 10000 / 11000 / 16384 rows 82.8 / 84.2 / 101.0 / 102.8 / 138 us and 82.2 / 84.0 /
    // 103.4 / 105.7 / 149; 361-2048-1024 on 4800 / 9001 / 16384 rows 65.8 / 93.4 / 163 and 68.2 / 99.6 / 172; 361-1024-512 on 16384 rows
    // 69.5 and 73.1
    const int pair_tiles = ((gp.M + 2 * BLOCK_M - 1) / (2 * BLOCK_M)) * gp.n_tiles_n * (DUAL ? 2 : 1);
    const bool bwd = gp.mask || gp.colsum_partial || gp.bits_in;
    // (the backward epilogue is the longer part of a tile when K is short, and the pair kernel runs it on
    // eight warps: it takes those products whenever its tiles fill the machine)
    const bool pairs = L.block_n == 256 && (force_pairs || (pair_tiles >= n_sm && gp.K_blocks >= 8) || (bwd && pair_tiles >= n_sm / 2));
    if (!bwd) return gp.bits_out ? dispatch_width<kFwdBits, DUAL>(L, L2, gp, n_sm, pairs, stream) : dispatch_width<kFwd, DUAL>(L, L2, gp, n_sm, pairs, stream);
    if (gp.bits_in) return dispatch_width<kBwdBits, DUAL>(L, L2, gp, n_sm, pairs, stream);
    if constexpr (DUAL) return cudaErrorInvalidValue;              // (refused by tc_gemm)
    else return dispatch_width<kBwdBoxes, false>(L, L2, gp, n_sm, pairs, stream);
}

// The same with both operands stored [contraction rows][M or N columns].
template <bool DUAL>
cudaError_t dispatch_mn(const TcLayer &L, const TcLayer *L2, const GemmParams &gp, bool pairs, int n_sm, cudaStream_t stream)
{
    if (pairs) return launch_hidden_pair<kFwd, true, DUAL>(L, L2, gp, n_sm, stream);
    switch (L.block_n) {
    case 256: return launch_hidden<256, true, kFwd, DUAL>(L, L2, gp, n_sm, stream);
    case 128: return launch_hidden<128, true, kFwd, DUAL>(L, L2, gp, n_sm, stream);
    default: return launch_hidden<64, true, kFwd, DUAL>(L, L2, gp, n_sm, stream);
    }
}

}  // namespace

im_status tc_policy_create(im_policy *p, const void *const *W, const float *const *b)
{
    const im_policy_config &cfg = p->cfg;
    const int nl = p->nl;
    if (nl < 2) return IM_ERR_UNSUPPORTED;
    for (int l = 1; l < nl; ++l)
        if (cfg.dims[l] % 64) return IM_ERR_UNSUPPORTED;
    if (cfg.dims[nl] > 80) return IM_ERR_UNSUPPORTED;      // staging of the head's output tiles is sized for this
    int dev = 0, cc_major = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&cc_major, cudaDevAttrComputeCapabilityMajor, dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (cc_major != 10 || !encode_tiled_fn()) return IM_ERR_UNSUPPORTED;

    im_policy_tc *tc = new (std::nothrow) im_policy_tc();
    if (!tc) return IM_ERR_ALLOC;
    p->tc = tc;
    tc->n_sm = n_sm;
    tc->d_in = nullptr;
    tc->d_hidden[0] = tc->d_hidden[1] = nullptr;
    tc->layers.resize(nl);
    for (auto &L : tc->layers) { L.d_W = nullptr; L.d_bias = nullptr; }
    const size_t mb = (size_t)cfg.max_batch;
    int max_hidden = 64;
    for (int l = 1; l < nl; ++l) max_hidden = cfg.dims[l] > max_hidden ? cfg.dims[l] : max_hidden;
    tc->ld_in = (cfg.dims[0] + BLOCK_K - 1) / BLOCK_K * BLOCK_K;
    tc->ld_hidden = max_hidden;
    if (cudaMalloc(&tc->d_in, mb * tc->ld_in * 2) != cudaSuccess ||
        cudaMalloc(&tc->d_hidden[0], mb * max_hidden * 2) != cudaSuccess ||
        cudaMalloc(&tc->d_hidden[1], mb * max_hidden * 2) != cudaSuccess)
        return IM_ERR_ALLOC;

    for (int l = 0; l < nl; ++l) {
        TcLayer &L = tc->layers[l];
        const bool last = l == nl - 1;
        L.N = cfg.dims[l + 1];
        L.K = cfg.dims[l];
        L.Kpad = (L.K + BLOCK_K - 1) / BLOCK_K * BLOCK_K;
        L.block_n = pick_block_n(1, L.N, last, 0);          // (no SMs: the widest)
        L.n_tiles_n = (L.N + L.block_n - 1) / L.block_n;
        const size_t rows = (size_t)L.n_tiles_n * L.block_n;
        std::vector<uint16_t> hw(rows * L.Kpad, 0);
        std::vector<float> hb(rows, 0.0f);
        const uint16_t *src = static_cast<const uint16_t *>(W[l]);
        for (int n = 0; n < L.N; ++n) {
            for (int k = 0; k < L.K; ++k) hw[(size_t)n * L.Kpad + k] = src[(size_t)n * L.K + k];
            hb[n] = b[l][n];
        }
        if (cudaMalloc(&L.d_W, hw.size() * 2) != cudaSuccess || cudaMalloc(&L.d_bias, hb.size() * 4) != cudaSuccess)
            return IM_ERR_ALLOC;
        if (cudaMemcpy(L.d_W, hw.data(), hw.size() * 2, cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(L.d_bias, hb.data(), hb.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess)
            return IM_ERR_CUDA;
        const __nv_bfloat16 *a_base = l == 0 ? tc->d_in : tc->d_hidden[(l - 1) & 1];
        const int a_ld = l == 0 ? tc->ld_in : tc->ld_hidden;
        if (!make_map(&L.map_a, a_base, mb, (uint64_t)L.Kpad, (uint64_t)a_ld, BLOCK_M) ||
            !make_map(&L.map_b, L.d_W, rows, (uint64_t)L.Kpad, (uint64_t)L.Kpad, (uint32_t)L.block_n))
            return IM_ERR_CUDA;
        if (!last && (!make_map(&L.map_b1, L.d_W, rows, (uint64_t)L.Kpad, (uint64_t)L.Kpad, 64) ||
                      !make_map(&L.map_b2, L.d_W, rows, (uint64_t)L.Kpad, (uint64_t)L.Kpad, L.block_n >= 128 ? 128 : 64)))
            return IM_ERR_CUDA;
        // hidden layers store 32-row x 64-column slabs of their output buffer
        if (!last && !make_map(&L.map_c, tc->d_hidden[l & 1], mb, rows, (uint64_t)tc->ld_hidden, 32))
            return IM_ERR_CUDA;
        for (int i = 0; last && i < 5; ++i)
            if (!make_map(&L.map_head[i], L.d_W, rows, (uint64_t)L.Kpad, (uint64_t)L.Kpad, 16 * (i + 1))) return IM_ERR_CUDA;
        L.map_m = L.map_c;               // the forward pass has no mask: a valid placeholder
    }
    return IM_OK;
}

void tc_policy_destroy(im_policy *p)
{
    im_policy_tc *tc = p->tc;
    if (!tc) return;
    for (auto &L : tc->layers) { cudaFree(L.d_W); cudaFree(L.d_bias); }
    cudaFree(tc->d_in); cudaFree(tc->d_hidden[0]); cudaFree(tc->d_hidden[1]);
    delete tc;
    p->tc = nullptr;
}

void tc_policy_layer(im_policy *p, int layer, void **W, int32_t *ld, float **bias)
{
    TcLayer &L = p->tc->layers[layer];
    *W = L.d_W;
    *ld = L.Kpad;
    *bias = L.d_bias;
}

void *tc_policy_input(im_policy *p, int32_t *ld)
{
    *ld = p->tc->ld_in;
    return p->tc->d_in;
}

namespace {

GemmParams head_params(const im_policy *p, uint32_t step, int n, float *mean, float *action, float *logp)
{
    const im_policy_config &cfg = p->cfg;
    GemmParams gp;
    std::memset(&gp, 0, sizeof(gp));
    gp.M = n; gp.act_floor = 0.0f; gp.n_batches = 1;
    gp.mean = mean; gp.action = action; gp.logp = logp;
    gp.sigma = cfg.sigma; gp.log_std = p->d_log_std; gp.seed_lo = (uint32_t)cfg.seed; gp.seed_hi = (uint32_t)(cfg.seed >> 32);
    gp.step = step; gp.env_id_base = cfg.env_id_base; gp.status = p->d_status;
    return gp;
}
void set_layer(GemmParams &gp, const TcLayer &L)
{
    gp.N = L.N; gp.K_blocks = L.Kpad / BLOCK_K; gp.n_tiles_n = L.n_tiles_n; gp.bias = L.d_bias;
}
// The layer with the tile width for `rows` row tiles.
TcLayer with_width(const TcLayer &Y, int rows, bool last, int n_sm)
{
    TcLayer L = Y;
    const int bn = pick_block_n(rows, L.N, last, n_sm);
    if (bn < L.block_n) {
        L.map_b = bn == 128 ? L.map_b2 : L.map_b1;
        L.block_n = bn;
        L.n_tiles_n = L.N / bn;
    }
    return L;
}

im_status convert_obs(im_policy *p, int n, const float *obs, int ld_obs)
{
    im_policy_tc *tc = p->tc;
    const long long chunks = (long long)n * (tc->ld_in / 8);
    const int block = 256;
    long long grid = (chunks + block - 1) / block;
    const long long most = (long long)tc->n_sm * 16;
    if (grid > most) grid = most;
    // The first GEMM is let in early while every block of this grid is about to start (64 rows of 361-1024-512-28: 16.8 -> 16.0
    // us a forward, 9001 rows 28.1 -> 27.7); its large CTAs would keep a longer grid's blocks waiting (65536 rows 142 -> 144)
    const dim3 blocks((unsigned)grid), threads(block);
    if (grid < most)
        launch_pdl(obs_to_bf16_kernel, blocks, threads, 0, p->stream, 0, obs, (int)ld_obs, (int)p->cfg.dims[0], tc->d_in, tc->ld_in, n, 1);
    else obs_to_bf16_kernel<<<blocks, threads, 0, p->stream>>>(obs, ld_obs, p->cfg.dims[0], tc->d_in, tc->ld_in, n, 0);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? IM_OK : IM_ERR_CUDA;
}

}  // namespace

// obs == nullptr: the bf16 input buffer has already been filled (by an attached environment); it is
// this policy's own buffer, or that of `src` (same input width), whose rows the first layer then reads.
// action_out == nullptr: no sampling, only the mean is written.
im_status tc_policy_forward(im_policy *p, uint32_t step, int32_t n, const float *obs, int32_t ld_obs,
                            float *mean_out, float *action_out, float *logp_out, im_policy *src)
{
    im_policy_tc *tc = p->tc;
    const im_policy_config &cfg = p->cfg;
    const bool external = !obs && src && src != p;
    if (external && (!src->tc || src->tc->ld_in != tc->ld_in || src->cfg.dims[0] != cfg.dims[0] || src->cfg.max_batch < n))
        return IM_ERR_INVALID_ARG;
    if (obs) {
        const im_status s = convert_obs(p, n, obs, ld_obs);
        if (s != IM_OK) return s;
    }
    GemmParams gp = head_params(p, step, n, mean_out, action_out, logp_out);
    for (int l = 0; l < p->nl; ++l) {
        const bool last = l == p->nl - 1;
        TcLayer L = cfg.impl == 2 ? tc->layers[l] : with_width(tc->layers[l], (n + BLOCK_M - 1) / BLOCK_M, last, tc->n_sm);
        if (l == 0 && external) L.map_a = src->tc->layers[0].map_a;
        set_layer(gp, L);
        const cudaError_t e = last ? dispatch_head<false>(L, gp, tc->n_sm, NoMaps(), p->stream)
                                   : dispatch_hidden<false>(L, nullptr, gp, tc->n_sm, cfg.impl == 2, p->stream);
        if (e != cudaSuccess) return IM_ERR_CUDA;
    }
    return IM_OK;
}

bool tc_can_pair_nets(const im_policy *a, const im_policy *c, int n)
{
    bool same = a->tensor_path && c->tensor_path && a != c && a->stream == c->stream && a->nl == c->nl && a->cfg.impl == 0 && c->cfg.impl == 0 &&
                a->cfg.max_batch >= n && c->cfg.max_batch >= n && a->cfg.dims[a->nl] >= c->cfg.dims[c->nl];
    for (int l = 0; same && l < a->nl; ++l) same = a->cfg.dims[l] == c->cfg.dims[l];
    return same;
}

// Policy and value head on the same observations: the layers of both nets, which have equal widths (tc_can_pair_nets), two by
// two in one launch.  Below some 16,000 rows a layer costs its fixed chain of barriers, loads and stores (about 5 us) rather than its arithmetic, and one
// net's tiles leave SMs idle: both nets in one launch cost hardly more than one.  Actor (361, 1024, 512, 28) and its
// critic, us for n = 64 / 1000 / 4096 / 9001 / 16384: one after the other 30.8 / 32.7 / 40.0 / 51.6 / 81.0, together
// 15.9 / 17.9 / 24.8 / 38.2 / 63.5; (577, 1024, 1024, 512, 69) 33.6 / 36.0 / 44.8 / 61.1 / 94.1 and 17.9 / 20.4 / 29.3 /
// 48.7 / 77.6.
im_status tc_policy_value_forward(im_policy *a, im_policy *c, uint32_t step, int32_t n, const float *obs, int32_t ld_obs,
                                  float *mean_out, float *action_out, float *logp_out, float *value_out)
{
    const int n_sm = a->tc->n_sm, rows = (n + BLOCK_M - 1) / BLOCK_M;
    if (obs) {
        const im_status s = convert_obs(a, n, obs, ld_obs);
        if (s != IM_OK) return s;
    }
    GemmParams gp = head_params(a, step, n, mean_out, action_out, logp_out);
    for (int l = 0; l < a->nl; ++l) {
        const bool last = l == a->nl - 1;
        TcLayer L = with_width(a->tc->layers[l], 2 * rows, last, n_sm), L2 = with_width(c->tc->layers[l], 2 * rows, last, n_sm);
        if (l == 0) L2.map_a = L.map_a;                          // one copy of the observations serves both
        set_layer(gp, L);
        gp.bias2 = L2.d_bias; gp.N2 = L2.N; gp.mean2 = value_out; gp.status2 = c->d_status;
        const cudaError_t e = last ? dispatch_head<true>(L, gp, n_sm, {L2.map_a, L2.map_b_head(L.block_n), L2.map_a}, a->stream)
                                   : dispatch_hidden<true>(L, &L2, gp, n_sm, false, a->stream);
        if (e != cudaSuccess) return IM_ERR_CUDA;
    }
    return IM_OK;
}


cudaError_t tc_set_wait_debug(unsigned long long limit_ns, int skip_loads)
{
    cudaError_t e = cudaMemcpyToSymbol(g_wait_limit_ns, &limit_ns, sizeof(limit_ns));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_skip_loads, &skip_loads, sizeof(skip_loads));
    return e;
}

namespace {

bool layer_of(TcLayer &L, const GemmOperands &o, int M, int N, int K, int block_n)
{
    L.N = N; L.K = K; L.Kpad = K;
    L.block_n = block_n;
    L.n_tiles_n = N / block_n;
    L.d_W = nullptr; L.d_bias = nullptr;
    if (!make_map(&L.map_a, o.A, (uint64_t)M, (uint64_t)K, (uint64_t)o.lda, BLOCK_M) ||
        !make_map(&L.map_b, o.B, (uint64_t)N, (uint64_t)K, (uint64_t)o.ldb, (uint32_t)block_n) ||
        !make_map(&L.map_c, o.C, (uint64_t)M, (uint64_t)N, (uint64_t)o.ldc, 32))
        return false;
    if (block_n == 256 && !make_map(&L.map_b2, o.B, (uint64_t)N, (uint64_t)K, (uint64_t)o.ldb, 128)) return false;
    L.map_m = L.map_c;
    return !o.mask || make_map(&L.map_m, o.mask, (uint64_t)M, (uint64_t)N, (uint64_t)o.ld_mask, 32);
}

}  // namespace

// C[M][N] = act(A[M][K] B[N][K]^T + bias) on the hidden-layer kernels, operands anywhere in device
// memory: the tensor maps are encoded for this call and travel as kernel parameters.  y: a second product of the same
// sizes in the same launch, or null: two forward products (both with bits_out or neither), or two backward products with
// their masks as bits (both with column sums or neither).
im_status tc_gemm(const GemmOperands &x, const GemmOperands *y, int M, int N, int K, bool relu, int ld_partial, uint32_t *status, uint32_t *status2,
                  cudaStream_t stream)
{
    const int n_sm = device_sm_count();          // 0 unless the current device is an sm_100 part
    if (n_sm <= 0 || !encode_tiled_fn()) return IM_ERR_UNSUPPORTED;
    const bool bwd = x.mask || x.colsum_partial || x.bits_in;
    if (y && ((bwd && !x.bits_in) || y->mask || !x.bits_in != !y->bits_in || !x.bits_out != !y->bits_out || !x.colsum_partial != !y->colsum_partial))
        return IM_ERR_INVALID_ARG;
    TcLayer L, L2;
    const int block_n = pick_block_n((M + BLOCK_M - 1) / BLOCK_M * (y ? 2 : 1), N, false, n_sm);
    if (!layer_of(L, x, M, N, K, block_n) || (y && !layer_of(L2, *y, M, N, K, block_n))) return IM_ERR_CUDA;
    GemmParams gp;
    std::memset(&gp, 0, sizeof(gp));
    gp.M = M; gp.N = N; gp.K_blocks = K / BLOCK_K; gp.n_tiles_n = L.n_tiles_n; gp.bias = x.bias;
    gp.act_floor = relu ? 0.0f : -INFINITY;
    gp.n_batches = 1;
    if (bwd) gp.bias = nullptr;     // the backward product has no bias: its epilogue skips the add
    else if (y) gp.bias2 = y->bias;
    gp.mask = static_cast<const __nv_bfloat16 *>(x.mask);
    gp.colsum_partial = x.colsum_partial; gp.ld_partial = ld_partial;
    gp.bits_out = x.bits_out; gp.bits_in = x.bits_in; gp.ld_bits = x.ld_bits;
    if (y) { gp.colsum_partial2 = y->colsum_partial; gp.bits_out2 = y->bits_out; gp.bits_in2 = y->bits_in; }
    gp.status = status; gp.status2 = status2;
    const cudaError_t e = y ? dispatch_hidden<true>(L, &L2, gp, n_sm, false, stream) : dispatch_hidden<false>(L, nullptr, gp, n_sm, false, stream);
    return e == cudaSuccess ? IM_OK : IM_ERR_CUDA;
}

// CTA pairs (256 x 256 tiles, half of the N operand per SM) when the output splits into whole 256-row tiles, the
// slices' pitch keeps those tiles apart and there are tiles for most pairs.
static bool tn_takes_pairs(int Mo, int No, int R, int slices, int c_pitch, int n_sm, int nets)
{
    const int tiles = (Mo / 256) * ((No + 255) / 256) * slices * nets;
    return (No > 256 || No % 256 == 0) && Mo % 256 == 0 && c_pitch % 256 == 0 && tiles >= n_sm / 3 && R / BLOCK_K / slices >= 8;
}

// Row slices of a transposed product (see tc_gemm_tn) on R rows: the count with the least modelled time.  A wave of
// tiles takes 0.32 us per k-block (128 x 256 per SM: 5 ns a row, measured at 1024 x 1024 on 262144 rows) plus 4 us to
// fill, empty and write; every slice writes and the sum over slices reads the output once more in bf16 (1 ps an element).
int tc_tn_slices(int Mo, int No, int c_pitch, int R, int max_slices, int n_sm, int nets)
{
    const int kb = R / BLOCK_K, tiles_n = (No + 255) / 256;
    int best = 1;
    double best_cost = -1.0;
    for (int S = 1; S <= max_slices && S <= kb; ++S) {
        const bool pairs = tn_takes_pairs(Mo, No, R, S, c_pitch, n_sm, nets);
        const long long tiles = (long long)(pairs ? Mo / 256 : (Mo + 127) / 128) * tiles_n * S * nets, slots = pairs ? n_sm / 2 : n_sm;
        const double cost = (double)((tiles + slots - 1) / slots) * (0.32e-6 * (double)((kb + S - 1) / S) + 4e-6) + 1e-12 * (double)S * nets * c_pitch * No;
        if (best_cost < 0.0 || cost < best_cost * (1.0 - 1e-9)) { best = S; best_cost = cost; }
    }
    return best;
}

// C_s[Mo][No] = sum over the rows r of slice s of A[r][0..Mo) (x) B[r][0..No)  (bf16, fp32 accumulation):
// the transposed product A^T B of two row-major matrices over `slices` row ranges of whole 64-row blocks, the partial
// results stacked with a pitch of `c_pitch` rows.  Operands are read M/N-major, so no transposed copy
// of either matrix is needed.
im_status tc_gemm_tn(const GemmOperands &x, const GemmOperands *y, int R, int Mo, int No, int slices, int c_pitch, uint32_t *status,
                     uint32_t *status2, cudaStream_t stream)
{
    const int n_sm = device_sm_count();          // 0 unless the current device is an sm_100 part
    if (n_sm <= 0 || !encode_tiled_fn()) return IM_ERR_UNSUPPORTED;
    // wide outputs take 256-column tiles even when that leaves a ragged last tile (640 columns: three tiles,
    // a sixth of the MMAs wasted, against five 128-column tiles at little more than half the tensor-pipe rate);
    // TMA fills the operand columns past No with zeros and clips the stores
    const int block_n = No > 256 ? 256 : pick_block_n(1, No, false, 0);
    TcLayer L[2];
    for (int i = 0; i < (y ? 2 : 1); ++i) {
        const GemmOperands &o = i ? *y : x;
        L[i].N = No; L[i].K = R; L[i].Kpad = R;
        L[i].block_n = block_n;
        L[i].n_tiles_n = (No + block_n - 1) / block_n;
        L[i].d_W = nullptr; L[i].d_bias = nullptr;
        if (!make_map(&L[i].map_a, o.A, (uint64_t)R, (uint64_t)Mo, (uint64_t)o.lda, 64) ||
            !make_map(&L[i].map_b, o.B, (uint64_t)R, (uint64_t)No, (uint64_t)o.ldb, 64) ||
            !make_map(&L[i].map_c, o.C, (uint64_t)slices * (uint64_t)c_pitch, (uint64_t)No, (uint64_t)o.ldc, 32))
            return IM_ERR_CUDA;
        L[i].map_m = L[i].map_c;
    }
    GemmParams gp;
    std::memset(&gp, 0, sizeof(gp));
    gp.M = Mo; gp.N = No; gp.kb_total = R / BLOCK_K; gp.n_tiles_n = L[0].n_tiles_n; gp.bias = nullptr;    // no bias in this product
    gp.act_floor = -INFINITY;
    gp.n_batches = slices; gp.c_batch_rows = c_pitch;
    gp.status = status; gp.status2 = status2;
    const bool pairs = tn_takes_pairs(Mo, No, R, slices, c_pitch, n_sm, y ? 2 : 1);
    const cudaError_t e = y ? dispatch_mn<true>(L[0], &L[1], gp, pairs, n_sm, stream) : dispatch_mn<false>(L[0], nullptr, gp, pairs, n_sm, stream);
    return e == cudaSuccess ? IM_OK : IM_ERR_CUDA;
}

// mean[M][N] (fp32, dense) = A[M][K] B[N][K]^T + bias on the Gaussian-head kernel without sampling: o.C is the mean.
// B must hold ceil(N / 16) * 16 rows (rows beyond N zero), bias as many floats.  y: a second product in the same launch,
// of N2 <= N columns, or null.
im_status tc_gemm_head(const GemmOperands &x, const GemmOperands *y, int M, int N, int N2, int K, uint32_t *status, uint32_t *status2,
                       cudaStream_t stream)
{
    const int n_sm = device_sm_count();          // 0 unless the current device is an sm_100 part
    if (n_sm <= 0 || !encode_tiled_fn()) return IM_ERR_UNSUPPORTED;
    TcLayer L;
    L.N = N; L.K = K; L.Kpad = K;
    L.block_n = pick_block_n(1, N, true, n_sm);
    L.n_tiles_n = 1;
    L.d_W = nullptr; L.d_bias = nullptr;
    if (!make_map(&L.map_a, x.A, (uint64_t)M, (uint64_t)K, (uint64_t)x.lda, BLOCK_M) ||
        !make_map(&L.map_b, x.B, (uint64_t)L.block_n, (uint64_t)K, (uint64_t)x.ldb, (uint32_t)L.block_n))
        return IM_ERR_CUDA;
    GemmParams gp;
    std::memset(&gp, 0, sizeof(gp));
    gp.M = M; gp.N = N; gp.K_blocks = K / BLOCK_K; gp.n_tiles_n = 1; gp.bias = x.bias;
    gp.mean = static_cast<float *>(x.C); gp.sigma = 1.0f;
    gp.n_batches = 1;
    gp.status = status; gp.status2 = status2;
    if (!y) return dispatch_head<false>(L, gp, n_sm, NoMaps(), stream) == cudaSuccess ? IM_OK : IM_ERR_CUDA;
    DualMaps second;
    if (!make_map(&second.a, y->A, (uint64_t)M, (uint64_t)K, (uint64_t)y->lda, BLOCK_M) ||
        !make_map(&second.b, y->B, (uint64_t)((N2 + 15) / 16 * 16), (uint64_t)K, (uint64_t)y->ldb, (uint32_t)L.block_n))
        return IM_ERR_CUDA;
    second.c = second.a;
    gp.N2 = N2; gp.bias2 = y->bias; gp.mean2 = static_cast<float *>(y->C);
    return dispatch_head<true>(L, gp, n_sm, second, stream) == cudaSuccess ? IM_OK : IM_ERR_CUDA;
}

}  // namespace im
