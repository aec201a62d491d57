// The update phase behind the C ABI (the paper's `update_policy(storage)`, Figure 2): an MLP trainer
// handle (fp32 master weights, Adam state, bf16 working copies, activation and gradient buffers, the
// buffer plan and the row-slice choice of the dW products) and a PPO updater handle that sequences one
// minibatch update of an actor and a critic, or all epochs and minibatches of a collected rollout.
// Host code only: the products and the loss are the kernels that callers reach one by one, the steps between
// them those of update.cu.
#include <cmath>
#include <cstring>
#include <new>

#include "im_internal.h"
#include "mlp.h"
#include "update.h"

namespace {

int pad64(int x) { return (x + 63) / 64 * 64; }
int pad128(int x) { return (x + 127) / 128 * 128; }

// Device array of n elements, zeroed on `st` (the stream everything else of the handle runs on) unless told otherwise.
template <typename T> bool dev_alloc(T **p, size_t n, cudaStream_t st, bool zero = true)
{
    if (cudaMalloc(p, n * sizeof(T)) != cudaSuccess) { *p = nullptr; return false; }
    return !zero || cudaMemsetAsync(*p, 0, n * sizeof(T), st) == cudaSuccess;
}

// The most slices tc_tn_slices takes for a layer on up to max_rows rows.
int max_slices(int Np, int Kp, int max_rows, int max_split)
{
    int most = 1;
    for (int M = 64; M <= max_rows; M += 64) {
        const int S = im::tc_tn_slices(Np, Kp, pad128(Np), M, max_split, im::device_sm_count(), 1);
        most = S > most ? S : most;
        if (most == max_split) break;
    }
    return most;
}

bool adam_ok(const im_adam_config *c)
{
    return c->beta1 >= 0.0f && c->beta1 < 1.0f && c->beta2 >= 0.0f && c->beta2 < 1.0f && c->eps > 0.0f;
}

}  // namespace

struct im_trainer {
    int nl, Mb, t, max_split;
    int s_max[IM_MAX_LAYERS];                              // slices dWs has room for
    int dims[IM_MAX_LAYERS + 1], Kp[IM_MAX_LAYERS], Np[IM_MAX_LAYERS];
    cudaStream_t stream;
    float *W[IM_MAX_LAYERS], *b[IM_MAX_LAYERS], *mW[IM_MAX_LAYERS], *vW[IM_MAX_LAYERS], *mb[IM_MAX_LAYERS], *vb[IM_MAX_LAYERS];
    float *dW[IM_MAX_LAYERS], *db[IM_MAX_LAYERS];
    uint16_t *Wb[IM_MAX_LAYERS], *WbT[IM_MAX_LAYERS];      // bf16 [Np][Kp] and its transpose [Kp][Np]
    uint16_t *H[IM_MAX_LAYERS];                            // H[0]: input rows [Mb][Kp0]; H[l]: activations [Mb][Np[l-1]]
    uint2 *bits[IM_MAX_LAYERS];                            // which of H[l] are positive, a bit each [Kp[l] / 64][Mb]; the update's ReLU mask
    uint16_t *dZ[IM_MAX_LAYERS];                           // gradient at layer l's pre-activation [Mb][Np[l]]
    float *out;                                            // [Mb][dims[nl]]
    uint16_t *dWs[IM_MAX_LAYERS];                          // partial dW products, all row slices
    float *db_partial[IM_MAX_LAYERS];                      // partial column sums of dZ: per 32 rows, last layer per 128 rows; [.][Np]
    uint32_t *status;
};

namespace {

// One net on its input rows x, or two of equal widths (the last but) whose products of a kind share their launches: a
// layer's tiles seldom fill the last wave of SMs, and two nets' dW products need half the row slices each.  An update of an
// actor and a critic (361-1024-512-28 and ...-1) on 16000 rows, im_ppo_update in a CUDA graph: 279 -> 231 us (131072 rows of
// 577-1024-1024-512-69, where every product fills the machine many times over: 2904 -> 2886).
struct Nets {
    im_trainer *a, *c;                                     // c: null for one net
    uint16_t *xa, *xc;                                     // input rows (their own, or those of another trainer)
    // The forward pass leaves every hidden activation's sign as a bit, which the backward pass takes for the ReLU mask.  Only
    // within one update: between the calls of a forward and a backward pass the activations are the caller's to change.
    bool bits;
};
bool share_launches(const im_trainer *a, const im_trainer *c)
{
    bool same = a->nl == c->nl && a->dims[a->nl] >= c->dims[c->nl];
    for (int l = 0; same && l < a->nl; ++l) same = a->dims[l] == c->dims[l];
    return same;
}

im::GemmOperands operands(const void *A, int lda, const void *B, int ldb, void *C, int ldc, const float *bias = nullptr)
{
    return {A, lda, B, ldb, C, ldc, bias, nullptr, 0, nullptr};
}
im::GemmOperands forward_operands(im_trainer *tr, uint16_t *x, int l)
{
    const bool last = l == tr->nl - 1;
    return operands(l == 0 ? x : tr->H[l], tr->Kp[l], tr->Wb[l], tr->Kp[l], last ? (void *)tr->out : tr->H[l + 1], last ? tr->dims[tr->nl] : tr->Np[l],
                    tr->b[l]);
}
im_status forward_on(const Nets &n, int M)
{
    im_trainer *a = n.a;
    uint32_t *status2 = n.c ? n.c->status : nullptr;
    im_status s = IM_OK;
    for (int l = 0; l < a->nl && s == IM_OK; ++l) {
        im::GemmOperands x = forward_operands(a, n.xa, l), y = n.c ? forward_operands(n.c, n.xc, l) : x;
        if (n.bits && l < a->nl - 1) { x.bits_out = a->bits[l + 1]; y.bits_out = n.c ? n.c->bits[l + 1] : nullptr; x.ld_bits = a->Mb; }
        const im::GemmOperands *py = n.c ? &y : nullptr;
        if (l < a->nl - 1) s = im::tc_gemm(x, py, M, a->Np[l], a->Kp[l], true, 0, a->status, status2, a->stream);
        else s = im::tc_gemm_head(x, py, M, a->dims[a->nl], n.c ? n.c->dims[n.c->nl] : 0, a->Kp[l], a->status, status2, a->stream);
    }
    return s;
}

im::OutGrad out_grad(im_trainer *tr, const float *d_out)
{
    const int L = tr->nl - 1;
    return {d_out, tr->dZ[L], tr->db_partial[L], tr->dims[tr->nl], tr->Np[L]};
}

// The tensor-core products of the backward pass.  dW = dZ^T H over row slices (slices[net][layer] of them) in one launch
// (both operands read as they lie, M/N-major tensor-core operands: no transposed copies).  dH = (H > 0) * (dZ W); the
// product's epilogue applies the ReLU mask and leaves the column sums of every 32-row block, which add up to the bias
// gradient of the layer below.
im_status backward_of(im_trainer *tr, uint16_t *x, im_trainer *tr2, uint16_t *x2, bool bits, int l, int M, int *slices)
{
    const int Np = tr->Np[l], Kp = tr->Kp[l], Npb = pad128(Np);
    const int cap = tr2 && tr2->s_max[l] < tr->s_max[l] ? tr2->s_max[l] : tr->s_max[l];
    *slices = im::tc_tn_slices(Np, Kp, Npb, M, cap, im::device_sm_count(), tr2 ? 2 : 1);
    const auto dw = [&](im_trainer *t, uint16_t *in) { return operands(t->dZ[l], Np, l == 0 ? in : t->H[l], Kp, t->dWs[l], Kp); };
    const auto dh = [&](im_trainer *t) {
        im::GemmOperands o = operands(t->dZ[l], Np, t->WbT[l], Np, t->dZ[l - 1], Kp);
        if (bits) { o.bits_in = t->bits[l]; o.ld_bits = t->Mb; }
        else { o.mask = t->H[l]; o.ld_mask = Kp; }
        o.colsum_partial = t->db_partial[l - 1];
        return o;
    };
    im::GemmOperands o = tr2 ? dw(tr2, x2) : im::GemmOperands();
    uint32_t *status2 = tr2 ? tr2->status : nullptr;
    im_status s = im::tc_gemm_tn(dw(tr, x), tr2 ? &o : nullptr, M, Np, Kp, *slices, Npb, tr->status, status2, tr->stream);
    if (l == 0 || s != IM_OK) return s;
    if (tr2) o = dh(tr2);
    return im::tc_gemm(dh(tr), tr2 ? &o : nullptr, M, Kp, Np, false, Kp, tr->status, status2, tr->stream);
}
im_status backward_products(const Nets &n, int M, int (*slices)[IM_MAX_LAYERS])
{
    im_status s = IM_OK;
    for (int l = n.a->nl - 1; l >= 0 && s == IM_OK; --l) {
        if (n.c && n.c->Np[l] == n.a->Np[l]) {
            s = backward_of(n.a, n.xa, n.c, n.xc, n.bits, l, M, &slices[0][l]);
            slices[1][l] = slices[0][l];
        } else {
            s = backward_of(n.a, n.xa, nullptr, nullptr, n.bits, l, M, &slices[0][l]);
            if (n.c && s == IM_OK) s = backward_of(n.c, n.xc, nullptr, nullptr, n.bits, l, M, &slices[1][l]);
        }
    }
    return s;
}

void add_weight_grads(im::GradReduceArgs &ga, im_trainer *tr, const int *slices)
{
    for (int l = 0; l < tr->nl; ++l)
        im::grad_reduce_add(ga, tr->dWs[l], (long long)pad128(tr->Np[l]) * tr->Kp[l], tr->Kp[l], slices[l], tr->dims[l + 1], tr->dims[l], tr->dW[l]);
}
void add_bias_grads(im::GradReduceArgs &ga, im_trainer *tr, int M)
{
    for (int l = 0; l < tr->nl; ++l)
        im::grad_reduce_add(ga, tr->db_partial[l], l == tr->nl - 1 ? (M + 127) / 128 : M / 32, tr->Np[l], tr->dims[l + 1], tr->db[l]);
}

void add_adam(im::AdamMultiArgs &aa, im_trainer *tr)
{
    for (int l = 0; l < tr->nl; ++l) {
        const int N = tr->dims[l + 1], K = tr->dims[l];
        im::adam_multi_add(aa, tr->W[l], tr->dW[l], tr->mW[l], tr->vW[l], N, K, tr->Wb[l], tr->Kp[l], tr->WbT[l], tr->Np[l], tr->t);
        im::adam_multi_add(aa, tr->b[l], tr->db[l], tr->mb[l], tr->vb[l], 1, N, nullptr, 0, nullptr, 0, tr->t);
    }
}

}  // namespace

struct im_ppo_updater {
    im_trainer *actor, *critic;
    im_ppo_update_config cfg;
    int A, Mb, t;
    float *log_std, *log_std_old, *m_ls, *v_ls, *d_log_std, *lr, *scale, *moments, *summary, *d_mean, *d_value;
    void *ws;
    double *norm_partial;          // one sum of squares per block of the gradient reduction
    int *done;                     // [2] block counters: gradient norm, Adam
    float *g_action, *g_mean_old, *g_logp_old, *g_advantage, *g_value_old, *g_returns;   // gathered minibatch (shuffled updates)
    int g_rows;
};

// One minibatch update; the critic's input rows are critic_x (its own, or the actor's).
static im_status update_on(im_ppo_updater *u, int M, const im_ppo_minibatch *mb, uint16_t *critic_x)
{
    if (!mb || M < 64 || (M & 63) || M > u->Mb) return IM_ERR_INVALID_ARG;
    if (!mb->action || !mb->mean_old || !mb->logp_old || !mb->advantage || !mb->returns) return IM_ERR_INVALID_ARG;
    if (u->cfg.clip_value_loss && !mb->value_old) return IM_ERR_INVALID_ARG;
    if (!adam_ok(&u->cfg.adam) || !(u->cfg.kl_target > 0.0f) || !(u->cfg.lr_min > 0.0f)) return IM_ERR_INVALID_ARG;
    im_trainer *a = u->actor, *c = u->critic;
    cudaStream_t st = a->stream;
    const Nets both = {a, c, a->H[0], critic_x, true}, one_a = {a, nullptr, a->H[0], nullptr, true}, one_c = {c, nullptr, critic_x, nullptr, true};
    const bool shared = share_launches(a, c);
    im_status s = forward_on(shared ? both : one_a, M);
    if (s == IM_OK && !shared) s = forward_on(one_c, M);
    if (s != IM_OK) return s;
    const float *mom = nullptr;
    if (u->cfg.normalize_advantage) {
        s = im_moments(mb->advantage, M, u->moments, u->ws, st);
        if (s != IM_OK) return s;
        mom = u->moments;
    }
    const im_ppo_config pc = {u->cfg.clip, u->cfg.value_coef, u->cfg.entropy_coef, u->cfg.clip_value_loss};
    const im_ppo_batch pb = {a->out, u->log_std, mb->action, mb->logp_old, mb->mean_old,
                             mb->log_std_old ? mb->log_std_old : u->log_std_old, mb->advantage, mom, c->out, mb->value_old, mb->returns};
    im::OutGradArgs og = {};
    s = im::ppo_loss_rows(&pc, M, u->A, &pb, u->d_mean, u->d_log_std, u->d_value, u->summary, u->ws, st, &og.fin);
    if (s != IM_OK) return s;
    og.n_nets = 2; og.M = M; og.net[0] = out_grad(a, u->d_mean); og.net[1] = out_grad(c, u->d_value);
    if (im::launch_out_grads(og, st) != cudaSuccess) return IM_ERR_CUDA;
    int slices[2][IM_MAX_LAYERS];
    s = backward_products(shared ? both : one_a, M, slices);
    if (s == IM_OK && !shared) s = backward_products(one_c, M, slices + 1);
    if (s != IM_OK) return s;
    // every gradient tensor of both nets, and the global-norm clip factor over them and the log-std's
    im::GradReduceArgs ga = {};
    add_weight_grads(ga, a, slices[0]);
    add_weight_grads(ga, c, slices[1]);
    add_bias_grads(ga, a, M);
    add_bias_grads(ga, c, M);
    ga.extra = u->d_log_std; ga.n_extra = u->A;
    ga.partial = u->norm_partial; ga.done = u->done; ga.max_norm = u->cfg.max_grad_norm; ga.scale_out = u->scale;
    if (im::launch_grad_reduce(ga, st) != cudaSuccess) return IM_ERR_CUDA;
    im::AdamMultiArgs aa = {};
    aa.cfg = u->cfg.adam; aa.lr = u->lr; aa.grad_scale = u->scale;
    aa.kl = u->summary + 4; aa.kl_target = u->cfg.kl_target; aa.lr_min = u->cfg.lr_min; aa.lr_max = u->cfg.lr_max; aa.done = u->done + 1;
    a->t += 1; c->t += 1; u->t += 1;
    add_adam(aa, a);
    add_adam(aa, c);
    im::adam_multi_add(aa, u->log_std, u->d_log_std, u->m_ls, u->v_ls, 1, u->A, nullptr, 0, nullptr, 0, u->t);
    return im::launch_adam_multi(aa, st) == cudaSuccess ? IM_OK : IM_ERR_CUDA;
}

extern "C" {

/* Equal row slices for the dW product of a layer with Np (padded) outputs and Kp (padded) inputs on M rows through
 * im_gemm_bf16_tn (the trainer itself slices by whole 64-row blocks: tc_tn_slices).  dW contracts over the batch -- a long sum feeding few output tiles -- so the rows are cut into S slices that run as one launch.
 * S is the power of two (slices of whole 128-row blocks) with the least modelled time: waves of tiles on 148 SMs
 * times rows per slice (5 ns per row and wave, measured on a 1024 x 1024 layer), plus the pass that adds the S
 * partial products (1 ps per element).  any_rows: ignore the divisibility rule (an upper bound for sizing). */
int32_t im_trainer_dw_slices(int32_t Np, int32_t Kp, int64_t M, int32_t max_split, int32_t any_rows)
{
    const int npb = pad128(Np);
    const long long tiles = (long long)(npb / 128) * ((Kp + 255) / 256 > 1 ? (Kp + 255) / 256 : 1);
    int best = 1;
    double best_cost = -1.0;
    for (int S = 1; S <= max_split && (any_rows || M % (128LL * S) == 0); S *= 2) {
        const long long waves = (tiles * S + 147) / 148;
        const double cost = 5e-9 * (double)M * (double)waves / S + 1e-12 * (double)S * npb * Kp;
        if (best_cost < 0.0 || cost < best_cost * (1.0 - 1e-9)) { best = S; best_cost = cost; }
    }
    return best;
}

void im_trainer_destroy(im_trainer *tr)
{
    if (!tr) return;
    for (int l = 0; l < IM_MAX_LAYERS; ++l) {
        cudaFree(tr->W[l]); cudaFree(tr->b[l]); cudaFree(tr->mW[l]); cudaFree(tr->vW[l]); cudaFree(tr->mb[l]); cudaFree(tr->vb[l]);
        cudaFree(tr->dW[l]); cudaFree(tr->db[l]); cudaFree(tr->Wb[l]); cudaFree(tr->WbT[l]); cudaFree(tr->H[l]); cudaFree(tr->bits[l]); cudaFree(tr->dZ[l]);
        cudaFree(tr->dWs[l]); cudaFree(tr->db_partial[l]);
    }
    cudaFree(tr->out); cudaFree(tr->status);
    delete tr;
}

im_status im_trainer_create(int32_t n_layers, const int32_t *dims, const float *const *W, const float *const *b,
                            int32_t max_rows, void *cuda_stream, im_trainer **out)
{
    if (!dims || !W || !b || !out || n_layers < 2 || n_layers > IM_MAX_LAYERS) return IM_ERR_INVALID_ARG;
    if (max_rows < 64 || (max_rows & 63)) return IM_ERR_INVALID_ARG;
    for (int l = 0; l <= n_layers; ++l)
        if (dims[l] < 1) return IM_ERR_INVALID_ARG;
    for (int l = 1; l < n_layers; ++l)
        if (dims[l] & 63) return IM_ERR_UNSUPPORTED;                 // hidden widths are whole 64-column tiles
    if (dims[n_layers] > 80) return IM_ERR_UNSUPPORTED;              // the fp32-output head kernel
    for (int l = 0; l < n_layers; ++l)
        if (!W[l] || !b[l]) return IM_ERR_INVALID_ARG;
    if (im::device_sm_count() <= 0) return IM_ERR_UNSUPPORTED;
    im_trainer *tr = new (std::nothrow) im_trainer();
    if (!tr) return IM_ERR_ALLOC;
    std::memset(tr, 0, sizeof(*tr));
    tr->nl = n_layers; tr->Mb = max_rows; tr->max_split = 64; tr->stream = (cudaStream_t)cuda_stream;
    cudaStream_t st = tr->stream;
    for (int l = 0; l <= n_layers; ++l) tr->dims[l] = dims[l];
    bool ok = true;
    for (int l = 0; l < n_layers && ok; ++l) {
        const int N = dims[l + 1], K = dims[l], Np = pad64(N), Kp = pad64(K);
        tr->Np[l] = Np; tr->Kp[l] = Kp;
        const size_t wn = (size_t)N * K;
        ok = dev_alloc(&tr->W[l], wn, st, false) && dev_alloc(&tr->b[l], (size_t)Np, st) && dev_alloc(&tr->mW[l], wn, st) &&
             dev_alloc(&tr->vW[l], wn, st) && dev_alloc(&tr->mb[l], (size_t)N, st) && dev_alloc(&tr->vb[l], (size_t)N, st) &&
             dev_alloc(&tr->dW[l], wn, st) && dev_alloc(&tr->db[l], (size_t)N, st) && dev_alloc(&tr->Wb[l], (size_t)Np * Kp, st) &&
             dev_alloc(&tr->WbT[l], (size_t)Kp * Np, st) && dev_alloc(&tr->H[l], (size_t)max_rows * Kp, st) &&
             (l == 0 || dev_alloc(&tr->bits[l], (size_t)max_rows * (Kp / 64), st, false)) && dev_alloc(&tr->dZ[l], (size_t)max_rows * Np, st);
        // partial dW products: room for the most slices the model can choose for any number of rows
        tr->s_max[l] = max_slices(Np, Kp, max_rows, tr->max_split);
        ok = ok && dev_alloc(&tr->dWs[l], (size_t)tr->s_max[l] * pad128(Np) * Kp, st, false) &&
             dev_alloc(&tr->db_partial[l], (size_t)(l == n_layers - 1 ? (max_rows + 127) / 128 : max_rows / 32) * Np, st, false);
    }
    ok = ok && dev_alloc(&tr->out, (size_t)max_rows * dims[n_layers], st) && dev_alloc(&tr->status, 1, st);
    if (!ok) { im_trainer_destroy(tr); return IM_ERR_ALLOC; }
    // weights: fp32 masters as given; bf16 working copies (rounded on the device, zero padded) and their transposes
    for (int l = 0; l < n_layers; ++l) {
        const int N = dims[l + 1], K = dims[l];
        if (cudaMemcpyAsync(tr->W[l], W[l], (size_t)N * K * sizeof(float), cudaMemcpyHostToDevice, tr->stream) != cudaSuccess ||
            cudaMemcpyAsync(tr->b[l], b[l], (size_t)N * sizeof(float), cudaMemcpyHostToDevice, tr->stream) != cudaSuccess) {
            im_trainer_destroy(tr);
            return IM_ERR_CUDA;
        }
        im_status s = im_f32_to_bf16_padded(tr->W[l], K, N, K, tr->Wb[l], tr->Kp[l], tr->stream);
        if (s == IM_OK) s = im_transpose_bf16(tr->Wb[l], tr->Kp[l], tr->Np[l], tr->Kp[l], tr->WbT[l], tr->Np[l], tr->stream);
        if (s != IM_OK) { im_trainer_destroy(tr); return s; }
    }
    if (cudaStreamSynchronize(tr->stream) != cudaSuccess) { im_trainer_destroy(tr); return IM_ERR_CUDA; }   // W, b are the caller's
    *out = tr;
    return IM_OK;
}

im_status im_trainer_tensor(im_trainer *tr, int32_t which, int32_t layer, void **ptr, int64_t *rows, int64_t *cols,
                            int64_t *ld, int32_t *dtype)
{
    if (!tr || !ptr || !rows || !cols || !ld || !dtype) return IM_ERR_INVALID_ARG;
    const bool per_layer = which != IM_TRAINER_OUT && which != IM_TRAINER_STATUS;
    if (per_layer && (layer < 0 || layer >= tr->nl)) return IM_ERR_INVALID_ARG;
    const int l = per_layer ? layer : 0;
    const int64_t N = tr->dims[l + 1], K = tr->dims[l], Np = tr->Np[l], Kp = tr->Kp[l];
    *dtype = IM_DTYPE_F32;
    switch (which) {
    case IM_TRAINER_W: *ptr = tr->W[l]; *rows = N; *cols = K; *ld = K; break;
    case IM_TRAINER_B: *ptr = tr->b[l]; *rows = 1; *cols = N; *ld = Np; break;
    case IM_TRAINER_W_BF16: *ptr = tr->Wb[l]; *rows = Np; *cols = Kp; *ld = Kp; *dtype = IM_DTYPE_BF16; break;
    case IM_TRAINER_WT_BF16: *ptr = tr->WbT[l]; *rows = Kp; *cols = Np; *ld = Np; *dtype = IM_DTYPE_BF16; break;
    case IM_TRAINER_M_W: *ptr = tr->mW[l]; *rows = N; *cols = K; *ld = K; break;
    case IM_TRAINER_V_W: *ptr = tr->vW[l]; *rows = N; *cols = K; *ld = K; break;
    case IM_TRAINER_M_B: *ptr = tr->mb[l]; *rows = 1; *cols = N; *ld = N; break;
    case IM_TRAINER_V_B: *ptr = tr->vb[l]; *rows = 1; *cols = N; *ld = N; break;
    case IM_TRAINER_DW: *ptr = tr->dW[l]; *rows = N; *cols = K; *ld = K; break;
    case IM_TRAINER_DB: *ptr = tr->db[l]; *rows = 1; *cols = N; *ld = N; break;
    case IM_TRAINER_H: *ptr = tr->H[l]; *rows = tr->Mb; *cols = Kp; *ld = Kp; *dtype = IM_DTYPE_BF16; break;
    case IM_TRAINER_OUT: *ptr = tr->out; *rows = tr->Mb; *cols = tr->dims[tr->nl]; *ld = tr->dims[tr->nl]; break;
    case IM_TRAINER_STATUS: *ptr = tr->status; *rows = 1; *cols = 1; *ld = 1; *dtype = IM_DTYPE_U32; break;
    default: return IM_ERR_INVALID_ARG;
    }
    return IM_OK;
}

im_status im_trainer_set_step_count(im_trainer *tr, int32_t t)
{
    if (!tr || t < 0) return IM_ERR_INVALID_ARG;
    tr->t = t;
    return IM_OK;
}

im_status im_trainer_forward(im_trainer *tr, int32_t M)
{
    if (!tr || M < 1 || M > tr->Mb) return IM_ERR_INVALID_ARG;
    return forward_on({tr, nullptr, tr->H[0], nullptr, false}, M);
}

im_status im_trainer_backward(im_trainer *tr, const float *d_out, int32_t M)
{
    if (!tr || !d_out || M < 64 || (M & 63) || M > tr->Mb) return IM_ERR_INVALID_ARG;
    im::OutGradArgs og = {};
    og.n_nets = 1; og.M = M; og.net[0] = out_grad(tr, d_out);
    if (im::launch_out_grads(og, tr->stream) != cudaSuccess) return IM_ERR_CUDA;
    int slices[1][IM_MAX_LAYERS];
    const im_status s = backward_products({tr, nullptr, tr->H[0], nullptr, false}, M, slices);
    if (s != IM_OK) return s;
    im::GradReduceArgs ga = {};
    add_weight_grads(ga, tr, slices[0]);
    add_bias_grads(ga, tr, M);
    return im::launch_grad_reduce(ga, tr->stream) == cudaSuccess ? IM_OK : IM_ERR_CUDA;
}

im_status im_trainer_step(im_trainer *tr, const im_adam_config *adam, const float *lr, const float *grad_scale)
{
    if (!tr || !adam || !lr || !adam_ok(adam)) return IM_ERR_INVALID_ARG;
    im::AdamMultiArgs aa = {};
    aa.cfg = *adam; aa.lr = const_cast<float *>(lr); aa.grad_scale = grad_scale;      // (lr is only written with kl)
    tr->t += 1;
    add_adam(aa, tr);
    return im::launch_adam_multi(aa, tr->stream) == cudaSuccess ? IM_OK : IM_ERR_CUDA;
}

im_status im_trainer_push_to_policy(im_trainer *tr, im_policy *p)
{
    if (!tr || !p || p->nl != tr->nl || p->stream != tr->stream) return IM_ERR_INVALID_ARG;
    for (int l = 0; l <= tr->nl; ++l)
        if (p->cfg.dims[l] != tr->dims[l]) return IM_ERR_INVALID_ARG;
    for (int l = 0; l < tr->nl; ++l) {
        void *w = nullptr;
        int32_t ld = 0;
        float *bias = nullptr;
        im_status s = im_policy_layer_buffers(p, l, &w, &ld, &bias);
        if (s != IM_OK) return s;
        const int N = tr->dims[l + 1], K = tr->dims[l];
        if (p->tensor_path || p->cfg.dtype == 1) {
            s = im_f32_to_bf16_padded(tr->W[l], K, N, K, static_cast<uint16_t *>(w), ld, tr->stream);
        } else {
            s = cudaMemcpy2DAsync(w, (size_t)ld * 4, tr->W[l], (size_t)K * 4, (size_t)K * 4, N, cudaMemcpyDeviceToDevice, tr->stream) ==
                        cudaSuccess ? IM_OK : IM_ERR_CUDA;
        }
        if (s == IM_OK) s = im_copy_f32(bias, tr->b[l], N, tr->stream);
        if (s != IM_OK) return s;
    }
    return IM_OK;
}

/* ------------------------------------------------------------------ PPO updater */
void im_ppo_updater_destroy(im_ppo_updater *u)
{
    if (!u) return;
    cudaFree(u->log_std); cudaFree(u->log_std_old); cudaFree(u->m_ls); cudaFree(u->v_ls); cudaFree(u->d_log_std); cudaFree(u->lr);
    cudaFree(u->scale); cudaFree(u->moments); cudaFree(u->summary); cudaFree(u->d_mean); cudaFree(u->d_value); cudaFree(u->ws);
    cudaFree(u->norm_partial); cudaFree(u->done);
    cudaFree(u->g_action);
    delete u;
}

im_status im_ppo_updater_create(im_trainer *actor, im_trainer *critic, const float *log_std, const im_ppo_update_config *cfg,
                                im_ppo_updater **out)
{
    if (!actor || !critic || !log_std || !cfg || !out) return IM_ERR_INVALID_ARG;
    if (actor->stream != critic->stream || critic->dims[critic->nl] != 1 || actor->Mb != critic->Mb) return IM_ERR_INVALID_ARG;
    if (!(cfg->lr > 0.0f) || !(cfg->clip > 0.0f) || !(cfg->max_grad_norm > 0.0f) || !(cfg->lr_min <= cfg->lr_max)) return IM_ERR_INVALID_ARG;
    im_ppo_updater *u = new (std::nothrow) im_ppo_updater();
    if (!u) return IM_ERR_ALLOC;
    std::memset(u, 0, sizeof(*u));
    u->actor = actor; u->critic = critic; u->cfg = *cfg; u->A = actor->dims[actor->nl]; u->Mb = actor->Mb;
    const size_t A = (size_t)u->A;
    cudaStream_t st = actor->stream;
    size_t n_blocks = 1;
    for (im_trainer *t : {actor, critic})
        for (int l = 0; l < t->nl; ++l) n_blocks += im::grad_matrix_blocks(t->dims[l + 1], t->dims[l]) + im::grad_vector_blocks(t->dims[l + 1]);
    bool ok = dev_alloc(&u->norm_partial, n_blocks, st, false) && dev_alloc(&u->done, 2, st) && dev_alloc(&u->log_std, A, st) && dev_alloc(&u->log_std_old, A, st) && dev_alloc(&u->m_ls, A, st) && dev_alloc(&u->v_ls, A, st) &&
              dev_alloc(&u->d_log_std, A, st) && dev_alloc(&u->lr, 1, st) && dev_alloc(&u->scale, 2, st) && dev_alloc(&u->moments, 2, st) &&
              dev_alloc(&u->summary, 6, st) && dev_alloc(&u->d_mean, (size_t)u->Mb * A, st) && dev_alloc(&u->d_value, (size_t)u->Mb, st) &&
              cudaMalloc(&u->ws, im_ppo_workspace_bytes()) == cudaSuccess;
    if (!ok) { im_ppo_updater_destroy(u); return IM_ERR_ALLOC; }
    if (cudaMemcpyAsync(u->log_std, log_std, A * 4, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(u->log_std_old, log_std, A * 4, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(u->lr, &cfg->lr, 4, cudaMemcpyHostToDevice, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
        im_ppo_updater_destroy(u);
        return IM_ERR_CUDA;
    }
    *out = u;
    return IM_OK;
}

im_status im_ppo_updater_tensor(im_ppo_updater *u, int32_t which, float **ptr, int64_t *n)
{
    if (!u || !ptr || !n) return IM_ERR_INVALID_ARG;
    switch (which) {
    case IM_PPO_LOG_STD: *ptr = u->log_std; *n = u->A; break;
    case IM_PPO_LOG_STD_OLD: *ptr = u->log_std_old; *n = u->A; break;
    case IM_PPO_M_LOG_STD: *ptr = u->m_ls; *n = u->A; break;
    case IM_PPO_V_LOG_STD: *ptr = u->v_ls; *n = u->A; break;
    case IM_PPO_LR: *ptr = u->lr; *n = 1; break;
    case IM_PPO_GRAD_SCALE: *ptr = u->scale; *n = 2; break;
    case IM_PPO_SUMMARY: *ptr = u->summary; *n = 6; break;
    default: return IM_ERR_INVALID_ARG;
    }
    return IM_OK;
}

im_status im_ppo_updater_set_step_count(im_ppo_updater *u, int32_t t)
{
    if (!u || t < 0) return IM_ERR_INVALID_ARG;
    u->t = t;
    return IM_OK;
}

im_status im_ppo_update(im_ppo_updater *u, int32_t M, const im_ppo_minibatch *mb)
{
    if (!u) return IM_ERR_INVALID_ARG;
    return update_on(u, M, mb, u->critic->H[0]);
}

im_status im_ppo_update_rollout(im_ppo_updater *u, const im_rollout_view *v, int32_t epochs, int32_t n_minibatches,
                                const int32_t *perm)
{
    if (!u || !v || epochs < 1 || n_minibatches < 1) return IM_ERR_INVALID_ARG;
    if (!v->obs || !v->action || !v->mean || !v->logp || !v->advantage || !v->returns || !v->value) return IM_ERR_INVALID_ARG;
    const int64_t total = (int64_t)v->T * v->N;
    if (v->T < 1 || v->N < 1 || v->A != u->A || total % n_minibatches) return IM_ERR_INVALID_ARG;
    const int64_t M64 = total / n_minibatches;
    if (M64 % 64 || M64 > u->Mb) return IM_ERR_INVALID_ARG;
    const int M = (int)M64, A = u->A, D = u->actor->dims[0];
    if (u->critic->dims[0] != D || v->ld_obs < D) return IM_ERR_INVALID_ARG;
    cudaStream_t st = u->actor->stream;
    if (perm && u->g_rows < M) {
        // (first shuffled update of this size: buffers for the gathered minibatch)
        cudaFree(u->g_action);
        u->g_rows = 0;
        if (!dev_alloc(&u->g_action, (size_t)M * (2 * A + 4), st, false)) return IM_ERR_ALLOC;
        u->g_mean_old = u->g_action + (size_t)M * A;                  // (M is a multiple of 64: every part is 16-byte aligned)
        u->g_logp_old = u->g_mean_old + (size_t)M * A;
        u->g_advantage = u->g_logp_old + M; u->g_value_old = u->g_advantage + M; u->g_returns = u->g_value_old + M;
        u->g_rows = M;
    }
    for (int ep = 0; ep < epochs; ++ep) {
        for (int k = 0; k < n_minibatches; ++k) {
            const int64_t r0 = (int64_t)k * M;
            im_ppo_minibatch mb;
            im_status s = IM_OK;
            // one copy of the observations as bf16 rows, in the actor's input buffer, serves both nets; the critic's own holds
            // the last minibatch afterwards as well
            im_trainer *t = u->actor;
            uint16_t *critic_rows = ep == epochs - 1 && k == n_minibatches - 1 ? u->critic->H[0] : nullptr;
            if (!perm) {
                // contiguous block: the observations are converted, the rest is read in place
                s = im::f32_to_bf16_padded(v->obs + r0 * v->ld_obs, v->ld_obs, M, D, t->H[0], critic_rows, t->Kp[0], st);
                mb = {v->action + r0 * A, v->mean + r0 * A, nullptr, v->logp + r0, v->advantage + r0, v->value + r0, v->returns + r0};
            } else {
                const im::GatherArgs ga = {v->obs, v->action, v->mean, v->logp, v->advantage, v->value, v->returns, perm + (int64_t)ep * total + r0,
                                           v->ld_obs, total, M, D, A, t->Kp[0], t->H[0], critic_rows, u->g_action, u->g_mean_old, u->g_logp_old,
                                           u->g_advantage, u->g_value_old, u->g_returns, t->status};
                if (im::launch_gather_minibatch(ga, st) != cudaSuccess) s = IM_ERR_CUDA;
                mb = {u->g_action, u->g_mean_old, nullptr, u->g_logp_old, u->g_advantage, u->g_value_old, u->g_returns};
            }
            if (s == IM_OK) s = update_on(u, M, &mb, t->H[0]);
            if (s != IM_OK) return s;
        }
    }
    return IM_OK;
}

}  // extern "C"
