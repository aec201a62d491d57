"""The update's multi-tensor steps on odd shapes: input widths that are no multiple of four, one-column outputs, tile
remainders, rows that leave one 128-row block ragged; checked against the one-tensor entry points and fp64."""
import numpy as np
import pytest

from paper_2609_09821_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(361, 64, 128, 28), (66, 192, 64, 1), (129, 64, 80)])
@pytest.mark.parametrize("M", [64, 192, 1984])
def test_trainer_step_matches_single_tensor_adam(dims, M):
    import torch
    from paper_2609_09821_b200 import binding as B, trainer as T
    w = W.make_policy_weights(dims, "f32", seed=2)
    tr = T.MlpTrainer(dims, w["W"], w["b"], 1984)
    g = torch.Generator("cuda").manual_seed(M)
    rows = tr.input_rows(M)
    rows.zero_()
    rows[:, :dims[0]] = torch.randn(M, dims[0], device="cuda", generator=g).bfloat16()
    lr = torch.full((1,), 1e-3, device="cuda")
    scale = torch.full((1,), 0.7, device="cuda")
    ref = [[t.clone() for t in ts] for ts in (tr.W, tr.mW, tr.vW, tr.b, tr.mb, tr.vb)]
    for t in range(1, 4):
        tr.forward(M)
        tr.backward(torch.randn(M, dims[-1], device="cuda", generator=g), M)
        tr.step(lr, scale)
        for l in range(len(dims) - 1):
            B.adam_step(ref[0][l].view(-1), tr.dW[l].contiguous().view(-1), ref[1][l].view(-1), ref[2][l].view(-1), lr, t, grad_scale=scale)
            B.adam_step(ref[3][l], tr.db[l].clone(), ref[4][l], ref[5][l], lr, t, grad_scale=scale)
    torch.cuda.synchronize()
    for l in range(len(dims) - 1):
        for got, want in zip((tr.W, tr.mW, tr.vW, tr.b, tr.mb, tr.vb), ref):
            assert torch.equal(got[l], want[l])                  # the same fp32 operations
        N, K = dims[l + 1], dims[l]
        wb = torch.zeros_like(tr.Wb[l])
        wb[:N, :K] = tr.W[l].bfloat16()
        assert torch.equal(tr.Wb[l], wb) and torch.equal(tr.WbT[l], wb.T.contiguous())


@pytest.mark.parametrize("T_,N,mb,shuffled", [(4, 48, 1, True), (4, 50, 1, False), (8, 120, 3, True)])
def test_rollout_update_clip_factor_and_summary(T_, N, mb, shuffled):
    import torch
    from paper_2609_09821_b200 import rollout as R, trainer as T
    if T_ * N // mb % 64:
        N = 64 * mb
    dims, A = (361, 64, 128, 28), 28
    wa, wc = W.make_policy_weights(dims, "f32", 3), W.make_policy_weights(dims[:-1] + (1,), "f32", 4)
    rows = T_ * N // mb
    a, c = T.MlpTrainer(dims, wa["W"], wa["b"], rows), T.MlpTrainer(dims[:-1] + (1,), wc["W"], wc["b"], rows)
    upd = T.PpoUpdater(a, c, torch.full((A,), -1.0), lr=1e-5)
    st = R.RolloutStorage(T_, N, A, 384)
    g = torch.Generator("cuda").manual_seed(1)
    st.obs[..., :361] = torch.randn(T_ + 1, N, 361, device="cuda", generator=g)
    for x in (st.action, st.mean, st.logp, st.value, st.advantage, st.returns):
        x.copy_(torch.randn(x.shape, device="cuda", generator=g))
    x = st.obs[:T_, :, :361]
    for l in range(3):                                           # actions near the network's own means
        x = x @ torch.from_numpy(wa["W"][l]).cuda().T + torch.from_numpy(wa["b"][l]).cuda()
        x = torch.relu(x) if l < 2 else x
    z = torch.randn(st.action.shape, device="cuda", generator=g)
    st.mean.copy_(x)
    st.action.copy_(x + np.exp(-1.0) * z)
    st.logp.copy_(-0.5 * z.square().sum(2) + A - 0.5 * A * np.log(2 * np.pi))
    perm = torch.stack([torch.randperm(T_ * N, device="cuda", generator=g) for _ in range(2)]).to(torch.int32) if shuffled else None
    T.update_from_storage(upd, st, 2, mb, perm)
    torch.cuda.synchronize()
    norm2 = sum(float(x.double().square().sum()) for t in (a, c) for x in t.dW + t.db)
    # the last minibatch's gradients are still there; the log-std's own (28 sums of z^2 - 1 weighted by normalised
    # advantages over at least 192 samples) is small beside them
    norm = float(upd.scale[1])
    assert norm * 0.9 <= norm2 ** 0.5 <= norm * (1 + 1e-6) and bool(torch.isfinite(upd.summary).all())
    assert abs(float(upd.scale[0]) - min(1.0, 1.0 / (norm + 1e-6))) <= 1e-6
    assert a.device_status() == 0 and c.device_status() == 0


@pytest.mark.parametrize("n", [1, 2, 255, 2049, 16000, 2 ** 17, 2 ** 17 + 1, 300001])
def test_moments_of_any_length(n):
    import torch
    from paper_2609_09821_b200 import binding as B
    x = 3.0 + 2.0 * torch.randn(n + 8, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    out, ws = torch.empty(2, device="cuda"), B.ppo_workspace()
    B.moments(x[:n], out, ws)
    got = out.cpu().numpy().astype(np.float64)
    ref = x[:n].cpu().numpy().astype(np.float64)
    std = ref.std(ddof=1) if n > 1 else 0.0
    want = np.array([ref.mean(), 1.0 / (std + 1e-8)])
    assert np.all(np.abs(got - want) <= 2e-7 * np.abs(want))         # fp64 sums, one rounding to fp32


@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("D", [361, 70])
def test_both_nets_input_rows_hold_the_last_minibatch(shuffled, D):
    import torch
    from paper_2609_09821_b200 import rollout as R, trainer as T
    T_, N, A, ld = 4, 96, 5, (D + 63) // 64 * 64
    wa, wc = W.make_policy_weights((D, 64, A), "f32", 3), W.make_policy_weights((D, 128, 1), "f32", 4)
    M = T_ * N // 2
    a, c = T.MlpTrainer((D, 64, A), wa["W"], wa["b"], M), T.MlpTrainer((D, 128, 1), wc["W"], wc["b"], M)
    upd = T.PpoUpdater(a, c, torch.full((A,), -1.0), lr=1e-5)
    st = R.RolloutStorage(T_, N, A, ld)
    g = torch.Generator("cuda").manual_seed(1)
    for x in (st.obs, st.action, st.mean, st.logp, st.value, st.advantage, st.returns):
        x.copy_(torch.randn(x.shape, device="cuda", generator=g))
    perm = torch.stack([torch.randperm(T_ * N, device="cuda", generator=g) for _ in range(2)]).to(torch.int32) if shuffled else None
    T.update_from_storage(upd, st, 2, 2, perm)
    flat = st.obs[:T_].reshape(T_ * N, ld)[:, :D]
    want = torch.zeros(M, ld, dtype=torch.bfloat16, device="cuda")
    want[:, :D] = (flat[perm[1, M:].long()] if shuffled else flat[M:]).bfloat16()
    assert torch.equal(a.input_rows(M), want) and torch.equal(c.input_rows(M), want)
