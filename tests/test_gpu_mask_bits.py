"""A minibatch update takes the ReLU mask of its backward products from the bits that its forward products leave, a trainer's
own forward and backward calls from the activations.  The same products in the same order otherwise: bias gradients (sums of
the masked fp32 values) agree bit for bit, and the weights' as well where both sides cut the rows into the same slices, which
nets that share no launches do.  Every tile width, one CTA and pairs, ragged last tiles."""
import pytest

from paper_2609_09821_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [64, 448, 64 * 33, 64 * 61, 64 * 250])
@pytest.mark.parametrize("dims,cdims", [((361, 1024, 512, 28), (361, 512, 256, 1)), ((70, 64, 320, 80), (70, 128, 64, 1)),
                                        ((361, 1024, 512, 28), (361, 1024, 512, 1))])
def test_mask_bits_give_the_gradients_of_the_activations(M, dims, cdims):
    import torch
    from paper_2609_09821_b200 import binding as B, trainer as T
    A, shared = dims[-1], dims[:-1] == cdims[:-1]
    wa, wc = W.make_policy_weights(dims, "f32", 5), W.make_policy_weights(cdims, "f32", 6)
    make = lambda: (T.MlpTrainer(dims, wa["W"], wa["b"], M), T.MlpTrainer(cdims, wc["W"], wc["b"], M))
    nets, ref = make(), make()
    g = torch.Generator("cuda").manual_seed(M + A)
    x = torch.randn(M, dims[0], device="cuda", generator=g).bfloat16()
    x[M // 2] = 0.0                                    # a row whose activations are the biases alone
    for t in nets + ref:
        rows = t.input_rows(M)
        rows.zero_()
        rows[:, :dims[0]] = x
    log_std = torch.full((A,), -0.5, device="cuda")
    mean, value = ref[0].forward(M).clone(), ref[1].forward(M).clone()
    col = lambda: torch.randn(M, device="cuda", generator=g)
    action = mean + 0.6 * torch.randn(M, A, device="cuda", generator=g)
    logp = -0.5 * (((action - mean) / log_std.exp()) ** 2).sum(1) - log_std.sum() - 0.5 * A * 1.8378770664
    batch = dict(action=action, mean_old=mean + 0.01, logp_old=logp, advantage=col(), value_old=col(), returns=col())
    upd = T.PpoUpdater(nets[0], nets[1], log_std.cpu(), lr=1e-6, normalize_advantage=False)
    upd.update(M, batch)
    torch.cuda.synchronize()
    assert torch.equal(nets[0].out[:M], mean) and torch.equal(nets[1].out[:M], value)
    d_mean, d_ls, d_value, summary = (torch.empty(M, A, device="cuda"), torch.empty(A, device="cuda"), torch.empty(M, device="cuda"),
                                      torch.empty(6, device="cuda"))
    B.ppo_loss(dict(batch, mean=mean, value=value[:, 0].contiguous(), log_std=log_std, log_std_old=log_std), d_mean, d_ls, d_value, summary,
               B.ppo_workspace(), 0.2, 2.0, 0.0, True)
    # the loss's sums, by another number of threads: added in fp64 in another order, one rounding to fp32 each
    assert torch.allclose(upd.summary, summary, rtol=2.5e-7, atol=1e-9 * float(summary.abs().max()))
    ref[0].backward(d_mean, M)
    ref[1].backward(d_value.view(M, 1), M)
    torch.cuda.synchronize()
    for got, want in zip(nets, ref):
        assert got.device_status() == 0
        for l in range(len(dims) - 1):
            assert torch.equal(got.db[l], want.db[l]), (l, M)
            if not shared:
                assert torch.equal(got.dW[l], want.dW[l]), (l, M)


def test_fewer_rows_than_the_trainer_has_room_for(monkeypatch):
    """The mask words' columns lie max_rows apart, not as many as the minibatch has rows."""
    from paper_2609_09821_b200 import trainer as T
    make = T.MlpTrainer
    monkeypatch.setattr(T, "MlpTrainer", lambda dims, W, b, rows: make(dims, W, b, rows + 192))
    for dims, cdims in (((361, 1024, 512, 28), (361, 512, 256, 1)), ((361, 1024, 512, 28), (361, 1024, 512, 1))):
        test_mask_bits_give_the_gradients_of_the_activations(64 * 61, dims, cdims)
