"""A minibatch update runs the tensor-core products of an actor and a critic of equal widths in common launches; the same
gradients as each net's own forward and backward from the same output gradients.  Row counts around the tile sizes and
beyond one wave of CTA pairs; last layers padded alike and not; nets of other widths, which share nothing."""
import pytest

from paper_2609_09821_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [64, 192, 2048, 64 * 61, 64 * 250])
@pytest.mark.parametrize("dims,cdims", [((361, 1024, 512, 28), (361, 1024, 512, 1)), ((70, 64, 320, 69), (70, 64, 320, 1)),
                                        ((129, 512, 256, 128, 80), (129, 512, 256, 128, 1)), ((361, 256, 128, 28), (361, 128, 64, 1))])
def test_update_matches_the_nets_one_by_one(M, dims, cdims):
    import torch
    from paper_2609_09821_b200 import binding as B, trainer as T
    A = dims[-1]
    wa, wc = W.make_policy_weights(dims, "f32", 3), W.make_policy_weights(cdims, "f32", 4)
    make = lambda: (T.MlpTrainer(dims, wa["W"], wa["b"], M), T.MlpTrainer(cdims, wc["W"], wc["b"], M))
    nets, ref = make(), make()
    g = torch.Generator("cuda").manual_seed(M + A)
    x = torch.randn(M, dims[0], device="cuda", generator=g).bfloat16()
    for t in nets + ref:
        rows = t.input_rows(M)
        rows.zero_()
        rows[:, :dims[0]] = x
    log_std = torch.full((A,), -0.5, device="cuda")
    mean, value = ref[0].forward(M).clone(), ref[1].forward(M).clone()
    action = mean + 0.6 * torch.randn(M, A, device="cuda", generator=g)
    col = lambda: torch.randn(M, device="cuda", generator=g)
    logp = -0.5 * (((action - mean) / log_std.exp()) ** 2).sum(1) - log_std.sum() - 0.5 * A * 1.8378770664
    batch = dict(action=action, mean_old=mean + 0.01, logp_old=logp + 0.05 * col(), advantage=col(), value_old=col(), returns=col())
    upd = T.PpoUpdater(nets[0], nets[1], log_std.cpu(), lr=1e-6, normalize_advantage=False)
    upd.update(M, batch)
    torch.cuda.synchronize()
    # bit for bit where the tiles have one width; a tile of another may add the same products along k in another order
    near = lambda a, b, tol: float((a - b).abs().max()) <= tol * float(b.abs().max() + b.square().mean().sqrt())
    assert near(nets[0].out[:M], mean, 1e-2) and near(nets[1].out[:M], value, 1e-2)
    d_mean, d_ls, d_value, summary = (torch.empty(M, A, device="cuda"), torch.empty(A, device="cuda"), torch.empty(M, device="cuda"),
                                      torch.empty(6, device="cuda"))
    B.ppo_loss(dict(batch, mean=nets[0].out[:M].contiguous(), value=nets[1].out[:M, 0].contiguous(), log_std=log_std, log_std_old=log_std),
               d_mean, d_ls, d_value, summary, B.ppo_workspace(), 0.2, 2.0, 0.0, True)
    ref[0].backward(d_mean, M)
    ref[1].backward(d_value.view(M, 1), M)
    torch.cuda.synchronize()
    for got, want in zip(nets, ref):
        assert got.device_status() == 0
        for l in range(len(dims) - 1):
            for a, b in ((got.dW[l], want.dW[l]), (got.db[l], want.db[l])):
                # one rounding to bf16 per row slice (2^-9 of a partial sum), other slices on the two sides, and a few
                # activations and dZ entries that round the other way (2^-8 of a sample's share)
                assert float((a - b).norm()) <= 1e-2 * float(b.norm()) + 1e-12, (l, M)
