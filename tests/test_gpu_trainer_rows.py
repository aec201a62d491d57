"""Backward pass on row counts that split unevenly: the dW products share whole 64-row blocks out over slices, so
the slices of one product differ by a block; one block, fewer blocks than slices, primes of blocks."""
import numpy as np
import pytest

from paper_2609_09821_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [64, 192, 64 * 13, 64 * 61, 64 * 250])
@pytest.mark.parametrize("dims", [(361, 1024, 512, 28), (70, 64, 320, 1), (577, 256, 256, 69)])
def test_backward_matches_fp64(M, dims):
    import torch
    from paper_2609_09821_b200 import trainer as T
    w = W.make_policy_weights(dims, "bf16", seed=5)
    tr = T.MlpTrainer(dims, w["W"], w["b"], 64 * 250)
    g = torch.Generator("cuda").manual_seed(M)
    x = torch.randn(M, dims[0], device="cuda", generator=g).to(torch.bfloat16)
    d_out = torch.randn(M, dims[-1], device="cuda", generator=g) / M
    rows = tr.input_rows(M)
    rows.zero_()
    rows[:, :dims[0]] = x
    tr.forward(M)
    tr.backward(d_out, M)
    torch.cuda.synchronize()
    assert tr.device_status() == 0
    bf = lambda t: t.to(torch.float32).to(torch.bfloat16).double()
    nl = len(dims) - 1
    Wd = [torch.from_numpy(a).cuda().double() for a in w["W"]]
    # the trainer's own activations: a rounding that makes one unit of one sample positive or not moves a gradient
    # entry by that sample's whole share, which at 64 rows is no small part of it
    H = [x.double()] + [tr._tensor(T._H, l)[:M].double() for l in range(1, nl)]
    for l in range(nl - 1):
        z = bf((H[l] @ Wd[l].T + torch.from_numpy(w["b"][l]).cuda().double()).clamp_min(0))
        assert float(((H[l + 1] - z).abs() / (z.abs() + z.square().mean().sqrt())).max()) < 2e-2
    dz = d_out.double()
    for l in reversed(range(nl)):
        q = bf(dz)
        for got, want in ((tr.dW[l], q.T @ H[l]), (tr.db[l], dz.sum(0))):
            rms = want.square().mean().sqrt()
            # dZ's roundings to bf16 that fall the other way (2^-8 of a sample's share each) and one rounding to bf16
            # per slice (2^-9 of a partial sum): standard deviations of 2^-9 rms, five of them 1e-2
            assert float(((got.double() - want).abs() / (want.abs() + rms)).max()) < 2e-2, (l, M)
        if l:
            dz = (q @ Wd[l]) * (H[l] > 0)


@pytest.mark.parametrize("M,A", [(64, 28), (64 * 61, 1), (64 * 61, 80), (1 << 20, 28)])
def test_bias_gradients_are_rounded_once(M, A):
    """Whole numbers whose sums over 1024 rows fit fp32: the sum over the batch is exact but for its one rounding, however
    many rows there are."""
    import torch
    from paper_2609_09821_b200 import trainer as T
    w = W.make_policy_weights((64, 64, A), "f32", seed=5)
    tr = T.MlpTrainer((64, 64, A), w["W"], w["b"], M)
    d_out = 2 * torch.randint(-2 ** 11, 2 ** 13, (M, A), device="cuda", generator=torch.Generator("cuda").manual_seed(M + A)) + 1
    tr.input_rows(M).zero_()
    tr.forward(M)
    tr.backward(d_out.float(), M)
    assert torch.equal(tr.db[1], d_out.sum(0).float()) and tr.device_status() == 0
