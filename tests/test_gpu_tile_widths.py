"""Hidden-layer products at row counts on either side of the points where the tile width changes (one wave of 64-,
128- and 256-column tiles on 148 SMs, then several waves), with ragged last row tiles: forward, and the backward
product with its ReLU mask and column sums."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 127, 1024, 1152, 1153, 2304, 2305, 4736, 4737])
@pytest.mark.parametrize("N,K", [(1024, 384), (512, 1024), (192, 128)])
def test_forward_product(M, N, K):
    import torch
    from paper_2609_09821_b200 import binding as B
    g = torch.Generator("cuda").manual_seed(M)
    # small integers: exact in bf16 operands, fp32 sums and (below 256) the bf16 output
    a = torch.randint(-2, 3, (M, K), device="cuda", generator=g).float() * (torch.rand(M, K, device="cuda", generator=g) < 0.1)
    w = torch.randint(-2, 3, (N, K), device="cuda", generator=g).float() * (torch.rand(N, K, device="cuda", generator=g) < 0.1)
    bias = torch.randint(-3, 4, (N,), device="cuda", generator=g).float()
    c = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.gemm_bf16(a.bfloat16(), w.bfloat16(), c[:M], bias, True, status)
    assert torch.equal(c[:M].float(), torch.relu(a @ w.T + bias))
    assert bool((c[M] == 7.0).all()) and status.item() == 0


@pytest.mark.parametrize("M", [32, 1152, 1184, 2336, 4768])
def test_backward_product(M):
    import torch
    from paper_2609_09821_b200 import binding as B
    N, K = 1024, 128
    g = torch.Generator("cuda").manual_seed(M)
    dz = torch.randint(-2, 3, (M, K), device="cuda", generator=g).float()
    wt = torch.randint(-1, 2, (N, K), device="cuda", generator=g).float() * (torch.rand(N, K, device="cuda", generator=g) < 0.3)
    h = torch.randint(-1, 2, (M, N), device="cuda", generator=g).bfloat16()
    dh = torch.zeros(M, N, dtype=torch.bfloat16, device="cuda")
    part = torch.zeros(M // 32, N, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.gemm_bf16_dgrad(dz.bfloat16(), wt.bfloat16(), dh, h, part, status)
    want = (dz @ wt.T) * (h > 0)
    assert torch.equal(dh.float(), want)
    assert torch.equal(part, want.view(M // 32, 32, N).sum(1)) and status.item() == 0
