"""fp32 policy layers at the edges of their tiles: row counts around 16 / 32 / 64, widths and depths that are no
multiples of a tile or of four, every choice of tile, action widths of one and of several 32-column groups."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2609_09821_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dims", [
    (1, (5, 3, 2)), (15, (361, 17, 28)), (17, (360, 1024, 512, 28)), (64, (361, 1024, 512, 33)), (65, (259, 130, 69)),
    (300, (577, 1024, 512, 69)), (1025, (362, 1021, 64, 300)), (33, (361, 1023, 530, 28)), (97, (361, 1024, 515, 28)),
    (127, (364, 1013, 260, 3)), (199, (70, 513, 620, 28)), (289, (361, 520, 517, 30)), (313, (1024, 480, 500, 9)),
])
def test_forward_matches_oracle(n, dims):
    import torch
    from paper_2609_09821_b200 import binding as B
    w = W.make_policy_weights(dims, "f32", seed=3)
    pol = B.Policy(dims, w["W"], w["b"], "f32", 0.2, 7, n)
    ld = B.padded_ld(dims[0], 4)
    obs = torch.randn(n, ld, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    mean, action = torch.empty(n, dims[-1], device="cuda"), torch.empty(n, dims[-1], device="cuda")
    logp = torch.empty(n, device="cuda")
    pol.forward(5, obs, mean, action, logp)
    m2 = torch.empty_like(mean)
    pol.forward(5, obs, m2, None)
    torch.cuda.synchronize()
    ref = O.policy_forward(dims, w["W"], w["b"], 0.2, 7, 5, obs[:, :dims[0]].cpu().numpy())
    for got, want, tol in ((mean, ref["mean"], 1e-4), (action, ref["action"], 1e-4)):
        got, want = got.cpu().numpy().astype(np.float64), np.asarray(want, np.float64)
        assert np.all(np.abs(got - want) <= tol * (np.abs(want) + np.sqrt(np.mean(want ** 2))))
    # fp32 sums of A squared normals, each with relative error 2^-23 and the noise's own 1e-6
    lp = np.asarray(ref["logp"], np.float64)
    assert np.all(np.abs(logp.cpu().numpy() - lp) <= 1e-3 + 1e-5 * np.abs(lp))
    assert torch.equal(mean, m2)


@pytest.mark.parametrize("A", [32, 33, 65, 256, 300])
@pytest.mark.parametrize("n", [1, 16, 17, 4001])
def test_log_probabilities_across_a_cluster(n, A):
    """Actions wider than one column tile: the CTAs of a row block send their sums of squares to the first of them, after a
    contraction of eight steps only, launch after launch."""
    import torch
    from paper_2609_09821_b200 import binding as B
    w = W.make_policy_weights((4, 8, A), "f32", seed=3)
    pol = B.Policy((4, 8, A), w["W"], w["b"], "f32", 0.2, 7, n)
    obs = torch.randn(n, 4, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    mean, action = torch.empty(n, A, device="cuda"), torch.empty(n, A, device="cuda")
    logps = torch.full((40, n), 7.0, device="cuda")
    for i in range(40):
        pol.forward(5, obs, mean, action, logps[i])
    ref = O.policy_forward((4, 8, A), w["W"], w["b"], 0.2, 7, 5, obs.cpu().numpy())
    lp = np.asarray(ref["logp"], np.float64)
    assert np.all(np.abs(logps[0].cpu().numpy() - lp) <= 1e-3 + 1e-5 * np.abs(lp))      # (as above)
    assert torch.equal(logps, logps[:1].expand(40, n))


@pytest.mark.parametrize("n,dims", [(129, (361, 1024, 512, 28)), (192, (70, 1009, 60, 5)), (193, (361, 1024, 96, 28)),
                                    (385, (577, 512, 530, 9)), (416, (362, 528, 485, 28)), (417, (40, 512, 28)), (832, (361, 240, 12, 3))])
def test_forward_around_the_largest_one_wave_tile(n, dims):
    test_forward_matches_oracle(n, dims)


@pytest.mark.parametrize("n,dims", [(300, (361, 1024, 512, 28)), (321, (362, 1021, 70, 5)), (384, (577, 1008, 33, 9)), (385, (40, 1000, 64)),
                                    (641, (70, 529, 260, 3)), (833, (5, 432, 40, 3)), (832, (1024, 490, 40, 3))])
def test_forward_on_64_by_48_tiles(n, dims):
    test_forward_matches_oracle(n, dims)
