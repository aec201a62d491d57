"""The policy forward on small batches (narrow tiles, several partial accumulators) against the same layers on CTA pairs:
ragged last row blocks, deep and shallow nets, value heads, per-dimension standard deviations, staged input."""
import pytest

from paper_2609_09821_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(361, 1024, 512, 28), (577, 1024, 1024, 512, 69), (361, 2048, 1024, 28), (100, 512, 1),
                                  (64, 512, 512, 512, 512, 512, 512, 80), (361, 256, 256, 17), (70, 64, 40)])
@pytest.mark.parametrize("n", [1, 128, 129, 1000, 2048, 2049, 4096, 4700])
def test_narrow_tiles_match_pairs(n, dims):
    import torch
    from paper_2609_09821_b200 import binding as B
    w = W.make_policy_weights(dims, "bf16", seed=1)
    pols = [B.Policy(dims, w["W_bf16"], w["b"], "bf16", 0.3, 9, n, env_id_base=5, impl=i) for i in (0, 2)]
    A = dims[-1]
    obs = torch.randn(n, B.padded_ld(dims[0]), device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    out = []
    for p in pols:
        got = []
        for ls in (None, torch.linspace(-2, 0, A, device="cuda")):
            p.set_log_std(ls)
            # one guard row behind each output
            mean, act, lp = torch.full((n + 1, A), 7.0, device="cuda"), torch.full((n + 1, A), 7.0, device="cuda"), torch.full((n + 1,), 7.0, device="cuda")
            for rep in range(2):
                p.forward(3, obs, mean, act, lp, n=n)
            val = torch.full((n + 1, A), 7.0, device="cuda")
            p.value_forward(obs, val, n=n)
            torch.cuda.synchronize()
            assert all(bool((t[n] == 7.0).all()) for t in (mean, act, lp, val))
            assert torch.equal(mean[:n], val[:n])
            got += [mean[:n], act[:n], lp[:n]]
        assert p.device_status() == 0
        out.append(got)
    for a, b, kind in zip(*out, ["mean", "action", "logp"] * 2):
        if kind == "logp":
            # sums of A squared normals in another order
            assert float((a - b).abs().max()) <= 1e-5 * A + 1e-6 * float(b.abs().max())
        else:
            # the same products added along k in another order: fp32 rounding, and a few hidden activations that round to the
            # neighbouring bf16 value (2^-8 of one of hundreds of terms)
            rms = float(b.square().mean().sqrt())
            assert float((a - b).abs().max()) <= 2e-2 * (float(b.abs().max()) + rms) and float((a - b).norm() / b.norm()) <= 2e-3


def test_forward_reads_another_policys_rows():
    import torch
    from paper_2609_09821_b200 import binding as B
    n, dims = 700, (361, 512, 256, 28)
    wa, wc = W.make_policy_weights(dims, "bf16", 1), W.make_policy_weights(dims[:-1] + (1,), "bf16", 2)
    actor = B.Policy(dims, wa["W_bf16"], wa["b"], "bf16", 0.3, 9, n)
    critic = B.Policy(dims[:-1] + (1,), wc["W_bf16"], wc["b"], "bf16", 0.3, 9, n)
    obs = torch.randn(n, 384, device="cuda")
    mean, act = torch.empty(n, 28, device="cuda"), torch.empty(n, 28, device="cuda")
    v0, v1 = torch.empty(n, 1, device="cuda"), torch.empty(n, 1, device="cuda")
    critic.value_forward(obs, v0)
    actor.forward(1, obs, mean, act)
    critic.value_forward_staged(n, v1, src=actor)
    assert torch.equal(v0, v1)
