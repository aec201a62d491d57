"""The policy forward on small batches (narrow tiles) against the same layers on CTA pairs:
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


@pytest.mark.parametrize("dims,dv", [((361, 1024, 512, 28), 1), ((577, 1024, 1024, 512, 69), 3), ((70, 64, 17), 1), ((361, 2048, 1024, 80), 33)])
@pytest.mark.parametrize("n", [1, 128, 129, 1000, 4096, 9600, 20000])
@pytest.mark.parametrize("staged", [False, True])
def test_joint_forward_matches_the_separate_calls(n, dims, dv, staged):
    import torch
    from paper_2609_09821_b200 import binding as B
    wa, wc = W.make_policy_weights(dims, "bf16", 1), W.make_policy_weights(dims[:-1] + (dv,), "bf16", 2)
    A = dims[-1]
    actor = B.Policy(dims, wa["W_bf16"], wa["b"], "bf16", 0.3, 9, n, env_id_base=5)
    critic = B.Policy(dims[:-1] + (dv,), wc["W_bf16"], wc["b"], "bf16", 0.3, 9, n)
    actor.set_log_std(torch.linspace(-2, 0, A, device="cuda"))
    obs = torch.randn(n, B.padded_ld(dims[0]), device="cuda", generator=torch.Generator("cuda").manual_seed(n))

    def outputs():                                   # one guard row behind each
        return [torch.full((n + 1, k), 7.0, device="cuda") for k in (A, A, 1, dv)]
    sep, joint = outputs(), outputs()
    actor.forward(3, obs, *sep[:3], n=n)             # leaves the rows staged
    critic.value_forward(obs, sep[3], n=n)
    for _ in range(2):
        actor.forward_with_value(3, critic, None if staged else obs, *joint, n=n)
    torch.cuda.synchronize()
    assert all(bool((t[n] == 7.0).all()) for t in joint)
    assert actor.device_status() == 0 and critic.device_status() == 0
    for i, (a, b) in enumerate(zip(joint, sep)):
        a, b = a[:n], b[:n]
        if i == 2:
            assert float((a - b).abs().max()) <= 1e-5 * A + 1e-6 * float(b.abs().max())
        else:
            # a tile of another width may add the same products along k in another order: the bounds of the test above
            rms = float(b.square().mean().sqrt())
            assert float((a - b).abs().max()) <= 2e-2 * (float(b.abs().max()) + rms) and float((a - b).norm() / b.norm()) <= 2e-3


def test_joint_forward_runs_nets_of_other_widths_one_after_the_other():
    import torch
    from paper_2609_09821_b200 import binding as B
    n, dims, cdims = 300, (361, 512, 256, 28), (361, 256, 128, 1)
    for dtype in ("bf16", "f32"):
        wa, wc = W.make_policy_weights(dims, dtype, 1), W.make_policy_weights(cdims, dtype, 2)
        key = "W_bf16" if dtype == "bf16" else "W"
        actor, critic = B.Policy(dims, wa[key], wa["b"], dtype, 0.3, 9, n), B.Policy(cdims, wc[key], wc["b"], dtype, 0.3, 9, n)
        obs = torch.randn(n, 384, device="cuda")
        sep, joint = [[torch.empty(n, k, device="cuda") for k in (28, 28, 1, 1)] for _ in range(2)]
        actor.forward(3, obs, *sep[:3])
        critic.value_forward(obs, sep[3])
        actor.forward_with_value(3, critic, obs, *joint)
        assert all(torch.equal(a, b) for a, b in zip(joint, sep))


@pytest.mark.parametrize("dims", [(361, 1024, 512, 28), (577, 1024, 1024, 512, 69), (433, 192, 64, 17)])
@pytest.mark.parametrize("n", [130, 2500, 9001, 20000])
def test_split_batches_are_the_whole_bit_for_bit(n, dims):
    """Tile width, CTA pairs and the critic's place in the actor's launches follow the row count; the results do not."""
    import torch
    from paper_2609_09821_b200 import binding as B
    wa, wc = W.make_policy_weights(dims, "bf16", 1), W.make_policy_weights(dims[:-1] + (1,), "bf16", 2)
    A = dims[-1]
    obs = torch.randn(n, B.padded_ld(dims[0]), device="cuda", generator=torch.Generator("cuda").manual_seed(n))

    def run(base, rows, joint):
        actor = B.Policy(dims, wa["W_bf16"], wa["b"], "bf16", 0.3, 9, rows, env_id_base=base)
        critic = B.Policy(dims[:-1] + (1,), wc["W_bf16"], wc["b"], "bf16", 0.3, 9, rows)
        out = [torch.full((rows, k), 7.0, device="cuda") for k in (A, A, 1, 1)]
        x = obs[base:base + rows]
        if joint:
            actor.forward_with_value(3, critic, x, *out)
        else:
            actor.forward(3, x, *out[:3])
            critic.value_forward(x, out[3])
        torch.cuda.synchronize()
        assert actor.device_status() == 0 and critic.device_status() == 0
        return out

    whole, step = run(0, n, False), (n + 6) // 7
    parts = [run(b, min(step, n - b), b % 2 == 1) for b in range(0, n, step)]
    for i, (a, b) in enumerate(zip(whole, run(0, n, True))):
        assert torch.equal(a, b) and torch.equal(a, torch.cat([p[i] for p in parts]))
