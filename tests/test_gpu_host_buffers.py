"""The host-buffer step with pinned, pageable and mixed buffers: the same numbers whichever way they travel."""
import numpy as np
import pytest

from paper_2609_09821_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 1001, 1504])
def test_pinned_and_pageable_buffers_agree(n):
    import torch
    from paper_2609_09821_b200 import binding as B
    skel, lib = W.make_skeleton("humanoid15", 0), W.make_clip_library(15, 3, (30, 60), 30.0, 0)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    w = W.make_policy_weights((361, 128, 28), "bf16", 0)
    sims = [torch.randn(195, n, generator=torch.Generator().manual_seed(s)) for s in range(3)]
    for s in sims:
        s[2] += 0.6
    out = []
    for pin in ((0, 0, 0, 0), (1, 1, 1, 1), (1, 0, 1, 0), (0, 1, 0, 1)):
        env = B.Env(sk, clips, B.make_env_config(n, 1 / 30, 0, W.REWARD_MULT, 0.3, 384))
        pol = B.Policy((361, 128, 28), w["W_bf16"], w["b"], "bf16", 0.1, 0, n)
        env.attach_policy(pol)
        env.reset_all_host(0)
        m = lambda t, p: t.pin_memory() if p else t
        # results land inside larger pinned arrays, the bytes around them stay as they are
        act, rew, fl = m(torch.full((n, 28), 7.0), pin[1]), m(torch.full((n + 2,), 7.0), pin[2]), m(torch.full((n + 2,), 9, dtype=torch.uint8), pin[3])
        got = []
        for s in range(3):
            B.step_host(env, pol, s + 1, m(sims[s], pin[0]), act, rew[1:], fl[1:])
            got += [act.clone(), rew.clone(), fl.clone()]
            assert rew[0] == 7.0 and rew[-1] == 7.0 and fl[0] == 9 and fl[-1] == 9
        out.append(got)
    assert any(bool((x != 0).any()) for x in out[0][2::3])
    for other in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(out[0], other))


@pytest.mark.parametrize("shift", [1, 2, 3])
def test_pinned_rewards_need_no_alignment(shift):
    """Rewards inside a packed record of the caller's: pinned, but not on a multiple of four bytes."""
    import torch
    from paper_2609_09821_b200 import binding as B
    n = 70
    skel, lib = W.make_skeleton("humanoid15", 0), W.make_clip_library(15, 3, (30, 60), 30.0, 0)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    w = W.make_policy_weights((361, 128, 28), "bf16", 0)
    sim = torch.randn(195, n, generator=torch.Generator().manual_seed(2)).pin_memory()
    out = []
    for off in (0, shift):
        env = B.Env(sk, clips, B.make_env_config(n, 1 / 30, 0, W.REWARD_MULT, 0.3, 384))
        pol = B.Policy((361, 128, 28), w["W_bf16"], w["b"], "bf16", 0.1, 0, n)
        env.attach_policy(pol)
        env.reset_all_host(0)
        raw = torch.full((4 * n + 8,), 9, dtype=torch.uint8).pin_memory()
        act, fl = torch.zeros(n, 28).pin_memory(), torch.zeros(n, dtype=torch.uint8).pin_memory()
        B.step_host(env, pol, 1, sim, act, raw[off:], fl)
        assert bool((raw[:off] == 9).all()) and bool((raw[off + 4 * n:] == 9).all())
        out.append((raw[off:off + 4 * n].clone(), act, fl))
    assert bool((out[0][0] != 9).any()) and all(torch.equal(a, b) for a, b in zip(*out))
