"""The env step has two kernels, chosen by the number of 32-env tiles.  A batch large enough for the chain kernel must
equal the same envs run in shards small enough for the role kernel (env_id_base), which the oracle tests cover, bit for
bit.  Options, records, wide trees, reward termination, an extended observation too wide to stage."""
import numpy as np
import pytest

from paper_2609_09821_b200 import workloads as W

pytestmark = pytest.mark.gpu
N = 9728            # 304 tiles: more than two per SM; shards of 4864 envs have one or two


def _tree(leaves):
    """Root with `leaves` two-body branches."""
    parents = [-1] + [0] * leaves + list(range(1, leaves + 1))
    g = np.random.default_rng(leaves)
    return dict(parents=np.asarray(parents, np.int32), offsets=g.uniform(-0.3, 0.3, (len(parents), 3)).astype(np.float32),
                masses=None, J=len(parents))


CASES = {
    "plain": dict(),
    "reward": dict(reward=W.REWARD_FIG5, r_min=0.3, write_back=True),
    "aos": dict(aos=True, write_back=True, h_min=0.8),
    "options": dict(options=True, r_min=0.1, reward=W.REWARD_ADD4),
    "aos_options": dict(options=True, aos=True, h_min=0.8),
    "wide_extension": dict(options=True, n_future=8, act_dim=900),
    "many_leaves": dict(leaves=12, options=True, h_min=0.8),
    "too_many_leaves_for_a_warp_each": dict(leaves=15, h_min=0.8),
    "one_chain": dict(leaves=1, h_min=0.8),
    "one_chain_reward": dict(leaves=1, reward=W.REWARD_FIG5, r_min=0.3, write_back=True),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("skeleton", ["humanoid15", "smpl24"])
def test_large_batch_equals_its_shards(name, skeleton):
    import torch
    from paper_2609_09821_b200 import binding as B
    c = CASES[name]
    if c.get("leaves") and skeleton == "smpl24":
        pytest.skip("the tree is the case's own")
    skel = _tree(c["leaves"]) if c.get("leaves") else W.make_skeleton(skeleton, 1)
    J = skel["J"]
    lib = W.make_clip_library(J, 4, (20, 40), 30.0, 1)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    options = c.get("options", False)
    if options:
        clips.set_cyclic([1, 0, 0, 1])
    n_future, act_dim = c.get("n_future", 2), c.get("act_dim", 7)
    extra = (n_future - 1) * 9 * sk.n_ee + act_dim if options else 0
    g = torch.Generator("cuda").manual_seed(3)
    sim = torch.randn(13 * J, N, device="cuda", generator=g) * 0.3
    sim[2] += 0.9
    prev = torch.randn(N, act_dim, device="cuda", generator=g)

    def run(base, n):
        cfg = B.make_env_config(n, 1 / 30, 5, c.get("reward", W.REWARD_MULT), c.get("h_min", 0.3), B.padded_ld(24 * J + 1 + extra),
                                r_min=c.get("r_min", -np.inf), env_id_base=base, write_back_reset=c.get("write_back", False),
                                **(dict(grace_steps=2, reset_noise_std=0.05) if options else {}))
        env = B.Env(sk, clips, cfg)
        acc = torch.zeros(4, dtype=torch.int64, device="cuda")
        if options:
            env.set_obs_extension(n_future, prev[base:base + n])
            env.set_reset_bins(3, np.arange(12, dtype=np.float32).reshape(4, 3))
            env.set_summary(acc)
        obs, rew, fl, terms = env.new_obs(), torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(7, n, device="cuda")
        env.reset_all(obs, 0)
        out = [obs.clone()]
        mine = sim[:, base:base + n].clone()
        for s in range(1, 4):
            if c.get("aos"):
                rec = [mine[a * J:b * J].view(J, b - a, n).permute(2, 0, 1).contiguous() for a, b in ((0, 3), (3, 7), (7, 10), (10, 13))]
                env.step_aos(s, *rec, obs, rew, fl, terms)
                mine = torch.cat([r.permute(1, 2, 0).reshape(-1, n) for r in rec])
            else:
                env.step(s, mine, obs, rew, fl, terms)
            out += [obs.clone(), rew.clone(), fl.clone(), terms.T.clone(), mine.T.clone()]
        out += list(env.get_state()) + [env.get_cycles()]
        assert env.device_status() == 0
        return out, acc

    whole, acc = run(0, N)
    (a, acc_a), (b, acc_b) = run(0, N // 2), run(N // 2, N // 2)
    assert bool((whole[3] != 0).any())
    for x, p, q in zip(whole, a, b):
        assert torch.equal(x, torch.cat([p, q]))
    if options:
        assert torch.equal(acc, acc_a + acc_b)


@pytest.mark.parametrize("records", [False, True])
@pytest.mark.parametrize("tree", ["humanoid15", "smpl24", 15, 31])
@pytest.mark.parametrize("n", [33, 2500, 9000])
def test_writing_reset_states_back_changes_nothing_else(n, tree, records):
    """The reset states go into the arrays that the same launch scores: flags, rewards, observations and terms are those
    of a launch that leaves the arrays alone, with a reward that cannot end an episode and with one that could but never
    does, and the written states are the same in both."""
    import torch
    from paper_2609_09821_b200 import binding as B
    if isinstance(tree, int):
        g = np.random.default_rng(tree)
        skel = dict(parents=np.asarray([-1] + [0] * tree, np.int32), offsets=g.uniform(-0.3, 0.3, (tree + 1, 3)).astype(np.float32), masses=None, J=tree + 1)
    else:
        skel = W.make_skeleton(tree, 1)
    J = skel["J"]
    lib = W.make_clip_library(J, 4, (20, 40), 30.0, 1)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    sims = (torch.randn(8, 13 * J, (n + 3) // 4 * 4, device="cuda", generator=torch.Generator("cuda").manual_seed(n)) * 0.3)[:, :, :n]
    sims[:, 2] += 0.85
    out = []
    for write_back, r_min in ((False, -np.inf), (True, -np.inf), (True, -1.0)):
        cfg = B.make_env_config(n, 1 / 30, 5, W.REWARD_MULT, 0.8, B.padded_ld(24 * J + 1), r_min=r_min, write_back_reset=write_back)
        env = B.Env(sk, clips, cfg)
        obs, rew, fl, terms = env.new_obs(), torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(7, n, device="cuda")
        env.reset_all(obs, 0)
        got, states = [], []
        for s in range(sims.shape[0]):
            if records:
                st = [sims[s, a * J:b * J].reshape(J, b - a, n).permute(2, 0, 1).contiguous() for a, b in ((0, 3), (3, 7), (7, 10), (10, 13))]
                env.step_aos(s + 1, *st, obs, rew, fl, terms)
            else:
                st = [torch.empty_strided((13 * J, n), sims[s].stride(), device="cuda").copy_(sims[s])]
                env.step(s + 1, st[0], obs, rew, fl, terms)
            got += [obs.clone(), rew.clone(), fl.clone(), terms.clone()] + list(env.get_state())
            states += st
        assert env.device_status() == 0
        out.append((got, states))
    assert bool((out[0][0][2] & 1).any()) and not bool((out[0][0][2] & 1).all())
    for got, states in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got, out[0][0]))
    assert all(torch.equal(a, b) for a, b in zip(out[1][1], out[2][1]))
    assert not torch.equal(out[0][1][0], out[1][1][0])


@pytest.mark.parametrize("skeleton", ["humanoid15", "smpl24"])
def test_every_warp_decides_alike_at_the_grace_limit(skeleton):
    """All envs lie below the termination height, half of them have one grace step left: the large batch's flags, state and
    observation rows (each chain's warp writes its own part of a row) are those of its shards, bit for bit."""
    import torch
    from paper_2609_09821_b200 import binding as B
    skel, J = W.make_skeleton(skeleton, 1), {"humanoid15": 15, "smpl24": 24}[skeleton]
    lib = W.make_clip_library(J, 4, (20, 40), 30.0, 1)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    sims = torch.randn(12, 13 * J, N, device="cuda", generator=torch.Generator("cuda").manual_seed(3)) * 0.3
    length = (torch.arange(N, device="cuda", dtype=torch.int32) * 7 % 5)

    def run(base, n):
        env = B.Env(sk, clips, B.make_env_config(n, 1 / 30, 5, W.REWARD_MULT, 10.0, B.padded_ld(24 * J + 1), env_id_base=base, grace_steps=3))
        obs, rew, fl = env.new_obs(), torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda")
        env.reset_all(obs, 0)
        env.set_state(ep_len=length[base:base + n].contiguous())
        out, want = [], length[base:base + n].clone()
        for s in range(sims.shape[0]):
            env.step(s + 1, sims[s, :, base:base + n].contiguous(), obs, rew, fl)
            assert torch.equal((fl & 1) != 0, want >= 3)
            want = torch.where(fl != 0, 0, want + 1)
            assert torch.equal(env.get_state()[2], want)
            out += [obs.clone(), rew.clone(), fl.clone()] + list(env.get_state()[:2])
        return out

    for whole, a, b in zip(run(0, N), run(0, N // 2), run(N // 2, N // 2)):
        assert torch.equal(whole, torch.cat([a, b]))


@pytest.mark.parametrize("options", [False, True])
@pytest.mark.parametrize("tree", ["humanoid15", "smpl24", 1, 9])
@pytest.mark.parametrize("n", [9472, 9473, 18944, 18945])
def test_reset_of_all_envs_equals_its_shards(n, tree, options):
    """Row counts on either side of what fits the SMs at once with two and with four CTAs each; shards of one CTA per SM."""
    import torch
    from paper_2609_09821_b200 import binding as B
    skel = W.make_skeleton(tree, 1) if isinstance(tree, str) else _tree(tree)
    J = skel["J"]
    lib = W.make_clip_library(J, 4, (20, 40), 30.0, 1)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    if options:
        clips.set_cyclic([1, 0, 0, 1])
    extra = 2 * 9 * sk.n_ee + 7 if options else 0

    def run(base, n):
        env = B.Env(sk, clips, B.make_env_config(n, 1 / 30, 5, W.REWARD_MULT, 0.3, B.padded_ld(24 * J + 1 + extra), env_id_base=base,
                                                 **(dict(grace_steps=2, reset_noise_std=0.05) if options else {})))
        if options:
            env.set_obs_extension(3, torch.ones(n, 7, device="cuda"))
            env.set_reset_bins(3, np.arange(12, dtype=np.float32).reshape(4, 3))
        obs = torch.full((n, env.ld_obs), 7.0, device="cuda")
        env.reset_all(obs, 3)
        starts = env.reset_stats()[0] if options else None
        return [obs] + list(env.get_state()), starts

    whole, starts = run(0, n)
    parts = [run(b, min(4736, n - b)) for b in range(0, n, 4736)]
    for i, x in enumerate(whole):
        assert torch.equal(x, torch.cat([p[0][i] for p in parts]))
    if options:
        assert torch.equal(starts, sum(p[1] for p in parts))


@pytest.mark.parametrize("staged", [False, True])
@pytest.mark.parametrize("skeleton", ["humanoid15", "smpl24"])
@pytest.mark.parametrize("n", [41, 4801, N])
def test_records_equal_rows(n, skeleton, staged):
    """The simulator's records, read in place or staged, and the transposed data as rows: one result, bit for bit."""
    import torch
    from paper_2609_09821_b200 import binding as B
    skel = W.make_skeleton(skeleton, 1)
    J = skel["J"]
    lib = W.make_clip_library(J, 4, (20, 40), 30.0, 1)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    sims = (torch.randn(4, 13 * J, (n + 3) // 4 * 4, device="cuda", generator=torch.Generator("cuda").manual_seed(n)) * 0.3)[:, :, :n]
    sims[:, 2] += 0.9
    out = []
    for records in (False, True):
        env = B.Env(sk, clips, B.make_env_config(n, 1 / 30, 5, W.REWARD_MULT, 0.8, B.padded_ld(24 * J + 1), write_back_reset=True))
        env.set_aos_staging(staged and records)
        obs, rew, fl, terms = env.new_obs(), torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(7, n, device="cuda")
        env.reset_all(obs, 0)
        got = []
        for s in range(sims.shape[0]):
            if records:
                rec = [sims[s, a * J:b * J].reshape(J, b - a, n).permute(2, 0, 1).contiguous() for a, b in ((0, 3), (3, 7), (7, 10), (10, 13))]
                env.step_aos(s + 1, *rec, obs, rew, fl, terms)
                sim = torch.cat([r.permute(1, 2, 0).reshape(-1, n) for r in rec])
            else:
                sim = torch.empty_strided((13 * J, n), sims[s].stride(), device="cuda").copy_(sims[s])
                env.step(s + 1, sim, obs, rew, fl, terms)
            got += [obs.clone(), rew.clone(), fl.clone(), terms.clone(), sim] + list(env.get_state())
        out.append(got)
    assert bool((out[0][2] & 1).any())
    assert all(torch.equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("options", [False, True])
@pytest.mark.parametrize("skeleton", ["humanoid15", "smpl24", 1])
@pytest.mark.parametrize("n", [41, 4801, N - 95])
def test_records_a_power_of_two_apart_equal_rows(n, skeleton, options):
    """Records whose envs lie a multiple of 256 bytes apart are staged before the walk; ragged last tiles, one and several tiles
    per SM, a single chain."""
    import torch
    from paper_2609_09821_b200 import binding as B
    skel = _tree(skeleton) if skeleton == 1 else W.make_skeleton(skeleton, 1)
    J, extra = skel["J"], 0
    lib = W.make_clip_library(J, 4, (20, 40), 30.0, 1)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    if options:
        extra = 2 * 9 * sk.n_ee
    sims = (torch.randn(3, 13 * J, (n + 3) // 4 * 4, device="cuda", generator=torch.Generator("cuda").manual_seed(n)) * 0.3)[:, :, :n]
    sims[:, 2] += 0.9
    out = []
    for records in (False, True):
        env = B.Env(sk, clips, B.make_env_config(n, 1 / 30, 5, W.REWARD_MULT, 0.8, B.padded_ld(24 * J + 1 + extra), write_back_reset=True,
                                                 **(dict(grace_steps=2, reset_noise_std=0.05) if options else {})))
        if options:
            env.set_obs_extension(3)
        obs, rew, fl, terms = env.new_obs(), torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(7, n, device="cuda")
        env.reset_all(obs, 0)
        got = []
        for s in range(sims.shape[0]):
            if records:
                rec = []
                for a, b in ((0, 3), (3, 7), (7, 10), (10, 13)):
                    w = b - a
                    wide = torch.zeros(n, (w * J + 63) // 64 * 64, device="cuda")
                    view = wide[:, :w * J].unflatten(1, (J, w))
                    view.copy_(sims[s, a * J:b * J].reshape(J, w, n).permute(2, 0, 1))
                    rec.append(view)
                env.step_aos(s + 1, *rec, obs, rew, fl, terms)
                sim = torch.cat([r.permute(1, 2, 0).reshape(-1, n) for r in rec])
            else:
                sim = torch.empty_strided((13 * J, n), sims[s].stride(), device="cuda").copy_(sims[s])
                env.step(s + 1, sim, obs, rew, fl, terms)
            got += [obs.clone(), rew.clone(), fl.clone(), terms.clone(), sim] + list(env.get_state())
        out.append(got)
    assert any(bool((fl & 1).any()) for fl in out[0][2::8])        # (in some step: with options the first two are grace steps)
    assert all(torch.equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("leaves,bodies,n,case", [
    (4, 26, 16384, dict(h_min=0.8)),
    (3, 21, 20000, dict(reward=W.REWARD_FIG5, r_min=0.3, write_back=True)),
    (5, 25, 16384, dict(options=True, h_min=0.8)),
    (10, 31, 12000, dict(h_min=0.8)),
    (10, 31, 12000, dict(options=True, r_min=0.1, reward=W.REWARD_ADD4)),
])
def test_trees_whose_rotations_are_not_staged(leaves, bodies, n, case, monkeypatch):
    """Trees of which an SM holds a CTA more without them, at sizes where that saves a wave; half of the envs fit one wave."""
    parents = np.asarray([-1] + [max(j - leaves, 0) for j in range(1, bodies)], np.int32)
    offsets = np.random.default_rng(leaves).uniform(-0.3, 0.3, (bodies, 3)).astype(np.float32)
    monkeypatch.setitem(globals(), "_tree", lambda _: dict(parents=parents, offsets=offsets, masses=None, J=bodies))
    monkeypatch.setitem(globals(), "N", n)
    monkeypatch.setitem(CASES, "tree", dict(case, leaves=leaves))
    test_large_batch_equals_its_shards("tree", "humanoid15")


@pytest.mark.parametrize("case", [dict(h_min=0.8), dict(reward=W.REWARD_FIG5, r_min=0.3, write_back=True), dict(aos=True, h_min=0.8)])
def test_trees_with_two_chains(case, monkeypatch):
    monkeypatch.setitem(CASES, "two_chains", dict(case, leaves=2))
    test_large_batch_equals_its_shards("two_chains", "humanoid15")


@pytest.mark.parametrize("form", ["plain", "reward", "extension", "rotations_only", "positions_only"])
@pytest.mark.parametrize("skeleton", ["humanoid15", "smpl24"])
@pytest.mark.parametrize("n", [41, 4700, 4801, N - 95])
def test_staged_records_equal_rows_in_every_form(n, skeleton, form):
    """Staged records of a step that leaves the states alone (no barrier before the decision), of one whose reward ends episodes, with
    an extension too wide to stage, and where the envs of one of the arrays alone lie a multiple of 256 bytes apart."""
    import torch
    from paper_2609_09821_b200 import binding as B
    skel = W.make_skeleton(skeleton, 1)
    J = skel["J"]
    lib = W.make_clip_library(J, 4, (20, 40), 30.0, 1)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    reward, extension = form == "reward", form == "extension"
    extra = 7 * 9 * sk.n_ee + 900 if extension else 0
    g = torch.Generator("cuda").manual_seed(n)
    sims = (torch.randn(3, 13 * J, (n + 3) // 4 * 4, device="cuda", generator=g) * 0.3)[:, :, :n]
    sims[:, 2] += 0.9
    prev = torch.randn(n, 900, device="cuda", generator=g)
    out = []
    for records in (False, True):
        env = B.Env(sk, clips, B.make_env_config(n, 1 / 30, 5, W.REWARD_FIG5 if reward else W.REWARD_MULT, 0.3 if reward else 0.8,
                                                 B.padded_ld(24 * J + 1 + extra), r_min=0.3 if reward else -np.inf))
        if extension:
            env.set_obs_extension(8, prev)
        obs, rew, fl, terms = env.new_obs(), torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(7, n, device="cuda")
        env.reset_all(obs, 0)
        got = []
        for s in range(sims.shape[0]):
            if records:
                rec = []
                for i, (a, b) in enumerate(((0, 3), (3, 7), (7, 10), (10, 13))):
                    w, crowded = b - a, i == dict(positions_only=0, rotations_only=1).get(form, i)
                    wide = torch.zeros(n, (w * J + 63) // 64 * 64 + (0 if crowded else 4), device="cuda")
                    view = wide[:, :w * J].unflatten(1, (J, w))
                    view.copy_(sims[s, a * J:b * J].reshape(J, w, n).permute(2, 0, 1))
                    rec.append(view)
                env.step_aos(s + 1, *rec, obs, rew, fl, terms)
            else:
                env.step(s + 1, torch.empty_strided((13 * J, n), sims[s].stride(), device="cuda").copy_(sims[s]), obs, rew, fl, terms)
            got += [obs.clone(), rew.clone(), fl.clone(), terms.clone()] + list(env.get_state())
        assert env.device_status() == 0
        out.append(got)
    assert any(bool((fl & 1).any()) for fl in out[0][2::7])
    assert all(torch.equal(a, b) for a, b in zip(*out))
