"""The work that users of this library have it do, as timed cases.

A case is a dict of plain values; `prepare` builds what a program holds before the calls (handles, weights,
input arrays on the GPU), `run` makes one pass through the public entry points, `work` states the bytes and
operations that the pass cannot do without.  Four kinds of pass:

  rollout   T control steps from fresh episodes: policy forward on the current observation, then the env step
            on that step's simulated body states (the per-step loop of a DeepMimic-style trainer, or of an
            evaluation run), every call on a CUDA stream as a training script issues it
  collect   the same loop with a critic, rollout storage and advantage estimation, captured once in a CUDA
            graph and replayed
  update    the PPO update over a stored rollout: epochs x minibatches of actor and critic
  host      rollout steps for a simulator that lives in host memory (one call per step, buffers pinned)
  act       one action for a handful of characters from caller-owned fp32 weights, without any allocation

Every pass starts its episodes again with the same reset draws, so a pass can be repeated; an update pass
carries on training from where the last one ended.
"""
import math

import numpy as np
import torch

from paper_2609_09821_b200 import binding as B
from paper_2609_09821_b200 import rollout as R
from paper_2609_09821_b200 import trainer as TR
from paper_2609_09821_b200 import workloads as W

NETS = {                      # hidden widths of the benchmark configurations
    "1024-512": (1024, 512),
    "2048-1024": (2048, 1024),
    "1024-1024-512": (1024, 1024, 512),
}
ACTIONS = {"humanoid15": 28, "smpl24": 69}
BODIES = {"humanoid15": 15, "smpl24": 24}


def listed():
    return [
        # the 64-env fp32 configuration: a debugging run or a handful of characters; latency and launches count
        dict(name="rollout_64_f32", kind="rollout", envs=64, steps=8, skeleton="humanoid15", clips=1, net="1024-512",
             dtype="f32", sim="rows", staged=False, options=False, resets="few"),
        # one motion, 4096 envs: the usual single-clip training run
        dict(name="rollout_4096", kind="rollout", envs=4096, steps=8, skeleton="humanoid15", clips=1, net="1024-512",
             dtype="bf16", sim="rows", staged=True, options=False, resets="few"),
        # a clip library at 16384 envs
        dict(name="rollout_16384_library", kind="rollout", envs=16384, steps=8, skeleton="humanoid15", clips=32, net="1024-512",
             dtype="bf16", sim="rows", staged=True, options=False, resets="few"),
        # the benchmark's headline configuration: 24-body character, 65536 envs
        dict(name="rollout_65536_smpl24", kind="rollout", envs=65536, steps=4, skeleton="smpl24", clips=32, net="1024-1024-512",
             dtype="bf16", sim="rows", staged=True, options=False, resets="few"),
        # early training: 10-30 % of the envs fall and are reset in every step; wide first layer
        dict(name="rollout_16384_resets", kind="rollout", envs=16384, steps=8, skeleton="humanoid15", clips=32, net="2048-1024",
             dtype="bf16", sim="rows", staged=True, options=False, resets="many"),
        # an env count that is a multiple of nothing, with the optional semantics on: extended observation, looped
        # clips, reset bins, motion noise, grace steps, summaries, the additive reward with its threshold
        dict(name="rollout_9001_options", kind="rollout", envs=9001, steps=4, skeleton="smpl24", clips=32, net="1024-512",
             dtype="bf16", sim="rows", staged=False, options=True, resets="few"),
        # a simulator's own arrays of structures read where they are, 12000 envs
        dict(name="rollout_12000_aos", kind="rollout", envs=12000, steps=4, skeleton="humanoid15", clips=32, net="1024-512",
             dtype="bf16", sim="aos", staged=True, options=False, resets="few"),
        # a whole rollout of the training loop (actor, critic, storage, GAE) replayed from one CUDA graph
        dict(name="collect_4096x32", kind="collect", envs=4096, steps=32, skeleton="humanoid15", clips=1, net="1024-512",
             staged=True, resets="few"),
        # the update phase of a small run: 64000 samples, shuffled, 2 epochs x 4 minibatches of 16000 rows
        dict(name="update_64x1000_shuffled", kind="update", envs=1000, steps=64, skeleton="humanoid15", net="1024-512",
             epochs=2, minibatches=4, shuffled=True),
        # one large minibatch of the headline configuration's networks: 131072 contiguous rows
        dict(name="update_131072_smpl24", kind="update", envs=16384, steps=8, skeleton="smpl24", net="1024-1024-512",
             epochs=1, minibatches=1, shuffled=False),
        # a CPU simulator: every step's body states come from pinned host memory, actions and rewards go back
        dict(name="host_4096", kind="host", envs=4096, steps=4, skeleton="humanoid15", clips=1, net="1024-512", resets="few"),
        # deployment: actions for 300 characters inside a process that may not allocate
        dict(name="act_300_f32", kind="act", envs=300, skeleton="humanoid15", net="1024-512"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rollout", "rollout", "rollout", "rollout", "collect", "update", "update", "host", "act"])
    skeleton = rng.choice(["humanoid15", "smpl24"])
    net = rng.choice(sorted(NETS))
    clips = rng.choice([1, 8, 32])
    resets = rng.choice(["few", "few", "many"])
    if kind == "rollout":
        dtype = rng.choice(["bf16", "bf16", "bf16", "bf16", "f32"])
        envs = _log_int(rng, 32, 2048) if dtype == "f32" else _log_int(rng, 64, 65000)
        steps = 4 if envs > 16384 else 8
        return dict(kind=kind, envs=envs, steps=steps, skeleton=skeleton, clips=clips, net="1024-512" if dtype == "f32" or envs > 16384 else net,
                    dtype=dtype, sim=rng.choice(["rows", "rows", "rows", "aos", "aos_staged"]),
                    staged=dtype == "bf16" and rng.random() < 0.75, **rng.choice([dict(options=False, resets=resets)] * 3 + [dict(options=True, resets="few")]))
    if kind == "collect":
        envs = _log_int(rng, 64, 2048) * 4                    # storage rows start on 16-byte boundaries
        return dict(kind=kind, envs=envs, steps=rng.choice([16, 32]), skeleton=skeleton, clips=clips, net="1024-512",
                    staged=rng.random() < 0.5, resets=resets)
    if kind == "update":
        envs = _log_int(rng, 32, 2000)                        # 64 steps: any env count gives whole 64-row minibatches
        return dict(kind=kind, envs=envs, steps=64, skeleton=skeleton, net="1024-512" if envs > 1000 else net,
                    epochs=1, minibatches=rng.choice([1, 2]) if envs % 2 == 0 else 1, shuffled=rng.random() < 0.5)
    if kind == "host":
        return dict(kind=kind, envs=_log_int(rng, 64, 32768), steps=2, skeleton=skeleton, clips=clips, net="1024-512", resets=resets)
    return dict(kind=kind, envs=rng.randrange(1, 1025), skeleton=skeleton, net="1024-512")


# ---------------------------------------------------------------------------------------------- shapes
def _ext(case):
    """Columns of the extended observation: one further frame of 5 end effectors' targets, the previous action."""
    return (9 * 5 + ACTIONS[case["skeleton"]]) if case.get("options") else 0


def _dims(case, out=None):
    A = ACTIONS[case["skeleton"]]
    return (24 * BODIES[case["skeleton"]] + 1 + _ext(case),) + NETS[case["net"]] + (A if out is None else out,)


def _workload(case, seed):
    """A benchmark workload of this case's shape: noise levels and termination height as in the configurations."""
    many = case.get("resets") == "many"
    return W.Workload("case", case["envs"], case["skeleton"], case.get("clips", 1), (60, 600) if case.get("clips", 1) > 1 else (150, 150),
                      case.get("steps", 1), _dims(case), case.get("dtype", "bf16"), sigma_q=0.3 if many else 0.05,
                      h_min=0.8 if many else 0.3, seed=seed)


# ---------------------------------------------------------------------------------------------- preparation
_STREAMS = []


def _stream():
    """The stream of the program: one for everything, so that passes follow one another as a training loop's do."""
    if not _STREAMS:
        _STREAMS.append(torch.cuda.Stream())
    return _STREAMS[0]


def _scene(case, seed, stream):
    """Skeleton, clip library and env of a case."""
    wl = _workload(case, seed)
    skel, lib = W.make_skeleton(wl.skeleton, seed), W.make_clip_library(BODIES[wl.skeleton], wl.n_clips, wl.frames, wl.fps, seed)
    sk = B.Skeleton(skel["parents"], skel["offsets"], skel["masses"])
    clips = B.Clips(sk, lib["n_frames"], lib["fps"], lib["root_pos"], lib["local_quat"])
    options = case.get("options", False)
    more = dict(r_min=0.15, grace_steps=2, reset_noise_std=0.02) if options else {}
    cfg = B.make_env_config(wl.n_envs, wl.dt, seed, W.REWARD_FIG5 if options else W.REWARD_MULT, wl.h_min,
                            B.padded_ld(24 * sk.J + 1 + _ext(case)), **more)
    if options:
        clips.set_cyclic([i % 2 for i in range(wl.n_clips)])
    env = B.Env(sk, clips, cfg, stream=stream)
    return wl, skel, lib, env


def _policy(dims, dtype, seed, rows, stream):
    w = W.make_policy_weights(dims, dtype, seed)
    return B.Policy(dims, w["W_bf16"] if dtype == "bf16" else w["W"], w["b"], dtype, 0.1, seed, rows, stream=stream)


def _sims(wl, skel, lib, env, obs, reward, flags, seed):
    """Body states of every step, [13 J, N] with rows padded to 16 bytes: the simulator stand-in follows each env's
    clip and time."""
    n_pad = (wl.n_envs + 3) // 4 * 4
    env.reset_all(obs, 0)

    def pad(sim):
        out = torch.zeros((sim.shape[0], n_pad), device="cuda")
        out[:, :sim.shape[1]] = sim
        return out[:, :sim.shape[1]]

    sims = []
    for s in range(1, wl.steps + 1):
        cid, t, _ = env.get_state()
        sim = pad(W.synth_sim_state_torch(skel, lib, cid.to(torch.int64), t.to(torch.float64) + wl.dt, s, wl, seed=seed % (1 << 20)))
        torch.cuda.synchronize()
        env.step(s, sim, obs, reward, flags)
        sims.append(sim)
    torch.cuda.synchronize()
    return sims


def _records(sim, J):
    """The same states as a simulator's arrays of structures: a leading world body, spatial velocities (six floats)."""
    n = sim.shape[1]
    pos, quat, vel = (torch.zeros((n, J + 1, c), device="cuda") for c in (3, 4, 6))
    pos[:, 1:] = sim[:3 * J].reshape(J, 3, n).permute(2, 0, 1)
    quat[:, 1:] = sim[3 * J:7 * J].reshape(J, 4, n).permute(2, 0, 1)
    vel[:, 1:, :3] = sim[7 * J:10 * J].reshape(J, 3, n).permute(2, 0, 1)
    vel[:, 1:, 3:] = sim[10 * J:].reshape(J, 3, n).permute(2, 0, 1)
    return pos[:, 1:], quat[:, 1:], vel[:, 1:, :3], vel[:, 1:, 3:]


def _prepare_rollout(case, seed):
    stream = _stream()
    with torch.cuda.stream(stream):
        wl, skel, lib, env = _scene(case, seed, stream)
        n, A, T = wl.n_envs, wl.act_dim, wl.steps
        st = dict(case=case, stream=stream, env=env, obs=env.new_obs(), mean=torch.zeros((n, A), device="cuda"),
                  action=torch.zeros((n, A), device="cuda"), logp=torch.zeros(n, device="cuda"),
                  rewards=torch.zeros((T, n), device="cuda"), flagss=torch.zeros((T, n), dtype=torch.uint8, device="cuda"),
                  terms=torch.zeros((7, n), device="cuda") if case["options"] else None)
        if case["options"]:
            env.set_obs_extension(2, st["action"])
            env.set_reset_bins(8, np.random.default_rng(seed).random((wl.n_clips, 8)).astype(np.float32) + 0.1)
            env.set_summary(torch.zeros(4, dtype=torch.int64, device="cuda"))
        policy = _policy(wl.mlp_dims, wl.mlp_dtype, seed, n, stream)
        if case["staged"]:
            env.attach_policy(policy)
        st.update(reward=list(st["rewards"]), flags=list(st["flagss"]))       # one row per step
        sims = _sims(wl, skel, lib, env, st["obs"], st["reward"][0], st["flags"][0], seed)
        if case["sim"] != "rows":
            env.set_aos_staging(case["sim"] == "aos_staged")
            sims = [_records(s, env.J) for s in sims]
    torch.cuda.synchronize()
    st.update(policy=policy, sims=sims)
    return st


def _run_rollout(st):
    case, env, policy, n = st["case"], st["env"], st["policy"], st["case"]["envs"]
    obs, mean, action, logp, reward, flags = (st[k] for k in ("obs", "mean", "action", "logp", "reward", "flags"))
    env.reset_all(obs, 0)
    for s in range(1, case["steps"] + 1):
        if case["staged"]:
            policy.forward_staged(s, n, mean, action, logp)
        else:
            policy.forward(s, obs, mean, action, logp)
        sim = st["sims"][s - 1]
        if case["sim"] == "rows":
            env.step(s, sim, obs, reward[s - 1], flags[s - 1], st["terms"])
        else:
            env.step_aos(s, *sim, obs, reward[s - 1], flags[s - 1], st["terms"])
    return dict(obs=obs, mean=mean, action=action, logp=logp, reward=st["rewards"], flags=st["flagss"], terms=st["terms"])


def _prepare_collect(case, seed):
    stream = _stream()
    with torch.cuda.stream(stream):
        wl, skel, lib, env = _scene(case, seed, stream)
        n, A, T = wl.n_envs, wl.act_dim, wl.steps
        actor = _policy(wl.mlp_dims, "bf16", seed, n, stream)
        critic = _policy(_dims(case, 1), "bf16", seed + 1, n, stream)
        if case["staged"]:
            env.attach_policy(actor)
        store = R.RolloutStorage(T, n, A, env.ld_obs)
        sims = _sims(wl, skel, lib, env, store.obs_row(0), store.reward[0], store.flags[0], seed)

        def whole():
            env.reset_all(store.obs_row(0), 0)
            R.collect(env, actor, critic, store, lambda s: sims[s - 1], 1, 0.99, 0.95, staged=case["staged"])

        whole()                                              # first calls set kernels up; not inside a capture
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            whole()
    torch.cuda.synchronize()
    return dict(case=case, stream=stream, env=env, actor=actor, critic=critic, store=store, sims=sims, graph=graph)


def _run_collect(st):
    with torch.cuda.stream(st["stream"]):
        st["graph"].replay()
    s = st["store"]
    return dict(obs=s.obs, action=s.action, mean=s.mean, logp=s.logp, value=s.value, reward=s.reward, flags=s.flags,
                advantage=s.advantage, returns=s.returns)


def _net(w, b, x):
    """The network with bf16 operands and fp32 sums (what the behaviour policy's means and values come from)."""
    bf = lambda t: t.to(torch.bfloat16).float()
    for l in range(len(w)):
        x = torch.addmm(torch.from_numpy(b[l]).cuda(), bf(x), bf(torch.from_numpy(w[l]).cuda()).T)
        x = torch.relu(x) if l + 1 < len(w) else x
    return x


class _Kept(dict):
    """Outputs that are arrays of the library's handles: they live as long as the state that owns them."""


def _prepare_update(case, seed):
    stream = _stream()
    with torch.cuda.stream(stream):
        wl, skel, lib, env = _scene(dict(case, clips=32), seed, stream)
        n, A, T, D = wl.n_envs, wl.act_dim, wl.steps, env.D
        wa, wc = W.make_policy_weights(_dims(case), "f32", seed), W.make_policy_weights(_dims(case, 1), "f32", seed + 1)
        rows = T * n // case["minibatches"]
        actor, critic = TR.MlpTrainer(_dims(case), wa["W"], wa["b"], rows, stream=stream), TR.MlpTrainer(_dims(case, 1), wc["W"], wc["b"], rows, stream=stream)
        # (a small, capped learning rate: every pass then trains on much the same network)
        upd = TR.PpoUpdater(actor, critic, torch.full((A,), -1.0), lr=3e-8, lr_min=1e-8, lr_max=3e-8)
        store = R.RolloutStorage(T, n, A, env.ld_obs)
        g = torch.Generator(device="cuda").manual_seed(seed)
        rnd = lambda *sh: torch.randn(*sh, device="cuda", generator=g)
        for t in range(T):                                   # observations of random clips and phases
            env.reset_all(store.obs[t], t)
        for t in range(T):                                   # what the behaviour policy and critic said about them
            x = store.obs[t, :, :D]
            store.mean[t] = _net(wa["W"], wa["b"], x)
            store.value[t] = _net(wc["W"], wc["b"], x)[:, 0]
        z, u = rnd(T, n, A), rnd(A)                          # some directions of the action paid off
        store.action.copy_(store.mean + math.exp(-1.0) * z)
        store.logp.copy_(-0.5 * z.square().sum(2) + A * 1.0 - 0.5 * A * math.log(2 * math.pi))
        store.returns.copy_(store.value[:T] + rnd(T, n))
        store.advantage.copy_(z @ (2.0 * u / u.norm()) + 0.5 * rnd(T, n) + 0.3)
        perm = None
        if case["shuffled"]:
            perm = torch.stack([torch.randperm(T * n, device="cuda", generator=g) for _ in range(case["epochs"])]).to(torch.int32)
    torch.cuda.synchronize()
    return dict(case=case, stream=stream, actor=actor, critic=critic, upd=upd, store=store, perm=perm)


def _run_update(st):
    case, upd = st["case"], st["upd"]
    TR.update_from_storage(upd, st["store"], case["epochs"], case["minibatches"], st["perm"])
    nets = (st["actor"], st["critic"])
    out = _Kept(W=[t.W for t in nets], b=[t.b for t in nets], mW=[t.mW for t in nets], mb=[t.mb for t in nets],
                log_std=upd.log_std, lr=upd.lr, summary=upd.summary)
    out.owner = st
    return out


def _prepare_host(case, seed):
    stream = _stream()
    with torch.cuda.stream(stream):
        wl, skel, lib, env = _scene(case, seed, stream)
        n, A, T = wl.n_envs, wl.act_dim, wl.steps
        policy = _policy(wl.mlp_dims, "bf16", seed, n, stream)
        env.attach_policy(policy)
        sims = _sims(wl, skel, lib, env, env.new_obs(), torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"), seed)
        sims = [s.contiguous().cpu().pin_memory() for s in sims]
    torch.cuda.synchronize()
    return dict(case=case, stream=stream, env=env, policy=policy, sims=sims, action=torch.zeros((T, n, A)).pin_memory(),
                reward=torch.zeros((T, n)).pin_memory(), flags=torch.zeros((T, n), dtype=torch.uint8).pin_memory())


def _run_host(st):
    env, policy = st["env"], st["policy"]
    env.reset_all_host(0)
    for s in range(1, st["case"]["steps"] + 1):
        B.step_host(env, policy, s, st["sims"][s - 1], st["action"][s - 1], st["reward"][s - 1], st["flags"][s - 1])
    return dict(action=st["action"], reward=st["reward"], flags=st["flags"])


def _prepare_act(case, seed):
    stream = _stream()
    with torch.cuda.stream(stream):
        wl, _, _, env = _scene(case, seed, stream)
        obs = env.new_obs()
        env.reset_all(obs, 0)
        w = W.make_policy_weights(wl.mlp_dims, "f32", seed)
        n, A = wl.n_envs, wl.act_dim
        st = dict(case=case, stream=stream, obs=obs, dims=wl.mlp_dims, W=[torch.from_numpy(x).cuda() for x in w["W"]],
                  b=[torch.from_numpy(x).cuda() for x in w["b"]], seed=seed, mean=torch.zeros((n, A), device="cuda"),
                  action=torch.zeros((n, A), device="cuda"), logp=torch.zeros(n, device="cuda"))
    torch.cuda.synchronize()
    return st


def _run_act(st):
    B.policy_forward_noalloc(st["dims"], st["W"], st["b"], 0.1, st["seed"], 1, st["obs"], st["mean"], st["action"], st["logp"],
                             stream=st["stream"])
    return dict(mean=st["mean"], action=st["action"], logp=st["logp"])


def prepare(case, seed):
    return {"rollout": _prepare_rollout, "collect": _prepare_collect, "update": _prepare_update, "host": _prepare_host,
            "act": _prepare_act}[case["kind"]](case, seed)


def run(state):
    return {"rollout": _run_rollout, "collect": _run_collect, "update": _run_update, "host": _run_host,
            "act": _run_act}[state["case"]["kind"]](state)


# ---------------------------------------------------------------------------------------------- work, tolerance
def work(case):
    n, T, kind = case["envs"], case.get("steps", 1), case["kind"]
    J, A = BODIES[case["skeleton"]], ACTIONS[case["skeleton"]]
    dims = _dims(case)
    D = dims[0]
    params = lambda d: sum(a * b + b for a, b in zip(d[:-1], d[1:]))
    flops = lambda d: sum(2 * a * b for a, b in zip(d[:-1], d[1:]))
    wb = 2 if case.get("dtype", "bf16") == "bf16" and kind != "act" else 4
    env_step = 52 * J + 4 * D + 5 + 24               # body states in; row, reward, flags out; clip, time, length in and out
    act = 8 * A + 4                                  # mean, action, log-probability out
    if kind == "act":
        return {"bytes": n * (4 * D + act) + 4 * params(dims), "flops": n * flops(dims)}
    if kind in ("rollout", "host"):
        per_step = n * (env_step + act) + wb * params(dims)
        return {"bytes": T * per_step + n * (4 * D + 12), "flops": T * n * flops(dims)}
    cdims = _dims(case, 1)
    if kind == "collect":
        per_step = n * (env_step + act + 4 + 17) + 2 * (params(dims) + params(cdims))
        return {"bytes": T * per_step + n * (4 * D + 16), "flops": T * n * flops(dims) + (T + 1) * n * flops(cdims)}
    samples = case["epochs"] * T * n
    # per sample: observation, action and mean, four scalars; per minibatch: parameters, moments (read and written)
    return {"bytes": samples * (4 * D + 8 * A + 16) + case["epochs"] * case["minibatches"] * 24 * (params(dims) + params(cdims)),
            "flops": 3 * samples * (flops(dims) + flops(cdims))}


def tolerance(case):
    """About four times what another correct implementation at the same precision was seen to differ by: fp32 sums
    in another order 6.8e-7 (rewards 2.4e-6, single ones 3.4e-5); bf16 operands with sums in another order flip the
    rounding of some hidden activations, 5e-4 on the policy's means (single ones 1.4e-2), 1e-2 on the gradients that
    the first moments of an update hold (single ones 0.12)."""
    if case["kind"] == "act" or case.get("dtype") == "f32":
        return {"rel": 1e-5, "max": 2e-4}
    if case["kind"] == "update":
        return {"rel": 3e-2, "max": 0.5}
    return {"rel": 2e-3, "max": 0.06}
