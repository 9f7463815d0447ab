"""The work that programs have this library do, as cases that can be timed and compared.

Every case is one call of the public binding (``paper_2609_13716_gb300.aht``) on inputs
made from a seed: trajectory collection (teammates drawn per call or per episode, or both
seats learning), cross-play matrices, the PPO update, GAE, a policy's outputs on given
observations and the recurrent S5 step.  Policies are random-init, weights and biases
N(0, 0.1), as everywhere in this repository.

Collection and cross-play sample actions, so their outputs are those of a game: a draw
that falls within rounding of an edge of its distribution takes the next action, and that
env's episode goes another way.  They have no 64-bit value (``exact`` is None); the
tolerance allows a few such episodes.  The other calls are checked against plain fp64
torch.
"""
import math

import numpy as np
import torch

from paper_2609_13716_gb300 import aht, workloads as W

FOOD, LEVEL = 3, 3
OBS = {"kitchen": 520, "hanabi": 660, "minihanabi": 156}
ACTIONS = {"lbf": 6, "kitchen": 6, "hanabi": 20, "minihanabi": 10}
# share of ones in a game's binary observation rows
ONES = {"kitchen": 0.06, "hanabi": 0.45, "minihanabi": 0.4}
# steps an env plays in cross-play with random-init policies (the kitchen's are fixed)
TURNS = {"hanabi": 15, "minihanabi": 6}


def listed():
    return [
        # Collection.  A small batch of the fp32 LBF configuration: one CTA, all latency.
        dict(name="collect_lbf7_64x50_f32", kind="collect", game="lbf", side=7, hidden=64, dtype="f32",
             pool=1, n=64, T=50, mode="call"),
        # The LBF 7x7 PPO configuration, teammates drawn from 32: the largest collection.
        dict(name="collect_lbf7_16384x128", kind="collect", game="lbf", side=7, hidden=128, dtype="bf16",
             pool=32, n=16384, T=128, mode="call"),
        # The 12x12 grid, whose observation is too wide for tensor memory.
        dict(name="collect_lbf12_4096x128", kind="collect", game="lbf", side=12, hidden=128, dtype="bf16",
             pool=8, n=4096, T=128, mode="call"),
        # PPO collection in the kitchen, at the kitchen configuration's policy sizes; ragged.
        dict(name="collect_kitchen_1000x64", kind="collect", game="kitchen", side=0, hidden=256, dtype="bf16",
             pool=8, n=1000, T=64, mode="call"),
        # Cross-play: the LBF, kitchen and Hanabi configurations.
        dict(name="xplay_lbf7_8x16x256_f32", kind="xplay", game="lbf", side=7, hidden=64, dtype="f32",
             n_ego=8, n_tm=16, per_pair=256, steps=128),
        dict(name="xplay_kitchen_8x8x64", kind="xplay", game="kitchen", side=0, hidden=256, dtype="bf16",
             n_ego=8, n_tm=8, per_pair=64, steps=400),
        dict(name="xplay_hanabi_16x16x32", kind="xplay", game="hanabi", side=0, hidden=512, dtype="bf16",
             n_ego=16, n_tm=16, per_pair=32, steps=100),
        # One policy's outputs for a batch of observations (analysis, imitation targets).
        dict(name="policy_hanabi_3001", kind="policy", game="hanabi", side=0, hidden=512, dtype="bf16", n=3001),
        # The PPO update of the LBF 7x7 collection: 4 epochs of 4 minibatches.
        dict(name="ppo_update_16384x128", kind="ppo", n=16384, T=128, epochs=4, minibatches=4, mode="update"),
        # GAE of a trajectory held by the caller.
        dict(name="gae_16384x128", kind="gae", n=16384, T=128),
        # One step of the recurrent actor-critic: for an evaluation's few envs, and a large batch.
        dict(name="s5_step_61", kind="s5", n=61, obs_dim=196, actions=6),
        dict(name="s5_step_16384", kind="s5", n=16384, obs_dim=196, actions=6),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["collect", "collect", "collect", "xplay", "xplay", "policy", "ppo", "gae", "s5"])
    if kind == "collect":
        game = rng.choice(["lbf", "lbf", "lbf", "kitchen"])
        mode = rng.choice(["call", "call", "episode", "ippo"])
        T = _log_int(rng, 4, 128)
        if game == "kitchen":
            return dict(kind=kind, game=game, side=0, hidden=256, dtype="bf16",
                        pool=_log_int(rng, 1, 16), n=_log_int(rng, 16, 64000 // T), T=T, mode=mode)
        side = rng.choice([5, 6, 7, 7, 12])
        dtype = rng.choice(["bf16", "f32"])
        steps = 1 << 21 if side < 12 else 1 << 19 if mode == "call" else 1 << 15
        return dict(kind=kind, game=game, side=side, hidden=64 if dtype == "f32" else rng.choice([64, 128]),
                    dtype=dtype, pool=_log_int(rng, 1, 32), n=_log_int(rng, 16, min(16384, steps // T)), T=T,
                    mode=mode)
    if kind == "xplay":
        game = rng.choice(["lbf", "lbf", "kitchen", "hanabi", "minihanabi"])
        if game == "lbf":
            dtype = rng.choice(["bf16", "f32"])
            return dict(kind=kind, game=game, side=rng.choice([5, 7, 12]),
                        hidden=64 if dtype == "f32" else rng.choice([64, 128]), dtype=dtype,
                        n_ego=rng.randint(1, 8), n_tm=rng.randint(1, 16), per_pair=_log_int(rng, 8, 256),
                        steps=rng.randint(30, 128))
        if game == "kitchen":
            return dict(kind=kind, game=game, side=0, hidden=256, dtype="bf16", n_ego=rng.randint(1, 8),
                        n_tm=rng.randint(1, 8), per_pair=_log_int(rng, 4, 64), steps=rng.randint(50, 400))
        return dict(kind=kind, game=game, side=0, hidden=512 if game == "hanabi" else 256, dtype="bf16",
                    n_ego=rng.randint(1, 16), n_tm=rng.randint(1, 16), per_pair=_log_int(rng, 4, 32), steps=100)
    if kind == "policy":
        game = rng.choice(["lbf", "kitchen", "hanabi", "minihanabi"])
        return dict(kind=kind, game=game, side=rng.choice([7, 12]) if game == "lbf" else 0,
                    hidden=rng.choice([64, 128, 256, 512]), dtype=rng.choice(["bf16", "f32"]),
                    n=_log_int(rng, 1, 8192))
    if kind == "ppo":
        minibatches = rng.choice([1, 2, 4])
        T = 8 * rng.randint(2, 16)
        return dict(kind=kind, n=8 * minibatches * _log_int(rng, 2, 16384 // (8 * minibatches)), T=T,
                    epochs=rng.randint(1, 4), minibatches=minibatches, mode=rng.choice(["update", "gradient"]))
    if kind == "gae":
        T = _log_int(rng, 1, 400)
        return dict(kind=kind, n=_log_int(rng, 1, (1 << 21) // T), T=T)
    wide = rng.choice([(196, 6), (576, 6), (520, 6), (660, 20)])
    return dict(kind="s5", n=_log_int(rng, 1, 16384), obs_dim=wide[0], actions=wide[1])


# ---- inputs ------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _obs_dim(case):
    return case["side"] ** 2 * 4 if case["game"] == "lbf" else OBS[case["game"]]


def _env(case, episode):
    if case["game"] == "lbf":
        return W.EnvSpec(kind=W.LBF, width=case["side"], height=case["side"], n_food=FOOD, max_agent_level=LEVEL,
                         episode_len=episode)
    if case["game"] == "kitchen":
        return W.EnvSpec(kind=W.OVERCOOKED, width=5, height=4, episode_len=episode, cook_time=20, soup_reward=20)
    return W.EnvSpec(kind=W.HANABI if case["game"] == "hanabi" else W.MINI_HANABI, episode_len=0)


def _mlp(g, obs_dim, hidden, outputs, dtype):
    dims = [obs_dim, hidden, hidden, outputs]
    to = torch.bfloat16 if dtype == "bf16" else torch.float32
    normal = lambda *shape: (torch.randn(*shape, generator=g, device="cuda") * 0.1).to(to)  # noqa: E731
    return [(normal(dims[i + 1], dims[i]), normal(dims[i + 1])) for i in range(3)]


def _context(case, g, heads, n, episode, seed):
    A = ACTIONS[case["game"]]
    policies = [_mlp(g, _obs_dim(case), case["hidden"], A + h, case["dtype"]) for h in heads]
    ctx = aht.aht_create(_env(case, episode), policies, n, seed, has_value_head=heads,
                         weight_dtype=aht.AHT_BF16 if case["dtype"] == "bf16" else aht.AHT_FP32)
    return ctx, policies


def _lbf_rows(g, n, side):
    """n LBF observations: two agents and up to three uneaten foods on distinct cells."""
    cells = torch.rand(n, side * side, generator=g, device="cuda").topk(2 + FOOD, dim=1).indices
    rows = torch.zeros(n, side * side, 4, dtype=torch.uint8, device="cuda")
    rows[:, :, 3] = 1
    at = torch.arange(n, device="cuda")
    for k in range(2 + FOOD):
        here = torch.ones(n, dtype=torch.bool, device="cuda")
        if k < 2:
            value = torch.randint(1, LEVEL + 1, (n,), generator=g, device="cuda")
        else:
            value = torch.randint(1, 2 * LEVEL + 1, (n,), generator=g, device="cuda")
            here = torch.rand(n, generator=g, device="cuda") < 0.6
        word = torch.zeros(n, 4, dtype=torch.uint8, device="cuda")
        word[:, min(k, 2)] = value.to(torch.uint8)
        rows[at[here], cells[here, k]] = word[here]
    return rows.reshape(n, side * side * 4)


def _rows(g, n, case):
    if case["game"] == "lbf":
        return _lbf_rows(g, n, case["side"])
    return (torch.rand(n, OBS[case["game"]], generator=g, device="cuda") < ONES[case["game"]]).to(torch.uint8)


def _forward(obs, layers):
    h = obs
    for W_, b in layers[:2]:
        h = torch.tanh(h @ W_.to(h.dtype).T + b.to(h.dtype))
    return h @ layers[2][0].to(h.dtype).T + layers[2][1].to(h.dtype)


def _policy_inputs(case, seed):
    g = _generator(seed)
    A = ACTIONS[case["game"]]
    layers = _mlp(g, _obs_dim(case), case["hidden"], A + 1, case["dtype"])
    return layers, _rows(g, case["n"], case)


def _ppo_inputs(case, seed):
    """A learner's weights and a trajectory collected by a slightly older copy of them."""
    g = _generator(seed)
    layers = _mlp(g, 196, 128, 7, "f32")
    old = [(W_ + 0.005 * torch.randn(W_.shape, generator=g, device="cuda"), b) for W_, b in layers]
    S = case["n"] * case["T"]
    obs = _lbf_rows(g, S, 7)
    z = torch.cat([_forward(o.float(), old) for o in obs.split(1 << 19)])
    logp = torch.log_softmax(z[:, :6], 1)
    actions = torch.multinomial(logp.exp(), 1, generator=g)
    advantages = 0.3 * torch.randn(S, generator=g, device="cuda")
    shape = (case["T"], case["n"])
    values = z[:, 6].contiguous()
    traj = dict(obs=obs.reshape(*shape, 196), actions=actions[:, 0].to(torch.uint8).reshape(shape),
                logp=logp.gather(1, actions)[:, 0].reshape(shape), values=values.reshape(shape),
                advantages=advantages.reshape(shape), targets=(values + advantages).reshape(shape))
    return layers, traj


def _gae_inputs(case, seed):
    g = _generator(seed)
    shape = (case["T"], case["n"])
    rewards = torch.rand(shape, generator=g, device="cuda")
    rewards = torch.where(torch.rand(shape, generator=g, device="cuda") < 0.05, rewards, torch.zeros_like(rewards))
    values = 0.5 * torch.randn(shape, generator=g, device="cuda")
    dones = (torch.rand(shape, generator=g, device="cuda") < 0.03).to(torch.uint8)
    return rewards, values, dones, 0.5 * torch.randn(case["n"], generator=g, device="cuda")


def _s5_inputs(case, seed, H=128, P=128, F=1024):
    rng = np.random.Generator(np.random.Philox(seed))
    f32 = lambda a: np.asarray(a, np.float32)  # noqa: E731
    normal = lambda *s: rng.standard_normal(s, np.float32)  # noqa: E731
    dense = lambda o, i: (f32(normal(o, i) / math.sqrt(i)), f32(0.1 * normal(o)))  # noqa: E731
    K, A, n = case["obs_dim"], case["actions"], case["n"]
    p = {}
    p["We1"], p["be1"] = dense(H, K)
    p["We2"], p["be2"] = dense(H, H)
    p["lam_re"] = f32(-np.exp(rng.uniform(math.log(0.05), 0.0, P)))
    p["lam_im"] = f32(rng.uniform(-math.pi, math.pi, P))
    p["log_dt"] = f32(rng.uniform(math.log(1e-3), math.log(1e-1), P))
    p["B_re"], p["B_im"] = f32(normal(P, H) / math.sqrt(2 * H)), f32(normal(P, H) / math.sqrt(2 * H))
    p["C_re"], p["C_im"] = f32(normal(H, P) / math.sqrt(2 * P)), f32(normal(H, P) / math.sqrt(2 * P))
    p["Dv"] = normal(H)
    for head, out in (("a", A), ("c", 1)):
        pairs = [dense(F, H), dense(F, F), dense(F, F), dense(out, F)]
        p["W" + head], p["b" + head] = [x[0] for x in pairs], [x[1] for x in pairs]
    g = _generator(seed)
    game = {520: "kitchen", 660: "hanabi"}.get(K)
    obs = _rows(g, n, dict(game=game)) if game else _lbf_rows(g, n, math.isqrt(K // 4))
    reset = (torch.rand(n, generator=g, device="cuda") < 0.02).to(torch.uint8)
    state = 0.3 * torch.randn(n, 2 * P, generator=g, device="cuda")
    legal = None
    if A == 20:
        legal = (torch.rand(n, A, generator=g, device="cuda") < 0.6).to(torch.uint8)
        legal[:, 0] = 1
    return p, obs, reset, state, legal


def prepare(case, seed):
    kind = case["kind"]
    empty = lambda *shape, dtype=torch.float32: torch.empty(shape, dtype=dtype, device="cuda")  # noqa: E731
    if kind == "collect":
        heads = [1, 1] if case["mode"] == "ippo" else [1] + [0] * case["pool"]
        ctx, _ = _context(case, _generator(seed), heads, case["n"], 50 if case["game"] == "lbf" else 400, seed)
        state = dict(case=case, ctx=ctx, traj=aht.traj_buffers(ctx, case["T"]))
        if case["mode"] == "ippo":
            state["traj"]["teammate"].zero_()
            state["traj1"] = {k: v for k, v in aht.traj_buffers(ctx, case["T"]).items() if k != "teammate"}
        elif case["mode"] == "episode":
            state["teammates"] = empty(case["T"], case["n"], dtype=torch.int32)
        return state
    if kind == "xplay":
        ne, nt, P = case["n_ego"], case["n_tm"], case["per_pair"]
        ctx, _ = _context(case, _generator(seed), [0] * (ne + nt), ne * nt * P,
                          case["steps"] if case["game"] in ("lbf", "kitchen") else 0, seed)
        state = dict(case=case, ctx=ctx, matrix=empty(ne, nt), steps=empty(ne, nt, P, dtype=torch.int32))
        if case["game"] == "lbf":
            state["returns"] = empty(ne, nt, P)
        else:  # these games' returns are mostly 0 with random-init policies: the replays too
            state["actions"] = empty(case["steps"], ne * nt * P, 2, dtype=torch.uint8)
        return state
    if kind == "policy":
        layers, obs = _policy_inputs(case, seed)
        ctx = aht.aht_create(_env(case, 0 if "hanabi" in case["game"] else 50), [layers], 64, seed, has_value_head=[1],
                             weight_dtype=aht.AHT_BF16 if case["dtype"] == "bf16" else aht.AHT_FP32)
        return dict(case=case, ctx=ctx, obs=obs, out=empty(case["n"], ACTIONS[case["game"]] + 1))
    if kind == "ppo":
        layers, traj = _ppo_inputs(case, seed)
        learner = aht.aht_learner_create(196, 6, layers, epochs=case["epochs"], minibatches=case["minibatches"],
                                         seed=seed)
        if case["mode"] == "gradient":
            out = dict(stats=empty(6), grad=empty(learner.n_params))
        else:
            out = dict(stats=empty(case["epochs"] * case["minibatches"], 6),
                       **{k: empty(learner.n_params) for k in ("params", "adam_m", "adam_v")})
        return dict(case=case, learner=learner, traj=traj, out=out)
    if kind == "gae":
        inputs = _gae_inputs(case, seed)
        return dict(case=case, inputs=inputs, advantages=torch.empty_like(inputs[0]), targets=torch.empty_like(inputs[0]))
    p, obs, reset, x, legal = _s5_inputs(case, seed)
    return dict(case=case, policy=aht.aht_s5_create(p, case["n"]), obs=obs, reset=reset, state=x, legal=legal,
                logits=empty(case["n"], case["actions"]), values=empty(case["n"]))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "collect":
        ctx, T, traj = state["ctx"], case["T"], state["traj"]
        if case["mode"] == "ippo":
            aht.aht_rollout_ippo(ctx, 0, 1, T, traj, state["traj1"])
            return {"seat0": traj, "seat1": state["traj1"]}
        pool = range(1, 1 + case["pool"])
        if case["mode"] == "episode":
            aht.aht_rollout_resample(ctx, 0, pool, T, traj, state["teammates"])
            return dict(traj, teammates=state["teammates"])
        aht.aht_rollout(ctx, 0, pool, T, traj)
        return traj
    if kind == "xplay":
        ne, nt = case["n_ego"], case["n_tm"]
        aht.aht_xplay_matrix(state["ctx"], range(ne), range(ne, ne + nt), case["per_pair"], case["steps"],
                             state["matrix"], state.get("returns"), state["steps"], state.get("actions"))
        return {k: state[k] for k in ("matrix", "returns", "steps", "actions") if k in state}
    if kind == "policy":
        aht.aht_policy_forward(state["ctx"], 0, state["obs"], state["out"])
        return state["out"]
    if kind == "ppo":
        out = state["out"]
        if case["mode"] == "gradient":  # of the next update's last minibatch
            aht.aht_ppo_grad(state["learner"], state["traj"], case["epochs"] - 1, case["minibatches"] - 1, out["grad"],
                             out["stats"])
            return out
        aht.aht_ppo_update(state["learner"], state["traj"], out["stats"])
        aht.aht_learner_get(state["learner"], out["params"], out["adam_m"], out["adam_v"])
        return out
    if kind == "gae":
        rewards, values, dones, last = state["inputs"]
        aht.aht_gae(rewards, values, dones, last, 0.99, 0.95, state["advantages"], state["targets"])
        return {"advantages": state["advantages"], "targets": state["targets"]}
    aht.aht_s5_step(state["policy"], state["obs"], state["reset"], state["state"], state["logits"], state["values"],
                    state["legal"])
    return {"logits": state["logits"], "values": state["values"], "state": state["state"]}


# ---- what a pass cannot do without ---------------------------------------------------------
def _mlp_flops(obs_dim, hidden, outputs):
    return 2 * (obs_dim * hidden + hidden * hidden + hidden * outputs)


def work(case):
    """Policy FLOPs as dense products (an observation's zeros counted), every input read and
    every output written once; weights once."""
    kind = case["kind"]
    if kind in ("collect", "xplay", "policy"):
        K, h, A = _obs_dim(case), case["hidden"], ACTIONS[case["game"]]
        weight = (K * h + h * h + h * A) * (2 if case["dtype"] == "bf16" else 4)
    if kind == "collect":
        steps, learners = case["n"] * case["T"], 2 if case["mode"] == "ippo" else 1
        flops = _mlp_flops(K, h, A + 1) + _mlp_flops(K, h, A + learners - 1)
        return {"bytes": steps * learners * (K + 2 + 1 + 5 * 4) + weight * (2 if learners == 2 else 1 + case["pool"]),
                "flops": steps * flops + case["n"] * learners * _mlp_flops(K, h, A + 1)}
    if kind == "xplay":
        envs = case["n_ego"] * case["n_tm"] * case["per_pair"]
        steps = envs * TURNS.get(case["game"], case["steps"])
        seats = 1 if "hanabi" in case["game"] else 2
        replay = 0 if case["game"] == "lbf" else 2 * envs * case["steps"]
        return {"bytes": envs * 8 + replay + weight * (case["n_ego"] + case["n_tm"]),
                "flops": steps * seats * _mlp_flops(K, h, A)}
    if kind == "policy":
        return {"bytes": case["n"] * (K + 4 * (A + 1)) + weight, "flops": case["n"] * _mlp_flops(K, h, A + 1)}
    if kind == "ppo":
        S = case["n"] * case["T"]
        passes = case["epochs"] if case["mode"] == "update" else 1 / case["minibatches"]
        # forward, weight gradients, and the input gradients of all but the first layer
        f, first = _mlp_flops(196, 128, 7), 2 * 196 * 128
        return {"bytes": S * (196 + 1 + 5 * 4) * passes, "flops": S * passes * (3 * f - first)}
    if kind == "gae":
        return {"bytes": case["n"] * case["T"] * (4 + 4 + 1 + 8), "flops": case["n"] * case["T"] * 8}
    H, P, F, K, A = 128, 128, 1024, case["obs_dim"], case["actions"]
    macs = K * H + H * H + H * 2 * P + 2 * P * H + 2 * (H * F + 2 * F * F) + F * (A + 1)
    return {"bytes": case["n"] * (K + 1 + 16 * P + 4 * (A + 1)) + 2 * macs, "flops": 2 * case["n"] * macs}


# ---- comparison ----------------------------------------------------------------------------
def tolerance(case):
    """About four times what another correct implementation differs by.  Games: the fp64
    oracle playing the same seeds (4 of 16384 episodes of 64 steps go another way: 2e-5 of
    the actions, values 5e-3); the others: plain fp64 torch (`exact`)."""
    if case["kind"] == "ppo":
        # an update's Adam steps divide small gradients by their own size and move weights
        # across bf16 rounding edges, which changes the gradients that follow
        return {"rel": 1e-4, "max": 5e-3} if case["mode"] == "gradient" else {"rel": 0.015, "max": 0.9}
    return {
        "collect": {"rel": 0.02, "max": 0.99, "differ": 3e-4},
        "xplay": {"rel": 0.02, "max": 0.99, "differ": 5e-3},
        "policy": {"rel": 5e-6, "max": 5e-5},
        "gae": {"rel": 2e-6, "max": 2e-5},
        "s5": {"rel": 1e-4, "max": 2e-3},
    }[case["kind"]]


def exact(case, seed):
    kind = case["kind"]
    if kind == "policy":
        layers, obs = _policy_inputs(case, seed)
        return _forward(obs.double(), layers)
    if kind == "gae":
        return _exact_gae(*(x.double() for x in _gae_inputs(case, seed)))
    if kind == "s5":
        return _exact_s5(*_s5_inputs(case, seed))
    if kind == "ppo":
        return _exact_ppo(case, seed, *_ppo_inputs(case, seed))
    return None


def _exact_gae(rewards, values, dones, last):
    advantages, a, v = torch.empty_like(rewards), torch.zeros_like(last), last
    for t in reversed(range(rewards.shape[0])):
        live = 1.0 - dones[t]
        a = rewards[t] + 0.99 * live * v - values[t] + 0.99 * 0.95 * live * a
        advantages[t], v = a, values[t]
    return {"advantages": advantages, "targets": advantages + values}


def _exact_s5(p, obs, reset, state, legal):
    f64 = lambda a: torch.from_numpy(np.asarray(a)).cuda().double()  # noqa: E731
    bf16 = lambda a: torch.from_numpy(a).cuda().bfloat16().double()  # noqa: E731
    h = torch.relu(obs.double() @ bf16(p["We1"]).T + f64(p["be1"]))
    u = torch.relu(h @ bf16(p["We2"]).T + f64(p["be2"]))
    lam = torch.complex(f64(p["lam_re"]), f64(p["lam_im"]))
    step = torch.exp(lam * torch.exp(f64(p["log_dt"])))
    P = lam.shape[0]
    live = (1.0 - reset.double())[:, None]
    before = torch.complex(state[:, :P].double() * live, state[:, P:].double() * live)
    Bbar = ((step - 1.0) / lam)[:, None] * torch.complex(f64(p["B_re"]), f64(p["B_im"]))
    x = step * before + torch.complex(u @ Bbar.real.T, u @ Bbar.imag.T)
    y = x.real @ f64(p["C_re"]).T - x.imag @ f64(p["C_im"]).T + f64(p["Dv"]) * u
    v = u + torch.nn.functional.gelu(y)
    outs = []
    for head in "ac":
        h = v
        for l in range(3):
            h = torch.relu(h @ bf16(p["W" + head][l]).T + f64(p["b" + head][l]))
        outs.append(h @ bf16(p["W" + head][3]).T + f64(p["b" + head][3]))
    logits = outs[0] if legal is None else outs[0].masked_fill(legal == 0, -math.inf)
    return {"logits": logits, "values": outs[1][:, 0], "state": torch.cat([x.real, x.imag], 1)}


def _mul32(a, x):
    """(high, low) 32 bits of a * x, a an int and x an int64 tensor, both below 2^32."""
    high, low = a * (x >> 16), a * (x & 0xFFFF)
    return (high + (low >> 16)) >> 16, (((high & 0xFFFF) << 16) + low) & 0xFFFFFFFF


def _philox_word0(x, c1, c2, c3, seed):
    """Word 0 of Philox4x32-10 of the counters (x, c1, c2, c3) under the 64-bit key `seed`."""
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    c = [x] + [torch.full_like(x, v) for v in (c1, c2, c3)]
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, c[0])
        h1, l1 = _mul32(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c[0]


def _permutation(S, epoch, seed):
    """The epoch's sample order as include/aht.h states it (a keyed Feistel network)."""
    w = max(2, (S - 1).bit_length())
    rb = w // 2
    y = torch.arange(S, device="cuda")
    todo = torch.ones(S, dtype=torch.bool, device="cuda")
    while bool(todo.any()):
        L, R = y[todo] >> rb, y[todo] & ((1 << rb) - 1)
        for r in range(4):
            if r % 2 == 0:
                L = (L ^ _philox_word0(R, epoch, 4, r, seed)) & ((1 << (w - rb)) - 1)
            else:
                R = (R ^ _philox_word0(L, epoch, 4, r, seed)) & ((1 << rb) - 1)
        y[todo] = (L << rb) | R
        todo = y >= S
    return y


def _exact_ppo(case, seed, layers, traj, clip=0.2, vf=0.5, ent=0.01, lr=2.5e-4, most=0.5, b1=0.9, b2=0.999, eps=1e-5):
    E, M, S = case["epochs"], case["minibatches"], case["n"] * case["T"]
    flat = {k: v.reshape(S, -1) if k == "obs" else v.reshape(S) for k, v in traj.items()}
    params = [t.double() for layer in layers for t in layer]
    m, v = [torch.zeros_like(t) for t in params], [torch.zeros_like(t) for t in params]
    stats = torch.empty(E * M, 6, dtype=torch.float64, device="cuda")
    gradient = case["mode"] == "gradient"
    join = lambda ts: torch.cat([t.detach().reshape(-1) for t in ts])  # noqa: E731
    for e in range(E - 1 if gradient else 0, E):
        order = _permutation(S, e, seed)
        for b in range(M - 1 if gradient else 0, M):
            at = order[b * (S // M):(b + 1) * (S // M)]
            # the products run on the bf16 copies of W1 and W2, the gradient goes to the master weights
            ws = [(t.float().bfloat16().double() if i in (0, 2) else t).requires_grad_() for i, t in enumerate(params)]
            adv_all = flat["advantages"][at].double()
            mean, std = adv_all.mean(), adv_all.std(unbiased=False)
            total = torch.zeros(6, dtype=torch.float64, device="cuda")
            grads = [torch.zeros_like(t) for t in params]
            for part in at.split(1 << 18):
                z = _forward(flat["obs"][part].double(), [(ws[2 * i], ws[2 * i + 1]) for i in range(3)])
                logp = torch.log_softmax(z[:, :6], 1)
                lp = logp.gather(1, flat["actions"][part].long()[:, None])[:, 0]
                old, v_old, target = (flat[k][part].double() for k in ("logp", "values", "targets"))
                adv = (flat["advantages"][part].double() - mean) / (std + 1e-8)
                rho = torch.exp(lp - old)
                pg = -torch.minimum(rho * adv, rho.clamp(1 - clip, 1 + clip) * adv)
                v_clip = v_old + (z[:, 6] - v_old).clamp(-clip, clip)
                lv = 0.5 * torch.maximum((z[:, 6] - target) ** 2, (v_clip - target) ** 2)
                entropy = -(logp.exp() * logp).sum(1)
                loss = pg + vf * lv - ent * entropy
                for s, t in zip(grads, torch.autograd.grad(loss.sum() / at.numel(), ws)):
                    s += t
                with torch.no_grad():
                    total += torch.stack([x.sum() for x in (loss, pg, lv, entropy, old - lp,
                                                            ((rho - 1).abs() > clip).double())])
            stats[e * M + b] = total / at.numel()
            if gradient:
                return {"stats": stats[-1], "grad": join(grads)}
            norm = math.sqrt(sum(float((t * t).sum()) for t in grads))
            scale = most / norm if norm >= most else 1.0
            k = e * M + b + 1
            for i, t in enumerate(grads):
                m[i] = b1 * m[i] + (1 - b1) * scale * t
                v[i] = b2 * v[i] + (1 - b2) * (scale * t) ** 2
                params[i] = params[i].detach() - lr * (m[i] / (1 - b1 ** k)) / ((v[i] / (1 - b2 ** k)).sqrt() + eps)
    return {"stats": stats, "params": join(params), "adam_m": join(m), "adam_v": join(v)}
