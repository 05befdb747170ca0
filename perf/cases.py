"""The work a user of this framework has it do, as timed cases.

One population-based training loop is: keep a payoff table of Kuhn or Leduc
policies (evaluation), solve the table as a matrix game (fictitious play or the
linear program), measure the exploitability of the mixtures, roll out policy
combinations in the particle scenarios, and update the policies from the
samples. Every case is one call, or the few calls that belong together, through
the public entry points of ``paper_2106_07551_gb300.Context``.

Sizes are those of this repository's workloads (Kuhn 4 x 4 x 10,000 hands; Leduc
8 x 8 x 65,536 with fp32 policies and 64 x 64 x 16,384 with bf16 policies; spread
with 4,096 and 65,536 environments), the 2,000 simulations per policy pair of the
Leduc population loop, and odd sizes in between. ``draw`` spreads over the same
ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2106_07551_gb300 as mb

DEV = "cuda:0"
SPREAD, ADVERSARY, SPEAKER, PUSH, TAG, REFERENCE = 3, 4, 5, 6, 7, 8

# scenario: env kind, agents, landmarks, observation floats, actions, hidden width, dtype
SCENARIOS = {
    "spread3": (SPREAD, 3, 3, 18, 5, 64, mb.MALIB_F32),
    "spread3_contact": (SPREAD, 3, 3, 18, 5, 64, mb.MALIB_F32),
    "adversary": (ADVERSARY, 3, 2, 14, 5, 64, mb.MALIB_F32),
    "speaker_listener": (SPEAKER, 2, 3, 11, 5, 64, mb.MALIB_F32),
    "push": (PUSH, 2, 1, 8, 5, 64, mb.MALIB_F32),
    "tag": (TAG, 4, 2, 16, 5, 64, mb.MALIB_F32),
    "reference": (REFERENCE, 2, 3, 14, 15, 64, mb.MALIB_F32),
    "spread8": (SPREAD, 8, 8, 34, 5, 256, mb.MALIB_BF16),
}
LEARNABLE = ("spread3", "adversary", "speaker_listener", "push", "tag")
STEPS = 25                       # steps of a particle episode
LR, GAMMA, ENTROPY, CLIP = 1e-4, 0.95, 1e-3, 0.2


def listed():
    return [
        # Kuhn: the smallest table, one short launch sequence
        {"name": "kuhn_table", "kind": "eval", "game": "kuhn", "rows": 4, "cols": 4, "hands": 10_000, "new_only": False},
        # Leduc: a whole table of fp32 policies, estimated closely
        {"name": "leduc_table_f32", "kind": "eval", "game": "leduc_f32_128", "rows": 8, "cols": 8, "hands": 65_536,
         "new_only": False},
        # Leduc: a whole table of bf16 policies, the largest evaluation
        {"name": "leduc_table_bf16", "kind": "eval", "game": "leduc_bf16", "rows": 64, "cols": 64, "hands": 16_384,
         "new_only": False},
        # Leduc: one step of the population loop, the new row and column only, from host pair lists
        # and read back on the host, 2,000 simulations per entry
        {"name": "leduc_row_bf16", "kind": "eval", "game": "leduc_bf16", "rows": 33, "cols": 33, "hands": 2_000,
         "new_only": True},
        # spread, 3 agents: the samples of one training batch, with the behaviour logits
        {"name": "spread3_rollout", "kind": "rollout", "scenario": "spread3", "combos": 32, "envs": 128, "episodes": 10,
         "logits": True},
        # spread, 8 agents, bf16: the largest rollout
        {"name": "spread8_rollout", "kind": "rollout", "scenario": "spread8", "combos": 512, "envs": 128, "episodes": 2,
         "logits": False},
        # tag: contact forces, a few combinations of ragged size, an odd number of episodes
        {"name": "tag_rollout", "kind": "rollout", "scenario": "tag", "combos": 9, "envs": 125, "episodes": 3,
         "logits": False},
        # every policy of a population updated by its policy gradient (batched step, Adam, write-back)
        {"name": "pg_step", "kind": "learn", "scenario": "spread3", "policies": 16, "combos": 32, "envs": 128,
         "episodes": 10, "ppo": False},
        # one epoch of clipped-surrogate updates on a small batch of ragged size
        {"name": "ppo_step", "kind": "learn", "scenario": "push", "policies": 3, "combos": 7, "envs": 60, "episodes": 5,
         "ppo": True},
        # the meta-solver of the loop on one evaluated table, and the payoffs under its mixtures
        {"name": "meta_fictitious_play", "kind": "fp", "games": 1, "rows": 64, "cols": 64, "iters": 2_000},
        # the exact equilibrium of one table
        {"name": "meta_lp", "kind": "lp", "games": 1, "rows": 100, "cols": 100},
        # convergence measure: exploitability of the two seats' mixtures
        {"name": "exploitability", "kind": "exploit", "game": "leduc_f32_128", "rows": 40, "cols": 40},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "rollout", "rollout", "rollout", "learn", "learn", "fp", "lp", "exploit"])
    if kind == "eval":
        game = rng.choice(["kuhn", "leduc_f32_128", "leduc_f32_128", "leduc_f32_64", "leduc_bf16", "leduc_bf16"])
        if game == "kuhn":
            rows, cols, hands = _log(rng, 1, 16), _log(rng, 1, 16), _log(rng, 100, 1_000_000)
        elif game == "leduc_bf16":
            rows, cols, hands = _log(rng, 1, 64), _log(rng, 1, 64), _log(rng, 200, 16_384)
        else:
            rows, cols, hands = _log(rng, 1, 16), _log(rng, 1, 16), _log(rng, 200, 20_000)
        return {"kind": kind, "game": game, "rows": rows, "cols": cols, "hands": hands, "new_only": rng.random() < 0.4}
    if kind == "rollout":
        sc = rng.choice(list(SCENARIOS))
        big = sc == "spread8"
        return {"kind": kind, "scenario": sc, "combos": _log(rng, 1, 400 if big else 64), "envs": _log(rng, 8, 128),
                "episodes": _log(rng, 1, 2 if big else 20), "logits": rng.random() < 0.4}
    if kind == "learn":
        return {"kind": kind, "scenario": rng.choice(LEARNABLE), "policies": _log(rng, 1, 16), "combos": _log(rng, 2, 40),
                "envs": _log(rng, 8, 128), "episodes": _log(rng, 1, 10), "ppo": rng.random() < 0.5}
    if kind == "fp":
        return {"kind": kind, "games": _log(rng, 1, 152), "rows": _log(rng, 2, 300), "cols": _log(rng, 2, 300),
                "iters": _log(rng, 100, 5_000)}
    if kind == "lp":
        return {"kind": kind, "games": _log(rng, 1, 32), "rows": _log(rng, 2, 140), "cols": _log(rng, 2, 140)}
    return {"kind": kind, "game": rng.choice(["kuhn", "leduc_f32_64", "leduc_f32_128", "leduc_f32_128", "leduc_bf16"]),
            "rows": _log(rng, 1, 64), "cols": _log(rng, 1, 64)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 1)


def _dims(case):
    if case["kind"] in ("rollout", "learn"):
        s = SCENARIOS[case["scenario"]]
        return (s[3], s[5], s[5], s[4])
    h = {"leduc_f32_64": 64, "leduc_f32_128": 128, "leduc_bf16": 256}[case["game"]]
    return (17, h, h, 3)


def _mlps(gen, n, dims):
    """n policies in the plain layout (W1, b1, W2, b2, W3, b3), weights N(0, 1/fan_in)."""
    i, h1, h2, o = dims
    parts = []
    for fan_in, fan_out in ((i, h1), (h1, h2), (h2, o)):
        parts.append(torch.randn((n, fan_out * fan_in), generator=gen, device=DEV) * (1.0 / math.sqrt(fan_in)))
        parts.append(torch.randn((n, fan_out), generator=gen, device=DEV) * 0.1)
    return torch.cat(parts, dim=1).contiguous()


def _poker_population(case, gen):
    """Parameters of all policies: the rows' (seat 0) first, then the columns' (seat 1)."""
    n = case["rows"] + case["cols"]
    if case["game"] == "kuhn":
        return torch.rand((n, 6), generator=gen, device=DEV)
    return _mlps(gen, n, _dims(case))


def _load_poker(case, params):
    ctx = mb.Context(0)
    rows = case["rows"]
    if case["game"] == "kuhn":
        spec = mb.make_spec(mb.MALIB_ENV_KUHN, 2, 0, 2)
        descs = [mb.policy_desc(mb.MALIB_POL_TABULAR, mb.MALIB_F32, int(i >= rows), (6, 0, 0, 1), p)
                 for i, p in enumerate(params)]
    else:
        spec = mb.make_spec(mb.MALIB_ENV_LEDUC, 2, 17, 3)
        dt = mb.MALIB_BF16 if case["game"] == "leduc_bf16" else mb.MALIB_F32
        descs = [mb.policy_desc(mb.MALIB_POL_MLP, dt, int(i >= rows), _dims(case), p) for i, p in enumerate(params)]
    torch.cuda.synchronize()
    ctx.pop_load(spec, descs)
    return ctx


def _poker_pairs(case):
    """All row-column pairs, or those of the newest row and the newest column."""
    r, c = case["rows"], case["cols"]
    if case["new_only"]:
        ij = [(r - 1, j) for j in range(c)] + [(i, c - 1) for i in range(r - 1)]
    else:
        ij = [(i, j) for i in range(r) for j in range(c)]
    return np.array([(i, r + j) for i, j in ij], np.int32)


def _combos(case, seed, n_pol):
    n = SCENARIOS[case["scenario"]][1]
    rng = np.random.default_rng(int(seed) + 17)
    return rng.integers(0, n_pol, size=(case["combos"], n)).astype(np.int32)


def _scenario_spec(case):
    kind, agents, marks, obs, acts, _, _ = SCENARIOS[case["scenario"]]
    flags = mb.MALIB_DUMP_LOGITS if case.get("logits") else 0
    if case["scenario"] == "spread3_contact":
        flags |= mb.MALIB_SPREAD_CONTACT
    return mb.make_spec(kind, agents, obs, acts, n_landmarks=marks, episode_len=STEPS,
                        n_envs=case["combos"] * case["envs"], flags=flags)


def _load_scenario(case, params, spec):
    ctx = mb.Context(0)
    dt = SCENARIOS[case["scenario"]][6]
    torch.cuda.synchronize()
    ctx.pop_load(spec, [mb.policy_desc(mb.MALIB_POL_MLP, dt, -1, _dims(case), p) for p in params])
    return ctx


def _forward(params, dims, x):
    """Logits of policies params [g][P] on x [g][n][in]."""
    i, h1, h2, o = dims
    sizes = [h1 * i, h1, h2 * h1, h2, o * h2, o]
    w1, b1, w2, b2, w3, b3 = torch.split(params, sizes, dim=1)
    g = params.shape[0]
    h = torch.relu(torch.baddbmm(b1[:, None], x, w1.reshape(g, h1, i).transpose(1, 2)))
    h = torch.relu(torch.baddbmm(b2[:, None], h, w2.reshape(g, h2, h1).transpose(1, 2)))
    return torch.baddbmm(b3[:, None], h, w3.reshape(g, o, h2).transpose(1, 2))


def _by_slot(t, case):
    """[E][T][V][N][...] -> [combination * agent][E * T * envs][...]."""
    n = SCENARIOS[case["scenario"]][1]
    e, c, v = case["episodes"], case["combos"], case["envs"]
    rest = t.shape[4:]
    t = t.reshape(e, STEPS, c, v, n, *rest)
    return t.permute(2, 4, 0, 1, 3, *range(5, 5 + len(rest))).reshape(c * n, e * STEPS * v, *rest)


def _from_slot(t, case):
    n = SCENARIOS[case["scenario"]][1]
    e, c, v = case["episodes"], case["combos"], case["envs"]
    rest = t.shape[2:]
    t = t.reshape(c, n, e, STEPS, v, *rest)
    return t.permute(2, 3, 0, 4, 1, *range(5, 5 + len(rest))).reshape(e, STEPS, c * v, n, *rest).contiguous()


def _samples(case, seed):
    """Policies, the combinations and a batch of samples as a rollout leaves them: bounded
    observations, actions drawn from the behaviour policy (the policy itself, or a slightly
    older one for the clipped surrogate), distance-like rewards."""
    g = _gen(seed)
    _, n, _, obs_dim, acts, _, _ = SCENARIOS[case["scenario"]]
    dims = _dims(case)
    params = _mlps(g, case["policies"], dims)
    combos = _combos(case, seed, case["policies"])
    e, envs = case["episodes"], case["combos"] * case["envs"]
    p4 = (obs_dim + 3) // 4 * 4
    obs = torch.rand((e, STEPS, envs, n, p4), generator=g, device=DEV) * 3.0 - 1.5
    obs[..., :2] *= 0.3
    obs[..., obs_dim:] = 0.0
    pol = torch.as_tensor(combos.reshape(-1).astype(np.int64), device=DEV)
    logits = _forward(params[pol], dims, _by_slot(obs, case)[..., :obs_dim])
    if case["ppo"]:
        logits = logits + 0.08 * torch.randn(logits.shape, generator=g, device=DEV)
    u = torch.rand((*logits.shape[:2], 1), generator=g, device=DEV)
    act = (torch.softmax(logits, -1).cumsum(-1) < u).sum(-1).clamp_(max=acts - 1).to(torch.uint8)
    reward = -(torch.rand((e, STEPS, envs, n), generator=g, device=DEV) * 2.0 + 0.5)
    traj = {"obs": obs, "action": _from_slot(act, case), "reward": reward}
    if case["ppo"]:
        traj["logits"] = _from_slot(logits, case)
    return params, combos, traj


def _tables(case, seed):
    """Payoff tables as an evaluation leaves them ([games][rows][cols][4], entry 0 the mean)."""
    g = _gen(seed)
    t = torch.randn((case["games"], case["rows"], case["cols"], 4), generator=g, device=DEV, dtype=torch.float64)
    skill_r = torch.randn((case["games"], case["rows"], 1), generator=g, device=DEV, dtype=torch.float64)
    skill_c = torch.randn((case["games"], 1, case["cols"]), generator=g, device=DEV, dtype=torch.float64)
    t[..., 0] += 0.5 * (skill_r - skill_c)
    return t


def _mixtures(case, seed):
    rng = np.random.default_rng(int(seed) + 29)
    x, y = rng.random(case["rows"]), rng.random(case["cols"])
    return x / x.sum(), y / y.sum()


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind == "eval":
        s["ctx"] = _load_poker(case, _poker_population(case, _gen(seed)))
        pairs = _poker_pairs(case)
        s["seed"] = int(seed) * 7919 + 11
        s["on_host"] = bool(case["new_only"])
        s["pairs"] = pairs if s["on_host"] else torch.as_tensor(pairs, device=DEV)
        s["out"] = (np.zeros((len(pairs), 4)) if s["on_host"]
                    else torch.zeros((len(pairs), 4), dtype=torch.float64, device=DEV))
    elif kind == "rollout":
        n_pol = 32 if case["scenario"] == "spread8" else 16
        spec = _scenario_spec(case)
        s["ctx"] = _load_scenario(case, _mlps(_gen(seed), n_pol, _dims(case)), spec)
        s["spec"], s["seed"] = spec, int(seed) * 7919 + 13
        s["combos"] = torch.as_tensor(_combos(case, seed, n_pol), device=DEV)
        s["traj"] = mb.alloc_traj(spec, case["episodes"], logits=case["logits"], device=DEV)
    elif kind == "learn":
        params, combos, s["traj"] = _samples(case, seed)
        s["spec"] = _scenario_spec(case)
        s["ctx"] = _load_scenario(case, params, s["spec"])
        s["params"], s["combos"] = params, torch.as_tensor(combos, device=DEV)
        s["grad"], s["m"], s["v"] = (torch.zeros_like(params) for _ in range(3))
        s["stats"] = torch.zeros((case["policies"], 4), dtype=torch.float64, device=DEV)
        s["ids"], s["step"] = np.arange(case["policies"], dtype=np.int32), 0
    elif kind in ("fp", "lp"):
        s["ctx"], s["table"] = mb.Context(0), _tables(case, seed)
        g, m, n = case["games"], case["rows"], case["cols"]
        new = lambda *shape: torch.zeros(shape, dtype=torch.float64, device=DEV)  # noqa: E731
        s["x"], s["y"], s["bounds"], s["value"] = new(g, m), new(g, n), new(g, 2), new(g)
        s["row"], s["col"] = new(g, m), new(g, n)
    else:
        s["ctx"] = _load_poker(case, _poker_population(case, _gen(seed)))
        s["x"], s["y"] = _mixtures(case, seed)
        s["ids0"] = np.arange(case["rows"], dtype=np.int32)
        s["ids1"] = np.arange(case["rows"], case["rows"] + case["cols"], dtype=np.int32)
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "eval":
        return ctx.eval_payoff(s["pairs"], case["hands"], s["seed"], s["out"])
    if kind == "rollout":
        ctx.rollout(s["spec"], s["combos"], case["episodes"], s["seed"], s["traj"])
        return s["traj"]
    if kind == "learn":
        s["step"] += 1
        if case["ppo"]:
            ctx.learn_ppo_batch(s["spec"], s["combos"], case["episodes"], s["traj"], s["ids"], GAMMA, ENTROPY, CLIP,
                                s["grad"], s["stats"])
        else:
            ctx.learn_pg_batch(s["spec"], s["combos"], case["episodes"], s["traj"], s["ids"], GAMMA, ENTROPY, s["grad"],
                               s["stats"])
        ctx.adam_step(s["params"], s["grad"], s["m"], s["v"], s["step"], LR)
        for i in range(case["policies"]):
            ctx.pop_update(i, s["params"][i])
        return {"grad": s["grad"], "stats": s["stats"], "params": s["params"]}
    if kind == "fp":
        ctx.meta_fictitious_play(s["table"], case["iters"], s["x"], s["y"], s["bounds"], stride=4)
        ctx.meta_aggregate(s["table"], s["x"], s["y"], s["row"], s["col"], s["value"], stride=4)
        return {k: s[k] for k in ("x", "y", "bounds", "row", "col", "value")}
    if kind == "lp":
        ctx.meta_lp_nash(s["table"], s["x"], s["y"], s["value"], stride=4)
        return {k: s[k] for k in ("x", "y", "value")}
    return np.array(ctx.exploitability(s["ids0"], s["x"], s["ids1"], s["y"]))


# ------------------------------------------------------------------ work and tolerance

def _mlp_flops(dims):
    i, h1, h2, o = dims
    return 2.0 * (i * h1 + h1 * h2 + h2 * o)


def work(case):
    kind = case["kind"]
    if kind == "eval":
        pairs = len(_poker_pairs(case))
        if case["game"] == "kuhn":
            # a deal and 2.3 decisions per hand, each a counter-based draw of about 80 integer operations
            return {"bytes": pairs * 40.0 + 24.0 * (case["rows"] + case["cols"]), "flops": pairs * case["hands"] * 3.3 * 80}
        d = _dims(case)
        size = (_mlp_flops(d) / 2) * (2 if case["game"] == "leduc_bf16" else 4)
        return {"bytes": pairs * 40.0 + size * (case["rows"] + case["cols"]),
                "flops": pairs * case["hands"] * 4.0 * _mlp_flops(d)}
    if kind in ("rollout", "learn"):
        _, n, _, obs, acts, _, dt = SCENARIOS[case["scenario"]]
        steps = case["episodes"] * STEPS * case["combos"] * case["envs"]
        if kind == "rollout":
            row = (obs + 3) // 4 * 16 + 5 + (4 * acts if case["logits"] else 0)
            return {"bytes": steps * (n * row + 1.0), "flops": steps * n * _mlp_flops(_dims(case))}
        i, h, _, o = _dims(case)
        per = _mlp_flops(_dims(case)) + 2.0 * (2 * h * o + 2 * h * h + h * i)
        return {"bytes": steps * n * (4.0 * obs + 5 + (20 if case["ppo"] else 0)), "flops": steps * n * per}
    g, m, n = case.get("games", 1), case["rows"], case["cols"]
    if kind == "fp":
        return {"bytes": g * 8.0 * (m * n + 2 * (m + n)), "flops": g * (case["iters"] * (m + n) + 4.0 * m * n)}
    if kind == "lp":
        # as many pivots as the smaller side, each a rank-one update of the table
        return {"bytes": g * 8.0 * (m * n + m + n), "flops": g * 2.0 * m * n * min(m, n)}
    if case["game"] == "kuhn":
        return {"bytes": 32.0 * (m + n), "flops": 100.0 * (m + n)}
    d = _dims(case)
    return {"bytes": (m + n) * (_mlp_flops(d) / 2) * (2 if case["game"] == "leduc_bf16" else 4),
            "flops": (m + n) * 144 * _mlp_flops(d)}


def tolerance(case):
    """Sampled paths draw actions by comparing a softmax with a uniform number: where another
    correct order of the forward's sums moves a probability across its number, that hand or
    episode goes another way. Measured by permuting the policies' hidden units, which changes
    nothing but the order of the sums: fp32 policies, no such hand or episode in most calls and
    logits 1.6e-7 apart; bf16 Leduc, 1.9e-4 (largest 2.4e-3) at 65 x 2,000 hands and 9.7e-6
    (4.6e-4) at 4,096 x 16,384; bf16 spread, 2.3e-4 (0.27; 3e-7 of the actions) at 131,072
    episodes. The tolerances let a few hands or episodes of the call go another way."""
    kind = case["kind"]
    if kind == "eval":
        if case["game"] == "kuhn":
            return "exact"                      # integer sums of hands drawn from tables
        return {"rel": min(0.03, 40.0 / (case["hands"] * math.sqrt(len(_poker_pairs(case))))),
                "max": min(0.9, 40.0 / case["hands"])}
    if kind == "rollout":
        n = case["episodes"] * case["combos"] * case["envs"]
        return {"rel": min(0.03, 1e-5 + 0.4 / math.sqrt(n)), "max": 0.99, "differ": min(0.01, 2.0 / n)}
    if kind == "learn":
        # the gradient is a small mean of terms of both signs: 1.3e-4 from 64 bits at 3 M samples
        return {"rel": 5e-4, "max": 0.02}
    if kind == "fp":
        return {"rel": 1e-12, "max": 1e-11}     # sums in play order; the plays themselves are whole
    if kind == "lp":
        return {"rel": 1e-10, "max": 1e-9}      # 1e-14 from 64 bits in another elimination order
    return {"rel": 1e-3, "max": 1e-3} if case["game"] == "leduc_bf16" else {"rel": 1e-6, "max": 1e-6}


# ------------------------------------------------------------------ the same in 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind == "eval":
        # Leduc entries are sums over hands whose draws compare an fp32 softmax with a number:
        # they have no value in 64 bits. Kuhn's draws compare stored table entries.
        return _exact_kuhn(case, seed) if case["game"] == "kuhn" else None
    if kind == "rollout":
        return None                             # the same: every step follows from drawn actions
    if kind == "learn":
        return _exact_learn(case, seed)
    if kind == "fp":
        return _exact_fp(case, seed)
    if kind == "lp":
        return _exact_lp(case, seed)
    if case["game"] == "leduc_bf16":
        return None                             # bf16 layer inputs: rounding is part of the policy
    return _exact_exploit(case, seed)


def _philox(g, step, agent, seed):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF
    c = [g & mask, (g >> 32) & mask, torch.full_like(g, step), torch.full_like(g, agent)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _exact_kuhn(case, seed):
    pairs, n = _poker_pairs(case), case["hands"]
    if len(pairs) * n > 200_000_000:
        return None
    table = _poker_population(case, _gen(seed)).double()
    s = int(seed) * 7919 + 11
    out = np.zeros((len(pairs), 4))
    for k, (p0, p1) in enumerate(pairs):
        g = torch.arange(k * n, (k + 1) * n, device=DEV, dtype=torch.int64)
        x = _philox(g, 0, 0xFFFFFFFF, s)
        c0 = (x[0] * 3) >> 32
        j = (x[1] * 2) >> 32
        c1 = j + (j >= c0)
        u = [(_philox(g, t, a, s)[0] >> 8).double() * 2.0 ** -24 for t, a in ((0, 0), (1, 1), (2, 0))]
        sd = torch.where(c0 > c1, 1, -1)
        a0 = (u[0] < table[p0][2 * c0]).long()
        a1 = u[1] < table[p1][2 * c1 + a0]
        a2 = u[2] < table[p0][2 * c0 + 1]
        pay = torch.where(a0 == 1, torch.where(a1, 2 * sd, 1), torch.where(a1, torch.where(a2, 2 * sd, -1), sd))
        s1, s2 = float(pay.sum()), float((pay * pay).sum())
        se = math.sqrt(max(0.0, (s2 - s1 * s1 / n) / (n - 1)) / n) if n > 1 else 0.0
        out[k] = (s1 / n, se, s1, s2)
    return out


def _exact_learn(case, seed):
    params, combos, traj = _samples(case, seed)
    dims = _dims(case)
    obs_dim = dims[0]
    x = _by_slot(traj["obs"], case)[..., :obs_dim]
    act = _by_slot(traj["action"], case).long()
    r = traj["reward"].double()
    ret, acc = torch.zeros_like(r), torch.zeros_like(r[:, 0])
    for t in range(STEPS - 1, -1, -1):
        acc = r[:, t] + np.float64(np.float32(GAMMA)) * acc
        ret[:, t] = acc
    ret = _by_slot(ret, case)
    behave = _by_slot(traj["logits"], case) if case["ppo"] else None
    slot_pol = combos.reshape(-1)
    beta, clip = float(np.float32(ENTROPY)), float(np.float32(CLIP))
    grads, stats, news = [], [], []
    for p in range(case["policies"]):
        theta = params[p].double().requires_grad_(True)
        mine = [int(k) for k in np.nonzero(slot_pol == p)[0]]
        total = len(mine) * x.shape[1]
        base = float(sum(ret[k].sum() for k in mine)) / total if total else 0.0
        loss_sum, ent_sum, grad = 0.0, 0.0, torch.zeros_like(theta)
        for k in mine:
            z = _forward(theta[None], dims, x[k].double()[None])[0]
            logp = torch.log_softmax(z, -1)
            ent = -(logp.exp() * logp).sum(-1)
            lp = logp.gather(1, act[k][:, None])[:, 0]
            adv = ret[k] - base
            if case["ppo"]:
                rho = (lp - torch.log_softmax(behave[k].double(), -1).gather(1, act[k][:, None])[:, 0]).exp()
                gain = torch.minimum(rho * adv, rho.clamp(1 - clip, 1 + clip) * adv)
            else:
                gain = adv * lp
            loss = -(gain + beta * ent).sum() / total
            grad += torch.autograd.grad(loss, theta)[0]
            loss_sum += float(loss.detach())
            ent_sum += float(ent.detach().sum()) / total
        b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
        m, v = (1 - b1) * grad, (1 - b2) * grad * grad
        step = float(np.float32(LR)) * (m / (1 - b1)) / ((v / (1 - b2)).sqrt() + float(np.float32(1e-8)))
        grads.append(grad)
        news.append(theta.detach() - step)
        stats.append([float(total), base, loss_sum, ent_sum])
    return {"grad": torch.stack(grads), "stats": torch.tensor(stats, dtype=torch.float64), "params": torch.stack(news)}


def _exact_fp(case, seed):
    a = _tables(case, seed)[..., 0].cpu().numpy()
    g, m, n = a.shape
    if case["iters"] * g * (m + n) > 4e8:
        return None
    ar = np.arange(g)
    ur, uc = np.zeros((g, m)), np.zeros((g, n))
    x, y = np.zeros((g, m)), np.zeros((g, n))
    i, j = np.zeros(g, np.int64), np.zeros(g, np.int64)
    for _ in range(case["iters"]):
        x[ar, i] += 1
        y[ar, j] += 1
        ur += a[ar, :, j]
        uc += a[ar, i, :]
        i, j = ur.argmax(1), uc.argmin(1)
    t = float(case["iters"])
    x, y = x / t, y / t
    row, col = np.einsum("gij,gj->gi", a, y), np.einsum("gi,gij->gj", x, a)
    return {"x": x, "y": y, "bounds": np.stack([uc.min(1) / t, ur.max(1) / t], 1), "row": row, "col": col,
            "value": (x * row).sum(1)}


def _exact_lp(case, seed):
    a = _tables(case, seed)[..., 0].cpu().numpy()
    xs, ys, vs = [], [], []
    for t in a:
        m, n = t.shape
        shift = 1.0 - t.min()
        tab = np.zeros((m + 1, n + m + 1))
        tab[:m, :n], tab[:m, n:n + m], tab[:m, -1], tab[m, :n] = t + shift, np.eye(m), 1.0, -1.0
        basis = np.arange(n, n + m)
        for _ in range(50 * (m + n)):
            q = int(tab[m, :-1].argmin())
            if tab[m, q] > -1e-12:
                break
            col = tab[:m, q]
            ratio = np.where(col > 1e-12, tab[:m, -1] / np.where(col > 1e-12, col, 1.0), np.inf)
            p = int(ratio.argmin())
            tab[p] /= tab[p, q]
            f = tab[:, q].copy()
            f[p] = 0.0
            tab -= f[:, None] * tab[p][None, :]
            basis[p] = q
        v = 1.0 / tab[m, -1]
        y = np.zeros(n + m)
        y[basis] = tab[:m, -1] * v
        xs.append(tab[m, n:n + m] * v)
        ys.append(y[:n])
        vs.append(v - shift)
    return {"x": np.array(xs), "y": np.array(ys), "value": np.array(vs)}


def _exact_exploit(case, seed):
    params = _poker_population(case, _gen(seed)).double().cpu().numpy()
    x, y = _mixtures(case, seed)
    seat = [params[:case["rows"]], params[case["rows"]:]]
    best = [_best_response(case, 0, seat[1], y), _best_response(case, 1, seat[0], x)]
    return np.array([best[0], best[1], 0.5 * (best[0] + best[1])])


def _best_response(case, br, opp, w):
    """Value of the best response of seat br against the mixture (opp, w): backward induction
    over the public tree, carrying each hidden card's probability times the members' reach."""
    sign = 1.0 if br == 0 else -1.0
    if case["game"] == "kuhn":
        def kuhn(own, h, reach):
            if h in ("pp", "pbp", "pbb", "bp", "bb"):
                total = 0.0
                for c, v in reach.items():
                    win = 1 if (own if br == 0 else c) > (c if br == 0 else own) else -1
                    total += v @ w * sign * {"pp": win, "pbp": -1, "pbb": 2 * win, "bp": 1, "bb": 2 * win}[h]
                return total
            actor, facing = {"": (0, 0), "p": (1, 0), "b": (1, 1), "pb": (0, 1)}[h]
            if actor == br:
                return max(kuhn(own, h + a, reach) for a in "pb")
            return sum(kuhn(own, h + a, {c: v * (opp[:, 2 * c + facing] if a == "b" else 1 - opp[:, 2 * c + facing])
                                         for c, v in reach.items()}) for a in "pb")
        return sum(kuhn(own, "", {c: np.full(len(w), 1 / 6) for c in range(3) if c != own}) for own in range(3))

    d = _dims(case)
    cuts = np.cumsum([d[1] * d[0], d[1], d[2] * d[1], d[2], d[3] * d[2]])
    w1, b1, w2, b2, w3, b3 = np.split(opp, cuts, axis=1)
    w1, w2, w3 = (v.reshape(len(opp), o, i) for v, o, i in ((w1, d[1], d[0]), (w2, d[2], d[1]), (w3, d[3], d[2])))
    known = {}

    def probs(rank, pub, rnd, con, raises, legal):
        """[members][3] of the acting opponent."""
        key = (rank, pub, rnd, con, raises, legal)
        if key not in known:
            o = np.zeros(17)
            o[rank] = o[3 + (pub if rnd else 3)] = o[7 + rnd] = o[11 + raises] = 1.0
            o[9], o[10] = np.float32(con[0]) / np.float32(13), np.float32(con[1]) / np.float32(13)
            o[14:17] = legal
            h = np.maximum(w1 @ o + b1, 0)
            h = np.maximum(np.einsum("pij,pj->pi", w2, h) + b2, 0)
            z = np.where(np.array(legal) > 0, np.einsum("pij,pj->pi", w3, h) + b3, -np.inf)
            e = np.exp(z - z.max(1, keepdims=True))
            known[key] = e / e.sum(1, keepdims=True)
        return known[key]

    def walk(own, pub, rnd, con, raises, acted, actor, reach):
        """con: both seats' contributions; reach: {opponent card: [members]}."""
        me, other = con[actor], con[1 - actor]
        legal = (int(other > me), 1, int(raises < 2))

        def after(a, reach):
            c = list(con)
            if a == 0:
                pay = -con[0] if actor == 0 else con[1]
                return sum(float(v @ w) for v in reach.values()) * sign * pay
            if a == 2:
                c[actor] = other + (2, 4)[rnd]
                return walk(own, pub, rnd, tuple(c), raises + 1, acted + 1, 1 - actor, reach)
            c[actor] = other
            if acted + 1 < 2:
                return walk(own, pub, rnd, tuple(c), raises, acted + 1, 1 - actor, reach)
            if rnd == 0:
                total = 0.0
                for p in range(6):
                    left = {k: v * 0.25 for k, v in reach.items() if k != p}
                    if p != own and left:
                        total += walk(own, p, 1, tuple(c), 0, 0, 0, left)
                return total
            total = 0.0
            for k, v in reach.items():
                r0, r1 = (own // 2, k // 2) if br == 0 else (k // 2, own // 2)
                win = 1 if r0 == pub // 2 else -1 if r1 == pub // 2 else (r0 > r1) - (r0 < r1)
                total += float(v @ w) * sign * (c[1] if win > 0 else -c[0] if win < 0 else 0)
            return total

        acts = [a for a in range(3) if legal[a]]
        if actor == br:
            return max(after(a, reach) for a in acts)
        pr = {k: probs(k // 2, pub // 2, rnd, (me, other), raises, legal) for k in reach}
        return sum(after(a, {k: v * pr[k][:, a] for k, v in reach.items()}) for a in acts)

    return sum(walk(own, 0, 0, (1, 1), 0, 0, 0, {k: np.full(len(w), 1 / 30) for k in range(6) if k != own})
               for own in range(6))
