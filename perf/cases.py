"""Performance cases: what users of this framework have it do, each through its public entry points.

Every case names one kind of call (see _KINDS), a board shape and the rules it plays under:

  step      one `Env.step` of every environment, actions chosen by the caller (RL acting, evaluation)
  rollout   `Env.rollout`, fused random-policy steps, with the per-step trajectory or, as in fitness
            evaluation, only the reward sums and the boards reached (`Env.get_state`)
  variant   `Env.rollout` with each rule applied once per step by random key and inhibiting the next
  expand    `Env.expand`, every frontier board stepped by all five actions
  search    `Env.search`, a whole best-first search (init, then expand and select per iteration)
  observe   `Env.observe`, the player-centred policy input
  mutate    `av_mutate`, the evolution loop's offspring, in place on maps and rule tables

Boards are drawn by `Env.reset`; rules come from the same distributions as the repository's workloads,
generated here on the GPU so that a state is made quickly.  Episodes end when no goal tile is left or after
200 steps and restart from the environment's own map, so repeated passes stay in the regime a long run is in.
All outputs are whole numbers and bytes and have to stay the same bit for bit (so there is no `exact`).
"""
import numpy as np
import torch

import paper_2407_04221_gb300 as av
import workload as wk

DEVICE = "cuda"
SHAPES = {  # pattern sizes (uniform) with the present / absent rate of an input entry
    "mixed": (((1, 2), (1, 3), (3, 3)), 0.15, 0.15),  # fire often
    "3x3": (((3, 3),), 0.15, 0.15),                   # almost never match by chance: play is the base game's
    "large": (((3, 3), (5, 5)), 0.03, 0.02),          # sparse enough to fire on most steps
}


def _case(kind, name=None, **kw):
    base = dict(kind=kind, batch=1, H=16, W=16, C=8, R=8, rules="3x3", base_game=True, shared=False, init="dirichlet")
    base.update(kw)
    return base if name is None else dict(base, name=name)


def listed():
    return [
        # one environment stepped by an interactive agent: the smallest call, all latency
        _case("step", "step-one-maze16", C=4, R=3, shared=True, init="maze"),
        # the acting step of RL training: 16,384 environments, two-byte cells, rules that fire often
        _case("step", "step-train-16384x16x16", batch=16384, C=10, R=12, rules="mixed", base_game=False),
        # odd, ragged boards past 512 cells (an evaluation set of larger maps)
        _case("step", "step-ragged-1000x23x41", batch=1000, H=23, W=41, C=12, R=16, rules="large"),
        # the RL training rollout with its trajectory of observations, rewards and done flags
        _case("rollout", "rollout-train-16384x16x16", batch=16384, C=10, R=12, rules="mixed", base_game=False,
              steps=500, trajectory=True),
        # fitness of 1,024 evolved games under a random player who moves: rewards and final boards only
        _case("rollout", "rollout-play-1024x16x16", batch=1024, steps=1000, trajectory=False),
        # large boards, many rules, most steps rewriting the board
        _case("rollout", "rollout-4096x64x64", batch=4096, H=64, W=64, C=16, R=24, rules="large", steps=100,
              trajectory=False),
        # the largest boards, beyond one CTA's shared memory
        _case("rollout", "rollout-256x256x256", batch=256, H=256, W=256, C=16, R=24, rules="large", steps=20,
              trajectory=False),
        # variant semantics: random application order, inhibition
        _case("variant", "variant-1024x16x16", batch=1024, steps=200, trajectory=False),
        # one expansion of a full frontier
        _case("expand", "expand-64x256x16x16", batch=64, frontier=256, init="maze"),
        # a whole search: frontiers grow from one board to 256, states repeat
        _case("search", "search-64x256-50", batch=64, frontier=256, iterations=50, init="maze"),
        # the policy input of the training shape, whole board visible
        _case("observe", "observe-16384-w31", batch=16384, C=10, R=2, shared=True, window=31),
        # offspring of 16,384 games
        _case("mutate", "mutate-16384x16x16", batch=16384, C=10, R=12, rules="mixed"),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One more case of the ranges above: any kind, batch 1 to 16,384, boards 5x5 to 64x64 (rollouts and steps
    sometimes up to 256x256), one- and two-byte cells, shared or own rule tables, small to large patterns."""
    kind = rng.choice(("step", "step", "rollout", "rollout", "variant", "expand", "search", "observe", "mutate"))
    small = kind in ("expand", "search")
    big = kind in ("step", "rollout") and rng.random() < 0.2
    H, W = ((rng.randint(65, 200), rng.randint(65, 256)) if big else
            (_log(rng, 5, 32), _log(rng, 5, 32)) if small else (_log(rng, 5, 64), _log(rng, 5, 64)))
    C = rng.randint(4, 16)
    R = rng.randint(2, 24)
    cells = H * W
    case = _case(kind, H=H, W=W, C=C, R=R, rules=rng.choice(sorted(SHAPES)), base_game=rng.random() < 0.7,
                 shared=rng.random() < 0.3, init=rng.choice(("maze", "dirichlet")))
    most = max(1, min(16384, 4_000_000 // cells, 150_000 // R))  # boards in all, rule tables in all
    if kind in ("rollout", "variant"):
        case["batch"] = _log(rng, 1, most)
        budget = (8e9 if kind == "rollout" else 4e8) / (case["batch"] * cells * R)  # steps that stay below the listed
        case["steps"] = max(1, min(_log(rng, 5, 1000), int(budget)))
        case["trajectory"] = rng.random() < 0.5 and case["batch"] * cells * case["steps"] < 5e8
    elif kind in ("expand", "search"):
        case["base_game"] = True
        case["batch"] = _log(rng, 1, 64)
        case["frontier"] = max(4, min(_log(rng, 4, 256), 4_000_000 // (case["batch"] * cells)))
        if kind == "search":
            case["iterations"] = rng.randint(3, 50)
    else:
        case["batch"] = _log(rng, 1, most)
        if kind == "observe":
            case["window"] = _log(rng, 3, 63)
            case["batch"] = max(1, min(case["batch"], 150_000_000 // (case["window"] ** 2 * C)))
    return case


def _ncell_bytes(case):
    return 1 if case["C"] <= 8 else 2


def _entries(case):
    """Average entries of a base pattern."""
    shapes = SHAPES[case["rules"]][0]
    return sum(h * w for h, w in shapes) / len(shapes)


def _make_rules(gen, case):
    """Packed rule tables [n_tables, R] of 408-byte records: pattern size uniform over the kind's shapes, input
    entries present / absent at its rates, outputs set / clear at 0.1 / 0.1, rewards in -3..3; with base_game
    the first two rules are the maze game's move and eat."""
    n = 1 if case["shared"] else case["batch"]
    R, C = case["R"], case["C"]
    shapes, p_pres, p_abs = SHAPES[case["rules"]]
    pick = torch.randint(len(shapes), (n, R), generator=gen, device=DEVICE)
    sizes = torch.tensor(shapes, device=DEVICE, dtype=torch.int32)
    hw = sizes[pick]
    rec = torch.zeros(n, R, 102, dtype=torch.int32, device=DEVICE)
    rec[:, :, 0] = hw[:, :, 0] | (hw[:, :, 1] << 8)
    rec[:, :, 1] = torch.randint(-3, 4, (n, R), generator=gen, device=DEVICE, dtype=torch.int32)
    inside = torch.arange(25, device=DEVICE) < (hw[:, :, 0] * hw[:, :, 1])[:, :, None]
    for c in range(C + 1):
        u = torch.rand(n, R, 25, generator=gen, device=DEVICE)
        rec[:, :, 2:27] |= ((u < p_pres) & inside).int() << c
        rec[:, :, 27:52] |= ((u >= p_pres) & (u < p_pres + p_abs) & inside).int() << c
        if c < C:
            u = torch.rand(n, R, 25, generator=gen, device=DEVICE)
            rec[:, :, 52:77] |= ((u < 0.1) & inside).int() << c
            rec[:, :, 77:102] |= ((u >= 0.1) & (u < 0.2) & inside).int() << c
    out = np.ascontiguousarray(rec.cpu().numpy()).view(wk.RULE_DTYPE).reshape(n, R)
    if case["base_game"] and R >= 2:
        out[:, :2] = wk.base_game_rules(C)
    return out


def _make_cum(gen, case):
    """Initial-map thresholds: floor / wall / goal 0.7 / 0.25 / 0.05 for every environment, or per environment
    Dirichlet(1) over the types but the player's."""
    C = case["C"]
    n = 1 if case["init"] == "maze" else case["batch"]
    if case["init"] == "maze":
        share = torch.zeros(1, C, dtype=torch.float64, device=DEVICE)
        share[0, wk.CH_EMPTY], share[0, wk.CH_WALL], share[0, wk.CH_GOAL] = 0.7, 0.25, 0.05
    else:
        u = torch.rand(n, C, generator=gen, device=DEVICE, dtype=torch.float64)
        share = -torch.log1p(-u)
        share[:, wk.CH_PLAYER] = 0.0
        share /= share.sum(1, keepdim=True)
    cum = (share.cumsum(1) * wk.ONE24).round().clamp(0, wk.ONE24).to(torch.int64)
    cum[:, -1] = wk.ONE24
    return cum.cpu().numpy().astype(np.uint32)


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    fields = dict(batch=case["batch"], H=case["H"], W=case["W"], C=case["C"], n_rules=case["R"],
                  rules_per_env=0 if case["shared"] else 1, max_steps=200, auto_reset=1, ch_player=wk.CH_PLAYER,
                  ch_goal=wk.CH_GOAL, ch_empty=wk.CH_EMPTY, ch_wall=wk.CH_WALL, border_wall=1,
                  cum_per_env=0 if case["init"] == "maze" else 1)
    rules, cum = _make_rules(gen, case), _make_cum(gen, case)
    kind, B = case["kind"], case["batch"]
    capacity = 1 + case["iterations"] * case["frontier"] if kind == "search" else 0
    s = dict(case=case, seed=seed, calls=0)
    if kind == "mutate":  # the parents, on the device as the evolution loop keeps them; every game has its tables
        fields["n_rules"], maker = 0, None
        env = av.Env(fields, rules[:, :0], cum)
        s["maps"] = env.reset(seed)
        s["rules"] = torch.from_numpy(rules.view(np.uint8).reshape(rules.shape[0], case["R"], av.RULE_BYTES)).to(DEVICE)
        if case["shared"]:
            s["rules"] = s["rules"].expand(B, -1, -1).contiguous()
        env.close()
        bits = case["H"] * case["W"] * case["C"]
        s["rates"] = dict(p_map=max(1, (10 << 24) // bits), map_channels=(1 << case["C"]) - 1, p_rule=1 << 21,
                          p_reward=1 << 22, reward_min=-3, reward_max=3,
                          mutable_rules=((1 << case["R"]) - 1) & ~(3 if case["base_game"] else 0))
        return s
    env = s["env"] = av.Env(fields, rules, cum, search_capacity=capacity)
    boards = env.reset(seed)
    if kind == "step":
        s["actions"] = [torch.randint(5, (B,), generator=gen, device=DEVICE, dtype=torch.uint8) for _ in range(8)]
    elif kind == "variant":
        R = case["R"]
        av.av_set_variant(env.h, random_keys=1, key_seed=seed, limit=[1] * R,
                          inhibit=[1 << ((r + 1) % R) for r in range(R)])
    elif kind == "expand":  # a frontier as a search has it: boards of each game a few moves apart
        walk = env.rollout(case["frontier"], seed, trajectory=True)["obs"]
        s["parents"] = walk.transpose(0, 1).contiguous()
    elif kind == "search":
        s["roots"] = boards
    elif kind == "observe":  # boards in mid-game
        env.rollout(60, seed)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    s["calls"] += 1
    if kind == "step":
        return s["env"].step(s["actions"][s["calls"] % 8])
    if kind in ("rollout", "variant"):
        out = s["env"].rollout(case["steps"], s["seed"] + s["calls"], trajectory=case["trajectory"])
        if case["trajectory"]:
            return out
        return out["rew_sum"], s["env"].get_state()
    if kind == "expand":
        return s["env"].expand(s["parents"])
    if kind == "search":
        return s["env"].search(s["roots"], case["iterations"], case["frontier"])
    if kind == "observe":
        return s["env"].observe(case["window"])
    av.av_mutate(case["batch"], case["H"], case["W"], case["C"], case["R"], s["rates"], s["seed"] + s["calls"],
                 s["maps"], s["rules"])
    return s["maps"], s["rules"]


def work(case):
    """Bytes only: the operations are bit tests, not arithmetic on a unit with a stated rate.  Boards, rewards
    and flags in and out once; of a rule table the four 32-bit masks of each pattern entry and its reward."""
    B, board = case["batch"], case["H"] * case["W"] * _ncell_bytes(case)
    tables = (1 if case["shared"] else B) * case["R"] * (16 * _entries(case) + 8)
    kind = case["kind"]
    if kind == "step":
        n = tables + B * (3 * board + 1 + 4 + 1 + 8)  # board in and out, its observation; action, reward, done, t
    elif kind in ("rollout", "variant"):
        n = tables + B * (3 * board + 4 + 8)  # boards in, out, and the initial maps
        n += B * case["steps"] * (board + 5) if case["trajectory"] else B * (2 * board + 8)  # get_state copies them
    elif kind == "expand":
        n = tables + B * case["frontier"] * (board + 5 * (board + 4 + 1 + 8))
    elif kind == "search":  # the final frontier has to be found and written; the states between are on the way
        n = tables + B * (case["iterations"] * case["frontier"] * (6 * board + 5 * 13) * 0.5 + case["frontier"] * board)
    elif kind == "observe":
        n = B * (board + case["window"] ** 2 * case["C"] + 8)
    else:
        n = 2 * B * (board + case["R"] * (16 * _entries(case) + 8))
    return {"bytes": float(n), "flops": 0.0}


def tolerance(case):
    return "exact"
