"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one call (or the calls of one frame) through the public binding
(`paper_2606_23348_gb300.generals`): stepping a batch with the fused benchmark
policy, rolling several frames out in one call, sampling actions from logits,
stepping with the feature tensor, the whole self-play frame, regenerating
maps, and the host-buffer step.  Boards, modes and counts are those of the
workloads, tests and benchmark of this repository, and `draw` gives others of
the same ranges.  Games are taken at mid-game (256 frames of the benchmark
policy after their first map) and are truncated at 512 turns, so that long
runs keep meeting opening, middle and restart.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2606_23348_gb300 import workloads
from paper_2606_23348_gb300.generals import GeneralsEnv, Outputs

MODES = {"1v1": ((0, 1.0),), "2v2": ((1, 1.0),), "ffa": ((2, 1.0),), "mixed": ((0, 0.4), (1, 0.3), (2, 0.3))}
# the map rules: the plain generator, BFS spacing, the spawn-distance
# curriculum's first cap, and BFS spacing with the castle guarantee
MAPS = {"plain": {}, "bfs": dict(bfs_distance=1, min_general_dist=17),
        "cap": dict(bfs_distance=1, min_general_dist=1, max_general_dist=4),
        "castle": dict(bfs_distance=1, min_general_dist=17, castle_radius=6)}
MAX_TURNS = 512
PREROLL = 256
POLICY_SEED = 2
HIST, WINDOW = 7, 512  # 38 channels and 512-frame temporal tokens
OWN_CELLS = 45  # cells a player holds at mid-game of a 24x24 1v1 game


def _case(kind, games, lo, hi, modes="1v1", maps="plain", castles=-1, frames=1, mask=False, ffa_players=8):
    return dict(kind=kind, games=games, side_lo=lo, side_hi=hi, modes=modes, maps=maps, castles=castles,
                frames=frames, mask=mask, ffa_players=ffa_players)


def listed():
    cases = {
        # a handful of small games, one step a call: an agent trying things out, latency and launches only
        "step-64-15x15": _case("step", 64, 15, 15, castles=8),
        # one frame of a self-play rollout at 512 games: sample, step, feature tensor and tokens
        "selfplay-512-24x24": _case("selfplay", 512, 24, 24, castles=12),
        # the benchmark's batch: every game of a large uniform 1v1 environment, one step a call
        "step-65536-24x24": _case("step", 65536, 24, 24, castles=12),
        # training over every board size and mode at once
        "step-32768-mixed20to40": _case("step", 32768, 20, 40, "mixed"),
        # training on maps with BFS spacing and a castle near every general
        "step-16384-24x24-castle": _case("step", 16384, 24, 24, maps="castle", castles=12),
        # a few games played ahead for many frames in one call
        "rollout-1024-24x24x64": _case("rollout", 1024, 24, 24, castles=12, frames=64),
        # many ragged games played ahead in one call
        "rollout-32768-ragged15to30x16": _case("rollout", 32768, 15, 30, frames=16),
        # actions from a policy head's logits for a large batch
        "sample-65536-24x24": _case("sample", 65536, 24, 24, castles=12),
        # the same with team and eight-player games, and the expanded mask that a policy loss needs
        "sample-mask-8192-mixed20to40": _case("sample", 8192, 20, 40, "mixed", mask=True),
        # one frame of a large training batch without sampling: step, feature tensor and tokens
        "features-16384-24x24": _case("features", 16384, 24, 24, castles=12),
        # a new set of maps under the full map rules for a large batch
        "reset-65536-24x24-castle": _case("reset", 65536, 24, 24, maps="castle", castles=12),
        # actors that live on the host: actions in, every output back, through pinned buffers
        "host-65536-24x24": _case("host", 65536, 24, 24, castles=12),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "rollout", "rollout", "sample", "sample", "features", "selfplay", "reset",
                       "host"])
    lo = rng.randint(10, 40)
    hi = lo if rng.random() < 0.5 else rng.randint(lo, 40)
    modes = rng.choice(["1v1", "1v1", "2v2", "ffa", "mixed"])
    maps = rng.choice(["plain", "plain", "plain", "bfs", "cap", "castle"])
    players = rng.randint(3, 8)
    frames = round(math.exp(rng.uniform(math.log(2), math.log(64)))) if kind == "rollout" else 1
    # as many games as keep the case's per-player cells (over all frames) within those of the listed cases
    per_game = {"1v1": 2, "2v2": 4, "ffa": players, "mixed": 0.4 * 2 + 0.3 * 4 + 0.3 * players}[modes]
    cells = per_game * (16 + ((lo + hi) / 2) ** 2 + (hi - lo) ** 2 / 12) * frames
    most = {"step": 1.2e8, "rollout": 4e8, "sample": 5e7, "features": 1.6e7, "selfplay": 1.6e7, "reset": 4e7,
            "host": 5e7}[kind]
    top = min(65536, int(most / cells))
    games = round(math.exp(rng.uniform(math.log(min(64, top)), math.log(top))))
    return _case(kind, games, lo, hi, modes, maps, castles=rng.choice([-1, -1, 8, 12]), frames=frames,
                 mask=kind == "sample" and rng.random() < 0.5, ffa_players=players)


# ---- shapes ------------------------------------------------------------------
def _shapes(case):
    """Per-game H, W, mode and players: the case's own, the same for every seed."""
    return workloads.shapes(case["games"], (case["side_lo"], case["side_hi"]), MODES[case["modes"]], seed=0,
                            ffa_players=case["ffa_players"])


def _params(case, seed):
    per_mille = 30 if case["modes"] == "mixed" else 20  # castles by area where their number is not given
    return dict(dict(seed=seed + 1, n_cities=case["castles"], city_per_mille=per_mille, max_turns=MAX_TURNS),
                **MAPS[case["maps"]])


def _environment(case, seed):
    H, W, mode, players = _shapes(case)
    return GeneralsEnv(H, W, mode, players, **_params(case, seed))


# ---- inputs ------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    env = _environment(case, seed)
    s = dict(kind=kind, env=env, frames=case["frames"], actions=env.new_actions(), out=env.new_outputs(case["frames"]))
    if kind in ("features", "selfplay"):
        s["features"] = env.features(HIST, WINDOW)
        s["tensor"], s["tokens"] = s["features"].new_output(), s["features"].new_series()
    if kind == "features":  # a position with its history behind it, every player waiting in the first frame
        for board in _positions(case, seed):
            env.write_state(*board)
            s["features"].build(s["tensor"], s["tokens"])
    elif kind != "reset":
        one = s["out"] if case["frames"] == 1 else env.new_outputs()
        env.policy(POLICY_SEED, s["actions"])
        for _ in range(PREROLL):
            env.step_policy(s["actions"], one, POLICY_SEED, s["actions"])
    if kind in ("sample", "selfplay"):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        spread = 2.0 if kind == "sample" else 1.0
        s["logits"] = torch.randn(int(env.layout.plane_cells) * 9, generator=gen, device="cuda").mul_(spread)
        s["seed"] = seed
    if kind == "sample":
        s["mask9"] = torch.empty(int(env.layout.plane_cells) * 9, dtype=torch.uint8, device="cuda") if case["mask"] \
            else None
    if kind == "host":
        s["h_out"] = Outputs(env.layout, pin_host=True)
        s["h_actions"] = s["actions"].cpu().pin_memory()
    return s


def run(s):
    kind, env, actions, out = s["kind"], s["env"], s["actions"], s["out"]
    if kind == "step":
        env.step_policy(actions, out, POLICY_SEED, actions)
        return [actions, *out.tensors()]
    if kind == "rollout":
        env.rollout(s["frames"], POLICY_SEED, actions, out)
        return [actions, *out.tensors()]
    if kind == "sample":
        env.sample_actions(s["logits"], s["seed"], actions, s["mask9"])
        return [actions] if s["mask9"] is None else [actions, s["mask9"]]
    if kind == "features":
        env.step_policy(actions, out, POLICY_SEED, actions)
        s["features"].build(s["tensor"], s["tokens"])
        return [s["tensor"], s["tokens"], actions, *out.tensors()]
    if kind == "selfplay":
        env.sample_actions(s["logits"], s["seed"], actions)
        env.step(actions, out)
        s["features"].build(s["tensor"], s["tokens"])
        return [s["tensor"], s["tokens"], actions, *out.tensors()]
    if kind == "reset":
        env.reset(out)
        return list(out.tensors())
    if kind == "host":
        env.step_host(s["h_actions"], s["h_out"], POLICY_SEED, s["h_actions"])
        return [s["h_actions"], *s["h_out"].tensors()]
    raise ValueError(kind)


def work(case):
    """Bytes of one pass: state, inputs and outputs once each (the sampler's
    logits: those of the cells a player holds); no contraction anywhere."""
    H, W, _, P = (x.astype(np.int64) for x in _shapes(case))
    npad = (H * W + 15) // 16 * 16
    G, cells, plane, slots = int(case["games"]), int(npad.sum()), int((P * npad).sum()), int(P.sum())
    kind, K = case["kind"], case["frames"]
    table = 32 * G  # the counters of every game
    outputs = 6 * plane + 12 * slots + G
    step = 2 * 4 * cells + 2 * table + 2 * 4 * slots + outputs
    sample = 4 * cells + table + 4 * slots + 36 * int((P * np.minimum(H * W // 2, OWN_CELLS)).sum())
    # rows, history planes, memory in and out, the newest planes, tokens in and out
    features = plane * (4 * (24 + 2 * HIST) + 4 * HIST + 7 + 7 + 4) + 4 * cells + 2 * 8 * WINDOW * slots
    b = {"step": step, "rollout": step + (K - 1) * outputs, "sample": sample + (9 * plane if case["mask"] else 0),
         "features": step + features, "selfplay": sample + step + features,
         "reset": 4 * cells + 2 * table + outputs, "host": step + outputs}[kind]
    return {"bytes": float(b), "flops": 0.0}


# ---- positions with a history, and their feature tensor in 64 bits -----------
@functools.lru_cache(maxsize=4)
def _grid(games, lo, hi, modes, players):
    """Dense [G][1][Hmax][Wmax] helpers over a ragged batch: cells on the board, players, teams."""
    H, W, mode, P = workloads.shapes(games, (lo, hi), MODES[modes], seed=0, ffa_players=players)
    t = lambda x: torch.as_tensor(x, dtype=torch.int64, device="cuda").view(-1, 1, 1)  # noqa: E731
    H, W, mode, P = t(H), t(W), t(mode), t(P)
    r = torch.arange(int(H.max()), device="cuda").view(1, -1, 1)
    c = torch.arange(int(W.max()), device="cuda").view(1, 1, -1)
    return dict(H=H, W=W, mode=mode, P=P, r=r, c=c, on=(r < H) & (c < W))


def _boards(case, seed):
    """HIST + 3 boards in a row, dense: terrain [G][H][W], then per frame owner
    and army.  Land lies around each player's general and comes and goes at
    its border; the last board is the one that the timed step starts from."""
    d = _grid(case["games"], case["side_lo"], case["side_hi"], case["modes"], case["ffa_players"])
    gen = torch.Generator(device="cuda").manual_seed(seed)
    on, r, c = d["on"], d["r"], d["c"]
    shape, G = on.shape, on.shape[0]
    rand = lambda: torch.rand(shape, generator=gen, device="cuda")  # noqa: E731
    kind = rand()
    terrain = torch.where(kind < 0.2, 1, torch.where(kind < 0.22, 2, 0)).to(torch.int64)
    pmax = int(d["P"].max())
    spots = torch.where(on, rand(), -1.0).view(G, -1).topk(pmax, dim=1).indices  # the generals' cells
    gr, gc = spots // shape[2], spots % shape[2]
    for p in range(pmax):
        here = (r == gr[:, p].view(-1, 1, 1)) & (c == gc[:, p].view(-1, 1, 1)) & (p < d["P"])
        terrain = torch.where(here, 3, terrain)
    base = (1 + (-6 * torch.log1p(-rand())).floor()).to(torch.int64).clamp(max=90)
    frames = []
    for f in range(HIST + 3):
        owner = torch.full(shape, -1, dtype=torch.int64, device="cuda")
        best = torch.full(shape, 1 << 20, dtype=torch.int64, device="cuda")
        for p in range(pmax):
            dist = (r - gr[:, p].view(-1, 1, 1)).abs() + (c - gc[:, p].view(-1, 1, 1)).abs()
            reach = 4 + (f // 3 + p) % 3
            take = (dist <= reach) & (dist < best) & (p < d["P"]) & (terrain != 1)
            best, owner = torch.where(take, dist, best), torch.where(take, p, owner)
        army = torch.where(owner >= 0, base + (rand() < 0.1).to(torch.int64), torch.where(terrain == 2, 40 + base % 11, 0))
        frames.append((torch.where(on, owner, -1), torch.where(on, army, 0)))
    return d, torch.where(on, terrain, 0), frames


def _flat(d, x, fill):
    """A dense board in the library's layout: games one after another, cells row-major, padded to 16."""
    n = (d["H"] * d["W"]).view(-1)
    npad = (n + 15) // 16 * 16
    off = torch.cumsum(npad, 0) - npad
    at = (off.view(-1, 1, 1) + d["r"] * d["W"] + d["c"])[d["on"]]
    y = torch.full((int(npad.sum()),), fill, dtype=x.dtype, device=x.device)
    y[at] = x[d["on"]]
    return y.cpu().numpy()


def _positions(case, seed):
    """The boards as write_state() takes them, with turn and frame counters."""
    d, terrain, frames = _boards(case, seed)
    t = _flat(d, terrain, 0).astype(np.int8)
    scalars = np.zeros((case["games"], 8), np.uint32)
    scalars[:, 3] = (1 << d["P"].view(-1).cpu().numpy()) - 1  # every player alive
    for f, (owner, army) in enumerate(frames):
        scalars[:, 0] = scalars[:, 1] = PREROLL + f
        yield _flat(d, army, 0).astype(np.int16), _flat(d, owner, -1).astype(np.int8), t, scalars


def exact(case, seed):
    """Feature tensor of a "features" case in plain torch, 64 bits.  The other
    outputs are whole numbers (or rewards of -1, 0 and 1), and the other
    cases' positions come from the framework's own games."""
    if case["kind"] != "features":
        return None
    d, terrain, frames = _boards(case, seed)
    H, W, mode, P, on = d["H"], d["W"], d["mode"], d["P"], d["on"]
    # the frame the timed step makes: every player waits, then armies grow
    owner, army = frames[-1]
    turn = PREROLL + len(frames)
    grows = (terrain >= 2) & (turn % 2 == 0) | (terrain == 0) & (turn % 50 == 0)
    frames.append((owner, army + (grows & (owner >= 0) & on).to(torch.int64)))
    C, n = 24 + 2 * HIST, (H * W).view(-1)
    npad = (n + 15) // 16 * 16
    plane = P.view(-1) * npad
    first = torch.cumsum(plane, 0) - plane
    out = torch.zeros(int(plane.sum()) * C, dtype=torch.float64, device="cuda")
    place = d["r"] * W + d["c"]
    team = lambda x: torch.where(mode == 1, x >> 1, x)  # noqa: E731
    per = lambda x: x.view(-1, 1, 1)  # noqa: E731
    for p in range(int(P.max())):
        there = on & (p < P)
        mine = team(torch.tensor(p, device="cuda"))
        seen = torch.zeros_like(on)
        enemy_seen, generals, castles, mountains = (torch.zeros_like(on) for _ in range(4))
        last_army, last_turn = torch.zeros_like(army), torch.zeros_like(army)
        planes = []
        for f, (o, a) in enumerate(frames):
            held = ((o >= 0) & (team(o) == mine)).to(torch.float32).unsqueeze(1)
            vis = (torch.nn.functional.max_pool2d(held, 3, 1, 1).squeeze(1) > 0) & on
            foe = vis & (o >= 0) & (team(o) != mine)
            last_army = torch.where(vis, torch.where(foe, a, 0), torch.where(seen, last_army, 0))
            last_turn = torch.where(foe, PREROLL + f, last_turn)
            seen, enemy_seen = seen | vis, enemy_seen | foe
            generals, castles = generals | vis & (terrain == 3), castles | vis & (terrain == 2)
            mountains = mountains | vis & (terrain == 1)
            planes.append((torch.where(o == p, a, 0), torch.where(foe, a, 0)))
        free, fog = vis & (o == -1), on & ~vis
        age = torch.where(fog & enemy_seen, turn - last_turn, 0).double()
        foes = on & (o >= 0) & (team(o) != mine)
        count = lambda m: per((m & on).sum((1, 2)))  # noqa: E731
        total = lambda m: per(torch.where(m & on, a, 0).sum((1, 2)))  # noqa: E731
        rows = [torch.where(vis, a, 0), planes[-1][0], planes[-1][1], torch.where(free, a, 0), seen, enemy_seen,
                generals, castles, mountains, free & (terrain != 1), o == p, foe, fog,
                fog & ((terrain == 1) | (terrain == 2) | generals), turn, (turn % 50) / 50.0, count(o == p),
                total(o == p), count(foes), total(foes), last_army, torch.log1p(age) / 5.0,
                d["c"] / (W - 1).clamp(min=1).double(), d["r"] / (H - 1).clamp(min=1).double()]
        for side in (0, 1):
            rows += [planes[-1 - k][side] - planes[-2 - k][side] for k in range(HIST)]
        base = per(first + p * npad) * C + place
        for ch, row in enumerate(rows):
            row = row if torch.is_tensor(row) else torch.tensor(float(row), device="cuda")
            out[(base + ch * per(npad))[there]] = row.double().expand(on.shape)[there]
    return [out] + [None] * 10
