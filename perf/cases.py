"""The calls whose speed counts, as a program that uses this library makes them.

One pass of a case is one call (or one round of calls) through the public
binding: a step, a rollout, a reset, a render, a step with host buffers, a
batched step or rollout over groups of different sizes, the replay of a
captured step graph, or one round of requests to the step server. The sizes
are those of the workload presets in ``inputs.py``, the tests and the
benchmark; ``draw`` spreads further cases over the same ranges.
"""

from __future__ import annotations

import numpy as np
import torch

from paper_2605_19926_gb300 import inputs, jx

ACTION_ROWS = 64  # a step case walks through this many rows of actions, then starts over


def listed() -> list[dict]:
    return [
        # the single-environment program: 16 x 16 rooms, one step call after the other
        dict(name="rooms_step_1", kind="step", task="rooms", envs=1, side=16, h=64, w=64, sprites=0, horizon=0),
        # a small actor group on a hand-drawn map with coloured keys and doors and shaded walls, a ragged env
        # count and a frame that is not square
        dict(name="ascii_step_250", kind="step", task="ascii", envs=250, side=24, h=48, w=80, sprites=4, horizon=200,
             shading=1),
        # the acting loop of the benchmark workload: the next actions depend on the frames
        dict(name="maze_step_4096", kind="step", task="maze", envs=4096, side=32, h=64, w=64, sprites=2, horizon=500),
        # action streams known in advance: a short launch, and the benchmark's long one
        dict(name="maze_rollout_4096x20", kind="rollout", task="maze", envs=4096, side=32, h=64, w=64, sprites=2,
             horizon=500, steps=20),
        dict(name="maze_rollout_4096x128", kind="rollout", task="maze", envs=4096, side=32, h=64, w=64, sprites=2,
             horizon=500, steps=128),
        # the start of a run: 4096 mazes generated and drawn
        dict(name="maze_reset_4096", kind="reset", task="maze", envs=4096, side=32, h=64, w=64, sprites=2, horizon=500),
        # frame-stacking agents: RGB and the 4-frame grayscale stack, 64 x 64 mazes with rooms and distractors
        dict(name="gray_step_1024", kind="step", task="maze_rooms", envs=1024, side=64, h=96, w=96, sprites=8,
             horizon=500, gray=1),
        # the large-scale workload's launches, at a quarter of its envs
        dict(name="large_rollout_16384x8", kind="rollout", task="maze_rooms", envs=16384, side=128, h=128, w=128,
             sprites=16, horizon=500, gray=1, steps=8),
        # uneven batching (16 groups of sides 16..128 and frames 32..128) with tiles an autotuner run chose:
        # rollouts, and the captured step pipeline
        dict(name="uneven_rollout_16384x16", kind="batch_rollout", envs=16384, steps=16, sprites=8, tuned=1),
        dict(name="uneven_graph_16384x8", kind="batch_graph", envs=16384, steps=8, sprites=8, tuned=1),
        # the step server: a round of requests of eight actor groups (16..4096 envs, 32 and 64 sided mazes)
        dict(name="serve_8", kind="serve", sessions=8),
        # an agent on the host: host actions in, frames back in pinned host memory
        dict(name="host_step_4096", kind="host", task="maze", envs=4096, side=32, h=64, w=64, sprites=2, horizon=500),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng) -> dict:
    kind = rng.choice(["step", "step", "step", "rollout", "rollout", "rollout", "reset", "render", "host",
                       "batch_step", "batch_rollout", "batch_graph", "serve"])
    if kind == "serve":
        return dict(kind=kind, sessions=rng.randint(1, 12))
    if kind.startswith("batch"):
        c = dict(kind=kind, envs=_log_int(rng, 200, 16384), sprites=rng.choice([0, 3, 8]), tuned=rng.randint(0, 1))
        if kind != "batch_step":
            c["steps"] = rng.randint(2, 12)
        return c
    task = rng.choice(["rooms", "rooms", "maze", "maze", "maze", "maze_rooms", "ascii"])
    side = {"rooms": lambda: rng.choice([9, 16, 24, 32, 45, 64, 100, 128]),
            "maze": lambda: rng.choice([8, 16, 18, 32, 32, 40, 64, 128]),
            "maze_rooms": lambda: rng.choice([32, 64, 128]),
            "ascii": lambda: rng.choice([20, 24, 32])}[task]()
    if kind == "reset":
        side = min(side, 64)
    h, w = rng.choice([(32, 32), (40, 48), (48, 80), (64, 64), (64, 64), (64, 64), (96, 96), (96, 128), (128, 128)])
    sprites = {"rooms": lambda: rng.choice([0, 4, 8]), "maze": lambda: 2, "maze_rooms": lambda: rng.choice([4, 16]),
               "ascii": lambda: 4}[task]()
    c = dict(kind=kind, task=task, side=side, h=h, w=w, sprites=sprites, horizon=rng.choice([200, 500]),
             shading=int(rng.random() < 0.2), gray=int(rng.random() < 0.2))
    c["envs"] = _log_int(rng, 1, 8192)
    if kind == "rollout":
        c["steps"] = _log_int(rng, 2, 128)
    # never more frame bytes than the largest listed case
    while c["envs"] * c.get("steps", 1) * h * w * 3 > 4 << 30:
        c["envs"] = c["envs"] // 2 + 1
    return c


def _config(case: dict, seed: int) -> dict:
    common = dict(n_envs=case["envs"], map_side=case["side"], frame_h=case["h"], frame_w=case["w"], seed=seed)
    if case["task"] == "rooms":
        cfg = dict(inputs.rooms(wall_prob=0.25, max_sprites=case["sprites"], **common), horizon=case["horizon"])
    elif case["task"] == "maze":
        cfg = inputs.maze_keydoor(horizon=case["horizon"], **common)
    elif case["task"] == "maze_rooms":
        cfg = inputs.maze_rooms(horizon=case["horizon"], max_sprites=case["sprites"], gray_stack=0, **common)
    else:
        cfg = inputs.ascii_env("coloured-rooms", horizon=case["horizon"], max_sprites=case["sprites"], **common)
    return dict(cfg, gray_stack=case.get("gray", 0), shading=case.get("shading", 0))


def _tiling(case: dict):
    """Tiles as an autotuner run over the uneven workload picks them, or the default ones."""
    if not case.get("tuned"):
        return None
    t = jx.Tiling()
    t.warps_per_block, t.cols_per_lane, t.bits_min_side, t.max_rows_per_block, t.staging_buffers = 2, 1, 8, 32, 1
    return t


def _groups(case: dict, seed: int) -> list[dict]:
    """The groups of the uneven workload (its sizes), with maps of their own."""
    groups = inputs.uneven_groups(n_envs=case["envs"], seed=2, max_sprites=case["sprites"])
    return [dict(g, seed=seed * 101 + k) for k, g in enumerate(groups)]


def _sessions(case: dict, seed: int) -> list[dict]:
    """The first session of each actor group of the serving workload (its sizes), with mazes of its own."""
    return [dict(inputs.serving_session(3, actor, 0), seed=seed * 101 + actor) for actor in range(case["sessions"])]


def _actions(seed: int, rows: int, n: int) -> torch.Tensor:
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(0, inputs.N_ACTIONS, (rows, n), generator=g, device="cuda", dtype=torch.uint8)


def _outputs(rows: int, n: int, frame_shape: tuple) -> dict:
    return dict(frames=torch.empty((rows,) + frame_shape, dtype=torch.uint8, device="cuda"),
                rewards=torch.empty((rows, n), dtype=torch.float32, device="cuda"),
                dones=torch.empty((rows, n), dtype=torch.uint8, device="cuda"))


def prepare(case: dict, seed: int) -> dict:
    """The environments, started, with the actions and output buffers of the coming calls."""
    kind = case["kind"]
    st = dict(kind=kind, at=0)
    if kind == "serve":
        server = jx.Server(budget_bytes=8 << 30, max_sessions=16, max_inflight=4, max_map_side=64)
        sessions = [server.open(cfg) for cfg in _sessions(case, seed)]
        rng = np.random.default_rng(seed)
        acts = [[rng.integers(0, inputs.N_ACTIONS, s.n, dtype=np.uint8) for s in sessions] for _ in range(ACTION_ROWS)]
        outs = [dict(frames=s.frames, rewards=s.rewards, dones=s.dones) for s in sessions]
        for o in outs:
            for t in o.values():
                t.server = server  # the tensors alias the server's arena: it lives as long as they do
        return dict(st, server=server, sessions=sessions, acts=acts, out=outs)
    if kind.startswith("batch"):
        groups = [jx.Env(g) for g in _groups(case, seed)]
        batch = jx.Batch(groups, _tiling(case))
        rows = case.get("steps", 1)
        out = _outputs(rows, batch.n, (batch.frame_bytes,))
        batch.reset(out["frames"][0])
        st.update(groups=groups, batch=batch, out=out)
        if kind == "batch_step":
            st["acts"] = list(_actions(seed, ACTION_ROWS, batch.n).unbind(0))
            st["out"] = {k: v[0] for k, v in out.items()}
        else:
            st["acts"] = _actions(seed, rows, batch.n)
            if kind == "batch_graph":
                torch.cuda.synchronize()
                st["graph"] = batch.capture(st["acts"], out["frames"], out["rewards"], out["dones"])
        return st
    env = jx.Env(_config(case, seed))
    n, shape = case["envs"], (case["envs"], case["h"], case["w"], 3)
    if kind == "rollout":
        out = _outputs(case["steps"], n, shape)
        env.reset(out["frames"][0])
        return dict(st, env=env, acts=_actions(seed, case["steps"], n), out=out)
    out = {k: v[0] for k, v in _outputs(1, n, shape).items()}
    env.reset(out["frames"])
    st.update(env=env, out=out)
    if kind in ("reset", "render"):
        st["out"] = dict(frames=out["frames"])
    else:
        acts = _actions(seed, ACTION_ROWS, n)
        if kind == "host":
            acts = acts.cpu().pin_memory()
            st["out"] = {k: torch.empty(v.shape, dtype=v.dtype, pin_memory=True) for k, v in out.items()}
        st["acts"] = list(acts.unbind(0))
    return st


def run(st: dict):
    kind, out = st["kind"], st["out"]
    if kind == "rollout":
        st["env"].rollout(st["acts"], out["frames"], out["rewards"], out["dones"])
    elif kind == "batch_rollout":
        st["batch"].rollout(st["acts"], out["frames"], out["rewards"], out["dones"])
    elif kind == "batch_graph":
        st["graph"].launch()
    elif kind == "reset":
        st["env"].reset(out["frames"])
    elif kind == "render":
        st["env"].render(out["frames"])
    else:
        acts = st["acts"][st["at"]]
        st["at"] = (st["at"] + 1) % ACTION_ROWS
        if kind == "step":
            st["env"].step(acts, out["frames"], out["rewards"], out["dones"])
        elif kind == "host":
            st["env"].step_host(acts, out["frames"], out["rewards"], out["dones"])
        elif kind == "batch_step":
            st["batch"].step(acts, out["frames"], out["rewards"], out["dones"])
        else:
            tickets = [s.submit(a) for s, a in zip(st["sessions"], acts)]
            for t in tickets:
                st["server"].wait(t)
    return out


def _env_bytes(n: int, side: int, h: int, w: int, sprites: int, steps: int, gray: int) -> float:
    """One launch over n envs: per step the frame, the action, reward and done flag; per launch the state
    fields read and the pose written, the grayscale planes it leaves (of the last four frames at most), and
    the map at the one bit a cell that movement and rays need."""
    per_step = 3 * h * w + 6
    per_launch = 53 + 9 * sprites + 19 + side * side / 8 + (min(steps, 4) * h * w if gray else 0)
    return float(n) * (steps * per_step + per_launch)


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "serve":
        total = sum(_env_bytes(c["n_envs"], c["map_side"], c["frame_h"], c["frame_w"], 2, 1, 0)
                    for c in _sessions(case, 0))
    elif kind.startswith("batch"):
        steps = case.get("steps", 1)
        reads = steps if kind == "batch_graph" else 1  # every captured step is a launch
        groups = _groups(case, 0)
        total = sum(_env_bytes(g["n_envs"], g["map_side"], g["frame_h"], g["frame_w"], case["sprites"],
                               steps // reads, 0) for g in groups) * reads
    else:
        n, side = case["envs"], case["side"]
        total = _env_bytes(n, side, case["h"], case["w"], case["sprites"], case.get("steps", 1), case.get("gray", 0))
        if kind == "reset":  # writes the map and the state instead of reading them, and all four planes
            total += n * (side * side * 7 / 8 + (3 * case["h"] * case["w"] if case.get("gray") else 0))
    return {"bytes": float(total), "flops": 0.0}


def exact(case: dict, seed: int):
    """The rooms task gives no reward. Every other output is whole numbers (frames, done flags) or follows
    from the walk through them (the rewards of keys and goals)."""
    if case["kind"] in ("reset", "render", "serve") or case.get("task", "rooms") != "rooms":
        return None
    n, steps = case["envs"], case.get("steps")
    return dict(frames=None, rewards=np.zeros(n if steps is None else (steps, n), np.float64), dones=None)
