"""What a user of this library has it do, as timed cases: the per-step calls of a simulator loop at the
benchmark's workload shapes, agent motion with the GUI overlay, episode resets, the voxel merge, the
host-memory step and the vectorised step() wrapper.

A case is a dict: `call` says which entry points a pass goes through, the rest is the shape.

  step    (boxes moved: mv_upload_worlds with the box list only,) mv_set_cameras, mv_render_batch
  agents  mv_move_agents, mv_set_overlays, mv_render_batch
  reset   mv_upload_worlds with every array, mv_set_cameras, mv_render_batch
  merge   mv_merge_voxels over all environments
  host    mv_step_host: cameras and boxes in from pinned host memory, frames out to it
  vecenv  VecRenderEnv.step: motion, auto-reset of the environments whose episode ends, time-left bar, render
"""
from __future__ import annotations

import math

import torch

from paper_2107_08170_b200 import binding, scenes, vecenv, workload

KEYS = ("call", "envs", "agents", "gx", "gy", "gz", "width", "height", "palette", "world", "boxes", "bodies")
EPISODE = 100           # steps per episode of the vectorised wrapper's cases
MERGE_MAX_OUT = 2048    # room for the merged boxes of one environment


def _case(name, *values):
    return {**({"name": name} if name else {}), **dict(zip(KEYS, values))}


def listed():
    return [
        # four small worlds, 64x36: a debugging session or a unit test; launches and latency count
        _case("tiny", "step", 4, 1, 16, 8, 16, 64, 36, 16, "segments", 0, False),
        # room worlds without boxes, two agents each: a mid-size trainer, a few waves of the GPU
        _case("rooms", "step", 1024, 2, 64, 16, 64, 128, 72, 64, "rooms", 0, False),
        # the full scene: movable boxes and agent bodies, re-sent every step, four agents per world
        _case("rooms_boxes", "step", 4096, 4, 64, 16, 64, 128, 72, 64, "rooms", 32, True),
        # the benchmark's headline: 16384 environments on 128x32x128 grids
        _case("headline", "step", 16384, 1, 128, 32, 128, 128, 72, 64, "columns", 16, False),
        # the resolution sweep's two ends: many small images, and large ones (the largest case)
        _case("sweep_64x36", "step", 8192, 2, 64, 16, 64, 64, 36, 64, "rooms", 32, False),
        _case("sweep_256x144", "step", 8192, 2, 64, 16, 64, 256, 144, 64, "rooms", 32, False),
        # motion, collision and the time-left bar at sizes that are multiples of nothing much
        _case("ragged_agents", "agents", 777, 3, 52, 20, 44, 104, 60, 23, "rooms", 13, True),
        # a grid too large for shared memory and more than 32 high
        _case("big_grid", "step", 512, 1, 192, 48, 192, 128, 72, 64, "columns", 16, False),
        # new episodes: 512 worlds packed and their first frames rendered
        _case("reset", "reset", 512, 1, 128, 32, 128, 128, 72, 64, "columns", 16, False),
        # the paper's greedy merge of voxels into boxes, at the start of an episode
        _case("merge", "merge", 512, 1, 128, 32, 128, 128, 72, 64, "columns", 16, False),
        # the paper's default hand-off: frames copied to host memory
        _case("host", "host", 512, 2, 64, 16, 64, 128, 72, 64, "rooms", 32, True),
        # the vectorised wrapper at the headline size: about one environment in a hundred resets per step
        _case("vecenv", "vecenv", 16384, 1, 128, 32, 128, 128, 72, 64, "columns", 16, False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step"] * 5 + ["agents", "reset", "merge", "host", "vecenv"])
    world = rng.choice(["rooms", "columns"])
    # grids: 16 to 192 cells wide, 16 to 64 high (multiples of 4); one-word columns are the usual ones
    gx, gz = 4 * _log_int(rng, 4, 48), 4 * _log_int(rng, 4, 48)
    gy = 4 * (_log_int(rng, 4, 8) if rng.random() < 0.75 else _log_int(rng, 9, 16))
    width = 8 * _log_int(rng, 6, 32)
    height = 4 * max(4, round(width * rng.uniform(0.5, 0.75) / 4))
    agents = rng.choice([1, 1, 2, 3, 4, 6])
    bodies = rng.random() < 0.5
    boxes = rng.choice([0, rng.randint(1, 15), rng.randint(16, 48)])
    envs = _log_int(rng, 1, 16384)
    # no more pixels, voxels, merged voxels or host bytes than the listed cases have
    envs = min(envs, 8192 * 2 * 256 * 144 // (agents * width * height), 16384 * 128 * 32 * 128 // (gx * gz * max(gy, 32)))
    if call in ("reset", "merge"):
        envs = min(envs, 512 * 128 * 32 * 128 // (gx * gy * gz))
    if call == "host":
        envs = min(envs, 512 * 2 * 128 * 72 // (agents * width * height))
    if call == "vecenv":
        envs = min(envs, 16384 // agents)
    return _case(None, call, max(envs, 1), agents, gx, gy, gz, width, height, rng.randint(2, 256), world, boxes, bodies)


def _config(case, seed):
    """The scene recipe of the repository's workloads with the obstacle density kept as the grid grows."""
    gx, gz = case["gx"], case["gz"]
    extra = {}
    if case["world"] == "columns":
        extra = {"n_rects": max(4, round(1050 * gx * gz / (128 * 128)))}
    elif case["world"] == "rooms":
        extra = {"n_lines": max(1, (min(gx, gz) - 1) // 9 - 1), "n_pillars": max(1, round(24 * gx * gz / (64 * 64)))}
    return scenes.SceneConfig(name=case["call"], num_envs=case["envs"], agents=case["agents"],
                              grid=(gx, case["gy"], gz), width=case["width"], height=case["height"],
                              palette_size=case["palette"], world=case["world"], movable_boxes=case["boxes"],
                              body_boxes=case["bodies"], cam_y_fixed=1.5 if case["world"] == "segments" else None,
                              seed=seed, extra=extra)


def _moves(cfg, seed, dev):
    """One step's motion commands: mostly forward, some strafing and turning.  A pass plays them and the next
    pass plays them backwards, so that the agents stay where episodes begin however many passes are made."""
    g = torch.Generator(device=dev).manual_seed(seed)
    u = torch.rand(cfg.num_obs, 4, generator=g, device=dev)
    m = (u - 0.5) * torch.tensor([0.4, 0.2, 0.3, 0.1], device=dev)
    return [m.contiguous(), (-m).contiguous()]


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    cfg = _config(case, seed)
    call = case["call"]
    s = {"call": call, "cfg": cfg, "pass": 0}
    if call in ("agents", "vecenv"):
        s["moves"] = _moves(cfg, seed, dev)
    if call == "vecenv":
        s["env"] = vecenv.VecRenderEnv(cfg, EPISODE, device=0, phase=torch.arange(cfg.num_envs) % EPISODE)
        s["env"].reset()
        return s
    s["batch"], s["cams"], _ = workload.build_batch(cfg, 0, max_overlay_rects=1 if call == "agents" else 0)
    if call == "merge":
        return s
    s["boxes"] = s["count"] = None
    if cfg.max_boxes > 0 and call in ("step", "reset", "host"):
        # the simulator's box list of this step
        s["boxes"] = torch.empty(cfg.num_envs, cfg.max_boxes, 8, dtype=torch.int32, device=dev)
        s["count"] = torch.empty(cfg.num_envs, dtype=torch.int32, device=dev)
        for e in range(0, cfg.num_envs, 512):
            n = min(512, cfg.num_envs - e)
            sc = scenes.make_scene(cfg, e, n, device=dev)
            s["boxes"][e:e + n], s["count"][e:e + n] = sc["boxes"], sc["box_count"]
    if call == "reset":
        worlds = scenes.make_worlds(cfg, device=dev)
        s["grid"], s["palette"] = worlds["grid"].contiguous(), worlds["palette"].contiguous()
    if call == "agents":
        left = torch.arange(cfg.num_envs) % EPISODE
        s["rects"] = vecenv.time_bar_rects(left, torch.full_like(left, EPISODE), cfg.width, cfg.agents).to(dev)
        s["rect_count"] = torch.ones(cfg.num_obs, dtype=torch.int32, device=dev)
    if call == "host":
        shape = (cfg.num_obs, cfg.height, cfg.width)
        s["rgb"] = torch.empty(*shape, 3, dtype=torch.uint8, pin_memory=True)
        s["depth"] = torch.empty(*shape, dtype=torch.float32, pin_memory=True)
        s["cams"] = s["cams"].cpu().pin_memory()
        if s["boxes"] is not None:
            s["boxes"], s["count"] = s["boxes"].cpu().pin_memory(), s["count"].cpu().pin_memory()
    else:
        s["rgb"], s["depth"] = s["batch"].alloc_outputs()
    return s


def run(s):
    call, cfg = s["call"], s["cfg"]
    if call in ("agents", "vecenv"):
        moves = s["moves"][s["pass"] & 1]
        s["pass"] += 1
    if call == "vecenv":
        rgb, depth, done = s["env"].step(moves)
        return {"rgb": rgb, "depth": depth, "done": done, "cams": s["env"].cams}
    batch = s["batch"]
    if call == "merge":
        boxes, counts = batch.merge_voxels(0, cfg.num_envs, MERGE_MAX_OUT)
        return {"boxes": boxes, "counts": counts}
    if call == "host":
        batch.step_host(s["cams"], s["rgb"], s["depth"], boxes=s["boxes"], box_count=s["count"])
        return {"rgb": s["rgb"], "depth": s["depth"]}
    if call == "agents":
        batch.move_agents(s["cams"], moves)
        batch.set_overlays(s["rects"], s["rect_count"])
        batch.render_batch(s["rgb"], s["depth"])
        return {"rgb": s["rgb"], "depth": s["depth"], "cams": s["cams"]}
    if call == "reset":
        batch.upload_worlds(0, cfg.num_envs, s["grid"], s["boxes"], s["count"], s["palette"])
    elif s["boxes"] is not None:
        batch.upload_worlds(0, cfg.num_envs, boxes=s["boxes"], box_count=s["count"])
    batch.set_cameras(s["cams"])
    batch.render_batch(s["rgb"], s["depth"])
    return {"rgb": s["rgb"], "depth": s["depth"]}


def work(case):
    cfg = _config(case, 0)
    call, E, O = case["call"], cfg.num_envs, cfg.num_obs
    gx, gy, gz = cfg.grid
    nvox, px = gx * gy * gz, cfg.width * cfg.height
    if call == "merge":
        # occupancy bits and the materials of the filled voxels in (about one in seven), merged boxes out
        return {"bytes": E * (nvox // 8 + nvox // 7 + MERGE_MAX_OUT * 32 + 4), "flops": 0}
    # cameras and boxes in, occupancy bits, one material byte and seven frame bytes per pixel
    n = workload.algorithmic_bytes(cfg) + 24 * O
    if call == "reset":
        n += E * (nvox + 3 * cfg.palette_size + 32 * cfg.max_boxes)
    if call == "agents":
        n += O * (16 + 24 + 16)
    if call == "vecenv":
        n += O * (16 + 24 + 16) + E * nvox // EPISODE
    # per ray: 12 for the direction, 3 reciprocals, 3 first crossings, 4 per cell and about 6 cells
    return {"bytes": n, "flops": 42 * O * px}


def tolerance(case):
    if case["call"] == "merge":
        return "exact"
    # depth is a sum of float crossing times; colours are table bytes that differ only where a ray passes
    # within rounding of an edge
    return {"rel": 1e-5, "differ": 1e-5}
