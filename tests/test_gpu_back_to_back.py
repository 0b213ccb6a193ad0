"""Steps queued back to back on one stream.  The kernels of a step overlap their launches, so each has to see what the one
before it wrote, and none may overwrite what the one before still reads: every step of a queue whose cameras, boxes,
overlays and worlds change from step to step gives the bytes that it gives when the GPU is waited for after every call."""
import numpy as np
import pytest
import torch

import parity
from paper_2107_08170_b200 import scenes

pytestmark = pytest.mark.gpu

STEPS, WORLDS = 16, 4


@pytest.mark.parametrize("name,envs,occ_in_global", [("tiny", 4, False), ("rooms_boxes", 24, False), ("rooms_boxes", 24, True),
                                                     ("headline", 40, False)])
def test_queued_steps_see_their_own_inputs(oracle, name, envs, occ_in_global):
    from paper_2107_08170_b200 import binding as B
    from gpu_util import scene_to_numpy, upload_scene
    cfg = scenes.config(name, num_envs=envs)
    A, W = cfg.agents, cfg.width
    dev = torch.device("cuda", 0)
    sets = [scenes.make_scene(cfg, k * envs, envs, device=dev) for k in range(WORLDS)]     # four worlds for every env
    has_boxes = cfg.max_boxes > 0
    rects = torch.zeros(STEPS, cfg.num_obs, 1, 4, dtype=torch.int32)                       # a bar that grows with the step
    rects[..., 1] = (torch.arange(1, STEPS + 1) * W // (2 * STEPS))[:, None, None] | (6 << 16)
    rects[..., 2] = 0x40A0F0
    rects, ones = rects.to(dev), torch.ones(cfg.num_obs, dtype=torch.int32, device=dev)
    moves = torch.from_numpy(np.random.default_rng(11).normal(0, 0.2, (STEPS, cfg.num_obs, 4)).astype(np.float32)).to(dev)
    # step k gives env (3 k) mod envs its world k mod 4, all envs the boxes of set k mod 4, and each env cameras of its world
    world = np.zeros((STEPS, envs), int)
    for k in range(1, STEPS):
        world[k] = world[k - 1]
        world[k, 3 * k % envs] = k % WORLDS
    all_cams = torch.stack([s["cams"].view(envs, A, 6) for s in sets])
    cams = [all_cams[torch.from_numpy(world[k]).to(dev), torch.arange(envs, device=dev)].reshape(-1, 6).contiguous() for k in range(STEPS)]

    def run(wait):
        batch = B.Batch(B.desc_from_config(cfg, 0, max_overlay_rects=1))
        if occ_in_global:
            batch.debug_occupancy_in_global(True)
        upload_scene(batch, sets[0])
        frames = [batch.alloc_outputs() for _ in range(STEPS)]
        cams_in = [c.clone() for c in cams]
        torch.cuda.synchronize()
        done = torch.cuda.synchronize if wait else (lambda: None)
        for k in range(STEPS):
            s, own = sets[k % WORLDS], slice(3 * k % envs, 3 * k % envs + 1)
            if k > 0:
                batch.upload_worlds(own.start, 1, s["grid"][own], None, None, s["palette"][own])
                done()
            if has_boxes:
                batch.upload_worlds(0, envs, None, s["boxes"], s["box_count"], None)
                done()
            if k % 4 == 3:
                batch.move_agents(cams_in[k], moves[k])                                    # (from step k's cameras)
            else:
                batch.set_cameras(cams_in[k])
            done()
            batch.set_overlays(rects[k], ones)
            done()
            batch.render_batch(*frames[k])
            done()
        torch.cuda.synchronize()
        assert batch.query_status() == 0
        batch.destroy()
        return frames

    want, got = run(True), run(False)
    for k in range(STEPS):
        assert torch.equal(want[k][0], got[k][0]) and torch.equal(want[k][1], got[k][1]), k
    assert all(not torch.equal(want[k][0], want[k + 1][0]) for k in range(STEPS - 1))      # the steps do differ
    # and the waited-for run is the right one: the env that has just changed its world, in a step without motion
    k = STEPS - 2
    e, bx = 3 * k % envs, scene_to_numpy(sets[k % WORLDS])
    grid, palette = bx["grid"][e], bx["palette"][e]
    boxes, count = (bx["boxes"][e], int(bx["box_count"][e])) if has_boxes else (None, 0)
    rgb, depth, rows = want[k][0].cpu().numpy(), want[k][1].cpu().numpy(), cams[k].cpu().numpy()
    od = oracle.desc_from_config(cfg)
    for o in range(e * A, e * A + A):
        o_rgb, o_depth, o_ids = oracle.render_obs(od, grid, boxes, count, palette, rows[o])
        o_rgb = oracle.overlay(np.ascontiguousarray(o_rgb), rects[k, o].cpu().numpy().reshape(-1).view(oracle.RECT_DTYPE), 1)
        st = parity.compare_obs(oracle, od, grid, boxes, count, palette, rows[o], rgb[o], depth[o], o_rgb, o_depth, o_ids)
        parity.assert_parity(st, (name, o))
