"""Occupancy that is read from global memory and asked for in L2: for which batches, with what frames, and what it may not cost."""
from __future__ import annotations

import pytest
import torch

pytestmark = pytest.mark.gpu


def _batch(grid, world, envs, agents, size, palette=64):
    """A batch of seeded scenes with its cameras set, read from global memory."""
    from paper_2107_08170_b200 import binding as B, scenes
    extra = {"n_rects": 1050 * grid[0] * grid[2] // 128 ** 2} if world == "columns" else {"n_lines": max(1, min(grid[0], grid[2]) // 9 - 2), "n_pillars": 24}
    cfg = scenes.config("rooms", num_envs=envs, agents=agents, grid=grid, width=size[0], height=size[1], palette_size=palette, movable_boxes=4,
                        world=world, extra=extra)
    batch = B.Batch(B.desc_from_config(cfg, 0))
    cams = torch.zeros(cfg.num_obs, 6, dtype=torch.int32, device="cuda")
    desc = scenes.native_desc(cfg)
    for e in range(0, envs, 512):
        at = torch.arange(e, min(e + 512, envs))
        scenes.native_upload(cfg, desc, at.cuda(), batch, at, cams)
    batch.set_cameras(cams)
    return batch, cams


@pytest.mark.parametrize("grid,envs,agents,size,asked", [
    ((192, 48, 192), 1, 1, (64, 36), True), ((192, 48, 192), 320, 1, (128, 72), True), ((192, 48, 192), 330, 1, (64, 36), False),
    ((192, 48, 192), 300, 1, (256, 144), False), ((192, 48, 192), 512, 1, (128, 72), False), ((192, 48, 192), 1024, 1, (128, 72), False),
    ((192, 48, 192), 2048, 1, (128, 72), True), ((192, 48, 192), 512, 4, (128, 72), True), ((192, 48, 192), 2048, 1, (64, 36), False),
    ((192, 48, 192), 512, 1, (256, 144), False), ((256, 64, 256), 2048, 1, (128, 72), False), ((64, 16, 64), 2048, 1, (128, 72), False)])
def test_which_batches_ask(grid, envs, agents, size, asked):
    """Batches that L2 holds beside their frames, and those whose frames push everything out; staged ones never."""
    from paper_2107_08170_b200 import binding as B
    batch = B.Batch(B.make_desc(envs, agents, grid, 4, *size, 64))
    assert batch.debug_prefetch(None) == asked == batch.debug_prefetch(None, ask=True)
    assert not batch.debug_prefetch(False)
    batch.destroy()


@pytest.mark.parametrize("grid,world,envs,agents", [((192, 48, 192), "columns", 5, 1), ((256, 64, 256), "rooms", 3, 3), ((16, 132, 20), "rooms", 4, 2),
                                                   ((4, 4, 4), "columns", 2, 1), ((192, 32, 192), "columns", 460, 1)])
def test_frames_are_the_same(grid, world, envs, agents):
    """Also with eyes below, above and beside the grid and a camera that is not a number: the plane asked for lies in the block."""
    batch, cams = _batch(grid, world, envs, agents, (64, 36))
    batch.debug_occupancy_in_global(True)
    f = cams.view(torch.float32)
    f[0, 1], f[-1, 1], f[envs // 2 * agents, 1] = -3.0, grid[1] + 5.0, float("nan")
    batch.set_cameras(cams)
    frames = []
    for on in (False, True):
        assert batch.debug_prefetch(on) == on
        rgb, depth = batch.alloc_outputs()
        batch.render_batch(rgb, depth)
        frames.append((rgb, depth))
    assert all(torch.equal(a, b) for a, b in zip(*frames))
    batch.destroy()


@pytest.mark.parametrize("grid,world,envs,agents,size", [
    ((192, 48, 192), "rooms", 2048, 1, (64, 36)), ((192, 48, 192), "columns", 640, 1, (128, 72)), ((192, 48, 192), "columns", 300, 1, (256, 144)),
    ((192, 48, 192), "rooms", 400, 1, (128, 72)), ((128, 48, 128), "rooms", 1024, 1, (128, 72)), ((192, 48, 192), "columns", 128, 4, (128, 72))])
def test_steps_with_nothing_in_between_lose_nothing(grid, world, envs, agents, size):
    """Cameras and frames again and again: what the library does is no slower than not asking (5 % is the spread of such a loop)."""
    batch, cams = _batch(grid, world, envs, agents, size)
    rgb, depth = batch.alloc_outputs()
    best = {False: float("inf"), None: float("inf")}
    for _ in range(6):
        for on in best:
            batch.debug_prefetch(on)
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            for i in range(12):
                if i == 4:
                    start.record()
                batch.set_cameras(cams)
                batch.render_batch(rgb, depth)
            end.record()
            torch.cuda.synchronize()
            best[on] = min(best[on], start.elapsed_time(end))
    assert best[None] <= 1.05 * best[False], best
    batch.destroy()
