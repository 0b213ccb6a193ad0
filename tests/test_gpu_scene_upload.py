"""Seeded scenes made straight in a batch: what an upload of their grids, boxes and palettes leaves, over environments that held something else."""
from __future__ import annotations

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,world,extra,palette,agents,boxes", [
    ((128, 32, 128), "columns", {}, 64, 1, 16), ((16, 64, 24), "rooms", {"n_lines": 1}, 7, 2, 3), ((20, 4, 12), "segments", {}, 2, 1, 0),
    ((8, 100, 1024), "columns", {}, 256, 3, 1), ((64, 36, 4), "rooms", {"n_lines": 0}, 1, 1, 4), ((4, 8, 4), "columns", {"n_rects": 0}, 3, 1, 0),
    ((36, 32, 44), "rooms", {"n_lines": 3}, 17, 4, 0)])
def test_scenes_made_in_the_batch(grid, world, extra, palette, agents, boxes):
    from paper_2107_08170_b200 import binding as B, scenes
    cfg = scenes.config("rooms", num_envs=9, agents=agents, grid=grid, width=40, height=24, palette_size=palette, movable_boxes=boxes,
                        body_boxes=agents > 1, world=world, extra=extra)
    desc = scenes.native_desc(cfg)
    ids = torch.tensor([5, 70001, 3, 12], device="cuda")
    at = [0, 3, 4, 8]
    slots = torch.tensor(at, dtype=torch.int32, device="cuda")
    results = []
    for direct in (False, True):
        batch = B.Batch(B.desc_from_config(cfg, 0))
        old = torch.full((9, grid[1], grid[2], grid[0]), min(1, palette - 1), dtype=torch.uint8, device="cuda")
        batch.upload_worlds(0, 9, old, palette=torch.full((9, palette, 3), 77, dtype=torch.uint8, device="cuda"))       # everything filled, for one thing
        cams = torch.zeros(9 * agents, 6, dtype=torch.int32, device="cuda")
        for _ in range(2):                                                       # (the second time over scenes made the same way)
            if direct:
                scenes.native_upload(cfg, desc, ids, batch, at, cams)
            else:
                w = scenes.make_worlds(cfg, device="cuda", env_ids=ids)
                e = scenes.native_entities(cfg, desc, ids, w["height"], cams, slots)
                batch.upload_worlds_at(at, w["grid"], e["boxes"] if cfg.max_boxes else None, e["box_count"] if cfg.max_boxes else None, w["palette"])
        batch.set_cameras(cams)
        rgb, depth = batch.alloc_outputs()
        batch.render_batch(rgb, depth)
        merged, count = batch.merge_voxels(0, 9, 4096)
        results.append((rgb, depth, merged, count, cams, torch.tensor(batch.query_status())))
        batch.destroy()
    for a, b in zip(*results):
        assert torch.equal(a, b)


def test_scenes_that_do_not_fit_the_batch_are_refused():
    from paper_2107_08170_b200 import binding as B, scenes
    make = lambda **over: scenes.config("rooms", **{**dict(num_envs=3, agents=1, grid=(16, 8, 16), movable_boxes=2, extra={"n_lines": 1}), **over})
    cfg = make()
    batch = B.Batch(B.desc_from_config(cfg, 0))
    ids = torch.tensor([1, 2], device="cuda")
    cams = torch.zeros(8, 6, dtype=torch.int32, device="cuda")
    for c, at in [(cfg, [1, 1]), (cfg, [2, 3]), (cfg, [-1, 0]), (make(grid=(16, 8, 20)), [0, 1]), (make(palette_size=9), [0, 1]),
                  (make(movable_boxes=3), [0, 1]), (make(agents=2), [0, 1])]:
        with pytest.raises(B.MvError) as refused:
            scenes.native_upload(c, scenes.native_desc(c), ids, batch, at, cams)
        assert refused.value.code == -1
    with pytest.raises(ValueError):
        scenes.native_upload(cfg, scenes.native_desc(cfg), ids, batch, [0], cams)
    batch.destroy()


def _both_ways(cfg, at):
    """The scenes 3, 10, 17 ... in the environments `at`: (direct, by their arrays) as functions of a batch and its cameras."""
    from paper_2107_08170_b200 import scenes
    desc = scenes.native_desc(cfg)
    ids = 3 + 7 * torch.arange(len(at), device="cuda")
    slots = torch.tensor(at, dtype=torch.int32, device="cuda")

    def by_arrays(batch, cams):
        w = scenes.make_worlds(cfg, device="cuda", env_ids=ids)
        e = scenes.native_entities(cfg, desc, ids, w["height"], cams, slots)
        batch.upload_worlds_at(at, w["grid"], e["boxes"], e["box_count"], w["palette"])

    return lambda batch, cams: scenes.native_upload(cfg, desc, ids, batch, at, cams), by_arrays


@pytest.mark.parametrize("grid,n", [((16, 1024, 16), 12), ((16, 1024, 16), 48), ((16, 1024, 16), 100), ((64, 1024, 64), 1), ((64, 256, 64), 21), ((20, 64, 12), 150)])
def test_high_worlds_in_slabs(grid, n):
    """Worlds stored by several CTAs above one another, as many as there are 32 heights and fewer (every slabs-th 32 heights and plane)."""
    from paper_2107_08170_b200 import binding as B, scenes
    cfg = scenes.config("rooms", num_envs=n, agents=1, grid=grid, width=40, height=24, palette_size=9, movable_boxes=2, world="segments", extra={"n_rects": 40})
    results = []
    for make in _both_ways(cfg, list(range(n))):
        batch = B.Batch(B.desc_from_config(cfg, 0))
        cams = torch.zeros(n, 6, dtype=torch.int32, device="cuda")
        make(batch, cams)
        batch.set_cameras(cams)
        rgb, depth = batch.alloc_outputs()
        batch.render_batch(rgb, depth)
        results.append((rgb, depth, cams, *batch.merge_voxels(0, n, 512)))
        batch.destroy()
    for a, b in zip(*results):
        assert torch.equal(a, b)


@pytest.mark.parametrize("grid,n", [((64, 1024, 64), 1), ((64, 1024, 64), 8), ((128, 32, 128), 1)])
def test_straight_into_the_batch_is_not_the_longer_way(grid, n):
    """One to a few worlds, also high ones, whose store is many bytes for few columns: no longer than their arrays made and uploaded."""
    from paper_2107_08170_b200 import binding as B, scenes
    cfg = scenes.config("rooms", num_envs=n, agents=1, grid=grid, width=40, height=24, movable_boxes=4, world="columns", extra={"n_rects": 200})
    batch = B.Batch(B.desc_from_config(cfg, 0))
    cams = torch.zeros(n, 6, dtype=torch.int32, device="cuda")
    best = [float("inf")] * 2
    for _ in range(6):
        for i, make in enumerate(_both_ways(cfg, list(range(n)))):
            make(batch, cams)
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            torch.cuda._sleep(4000000)                                           # (so that the host's share does not count)
            start.record()
            for _ in range(8):
                make(batch, cams)
            end.record()
            torch.cuda.synchronize()
            best[i] = min(best[i], start.elapsed_time(end))
    assert best[0] <= 1.1 * best[1], best
    batch.destroy()


@pytest.mark.parametrize("world,extra,keys", [("columns", {"n_rects": 5}, 1), ("columns", {"n_rects": 0}, 0), ("segments", {"n_rects": 0}, 0), ("rooms", {"n_lines": 0}, 1)])
def test_launches_are_counted(world, extra, keys):
    """Every kernel that was launched and no other: keys (without rectangles there is nothing to launch), the world store, palettes and boxes."""
    from paper_2107_08170_b200 import binding as B, scenes
    cfg = scenes.config("rooms", num_envs=3, agents=1, grid=(16, 8, 16), movable_boxes=2, world=world, extra=extra)
    batch = B.Batch(B.desc_from_config(cfg, 0))
    cams = torch.zeros(3, 6, dtype=torch.int32, device="cuda")
    before = batch.launch_count()
    scenes.native_upload(cfg, scenes.native_desc(cfg), torch.tensor([1, 2], device="cuda"), batch, [0, 2], cams)
    assert batch.launch_count() - before == keys + 2
    torch.cuda.synchronize()
    batch.destroy()


def test_more_agents_than_cells_are_refused():
    from paper_2107_08170_b200 import binding as B, scenes
    for agents, fits in ((16, True), (17, False)):
        cfg = scenes.config("rooms", num_envs=1, agents=agents, grid=(4, 8, 4), width=16, height=8, extra={"n_lines": 0, "n_pillars": 0})
        batch = B.Batch(B.desc_from_config(cfg, 0))
        cams = torch.zeros(agents, 6, dtype=torch.int32, device="cuda")
        make = lambda: scenes.native_upload(cfg, scenes.native_desc(cfg), torch.tensor([1], device="cuda"), batch, [0], cams)
        if fits:
            make()
            at = cams.view(torch.float32)[:, [0, 2]].floor().int()
            assert len(set(map(tuple, at.tolist()))) == agents and at.min() >= 0 and at.max() <= 3
        else:
            with pytest.raises(B.MvError) as refused:
                make()
            assert refused.value.code == -1
        batch.destroy()
