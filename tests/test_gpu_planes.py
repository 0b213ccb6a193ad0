"""Grids of several occupancy planes (more than 32 high), the CTA shapes of large blocks and the end of a large grid, against the
oracle and against each other."""
import numpy as np
import pytest
import torch

import parity
from helpers import cam_row
from test_gpu_parity import _binding, _pal, _render_custom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gy", [36, 60, 64, 96, 132, 1024])
def test_walks_that_cross_planes(oracle, gy):
    """A plane is 31 heights: worlds filled thinly, so that walks cross planes up and down, with solid slabs that end just
    below, at and just above a plane's first and last height; eyes in every plane, also next to its ends, looking up and
    down; one world filled only low down, one only high up, one eye above everything, one outside the grid."""
    rng = np.random.default_rng(gy)
    gx, gz, E = 20, 24, 14
    g = np.where(rng.random((E, gy, gz, gx)) < 0.01, rng.integers(1, 6, (E, gy, gz, gx)), 0).astype(np.uint8)
    g[:, 0] = 1
    cams = []
    for e in range(E):
        edge = 31 * (1 + e % ((gy - 1) // 31))                    # first height of a plane
        y = [edge - 1, edge, edge + 1, edge - 2, 1, gy - 3, edge - 8, min(edge + 8, gy - 2)][e % 8]
        if e < 6:                                                 # a slab with a hole, its top or bottom at the plane's edge
            lo = min(max(edge + (e % 3) - 1, 1), gy - 2)
            g[e, lo:lo + 2, :, :gx // 2] = 2
        if e == 8:
            g[e, 6:] = 0
            y = 3
        if e == 9:
            g[e, :gy - 8] = 0
            y = gy - 6
        if e == 10:
            g[e, gy - 20:] = 0
            y = gy - 10
        y = min(max(y, 1), gy - 2)
        at = np.array([rng.integers(3, gx - 3), y, rng.integers(3, gz - 3)])
        g[e, max(at[1] - 1, 1):at[1] + 2, at[2] - 1:at[2] + 2, at[0] - 1:at[0] + 2] = 0
        p = at + rng.uniform(0.1, 0.9, 3)
        if e == 11:
            p = np.array([-4.0, gy * 0.6, gz * 0.5])
        cams.append(cam_row(*p, rng.uniform(0, 6.28), [0.9, -0.9, 1.3, -1.3, 0.2, -0.3][e % 6]))
    frames = _render_custom(oracle, g, _pal(E, 6), np.stack(cams), 64, 36)
    assert frames[2] == 0
    parity.assert_parity(frames[3], f"planes {gy}")
    # the same bytes with the occupancy read from global memory
    B = _binding()
    batch = B.Batch(B.make_desc(E, 1, (gx, gy, gz), 0, 64, 36, 6))
    batch.upload_worlds(0, E, torch.from_numpy(g).cuda(), palette=torch.from_numpy(_pal(E, 6)).cuda())
    batch.set_cameras(torch.from_numpy(np.stack(cams)).cuda())
    batch.debug_occupancy_in_global(True)
    rgb, depth = batch.alloc_outputs()
    batch.render_batch(rgb, depth)
    assert (rgb.cpu().numpy() == frames[0]).all() and (depth.cpu().numpy() == frames[1]).all()
    batch.destroy()


@pytest.mark.parametrize("grid,agents", [((160, 12, 160), 1), ((192, 8, 192), 1), ((192, 8, 192), 3), ((100, 64, 120), 2)])
def test_large_blocks_in_wide_ctas(oracle, grid, agents):
    """Blocks that leave room for two CTAs on an SM, or for one: the oracle's frames, and the same ones staged and with the
    occupancy in global memory."""
    B = _binding()
    gx, gy, gz = grid
    rng = np.random.default_rng(gx + gy)
    E, P, mb = 3, 9, 5
    g = np.where(rng.random((E, gy, gz, gx)) < 0.03, rng.integers(1, P, (E, gy, gz, gx)), 0).astype(np.uint8)
    g[:, 0] = 3
    cams = np.stack([cam_row(*(np.array([gx, 0, gz]) * rng.uniform(0.3, 0.7, 3) + [0, rng.uniform(1.2, gy - 1.2), 0]), rng.uniform(0, 6.28),
                             rng.uniform(-0.5, 0.5)) for _ in range(E * agents)])
    boxes = np.zeros((E, mb, 8), np.float32)
    lo = rng.uniform(0.2, 0.8, (E, mb, 3)) * [gx, gy, gz]
    boxes[..., :3], boxes[..., 3:6] = lo, lo + rng.uniform(0.5, 3, (E, mb, 3))
    boxes = boxes.view(np.int32)
    boxes[..., 6] = rng.integers(0, P, (E, mb))
    count = np.full(E, mb, np.int32)
    rgb, depth, status, st = _render_custom(oracle, g, _pal(E, P), cams, 96, 52, boxes, count, agents, mb)
    assert status == 0
    parity.assert_parity(st, f"wide {grid}")
    batch = B.Batch(B.make_desc(E, agents, grid, mb, 96, 52, P))
    batch.upload_worlds(0, E, torch.from_numpy(g).cuda(), torch.from_numpy(boxes).cuda(), torch.from_numpy(count).cuda(),
                        torch.from_numpy(_pal(E, P)).cuda())
    batch.set_cameras(torch.from_numpy(cams).cuda())
    for in_global in (True, False):
        batch.debug_occupancy_in_global(in_global)
        out = batch.alloc_outputs()
        batch.render_batch(*out)
        assert (out[0].cpu().numpy() == rgb).all() and (out[1].cpu().numpy() == depth).all(), in_global
    batch.destroy()


@pytest.mark.parametrize("agents,size", [(1, (72, 52)), (1, (136, 72)), (2, (72, 52)), (3, (48, 40)), (6, (64, 36))])
def test_the_end_of_the_grid_in_parts(oracle, agents, size):
    """A few rounds of CTAs: the last observations in parts or one by one, behind CTAs that render whole ones or all agents of an
    environment; the same bytes as with every observation in one CTA and in three, overlays and bad cameras included."""
    from paper_2107_08170_b200 import scenes
    B = _binding()
    envs = 1500 // agents if agents < 6 else 450
    cfg = scenes.config("rooms", num_envs=envs, agents=agents, grid=(16, 12, 16), width=size[0], height=size[1], movable_boxes=4,
                        extra={"n_lines": 1})
    sc = scenes.make_scene(cfg, device="cuda")
    batch = B.Batch(B.desc_from_config(cfg, 0, max_overlay_rects=1))
    batch.upload_worlds(0, envs, sc["grid"], sc["boxes"], sc["box_count"], sc["palette"])
    for o in (0, cfg.num_obs // 2, cfg.num_obs - 1):
        sc["cams"][o, 3] = torch.tensor([float("nan")]).view(torch.int32).item()
    rects = torch.zeros(cfg.num_obs, 1, 4, dtype=torch.int32)
    rects[..., 1], rects[..., 2] = size[0] // 2 | (3 << 16), 0x20C0FF
    batch.set_overlays(rects.cuda(), torch.ones(cfg.num_obs, dtype=torch.int32, device="cuda"))
    batch.set_cameras(sc["cams"])
    assert batch.query_status(clear=True) == B.FLAG_BAD_CAMERA
    want = None
    for apc in sorted({1, agents}):
        for parts in (1, 3, 0):
            assert batch.debug_parts(parts) == max(parts, 1)                 # (0: the library's choice, which begins with whole ones)
            whole = batch.debug_agents_per_cta(apc)
            assert whole == 0 if parts else 0 < whole <= envs * agents // apc
            rgb, depth = batch.alloc_outputs()
            rgb.fill_(9); depth.fill_(-3.0)
            batch.render_batch(rgb, depth)
            want = want or (rgb, depth)
            assert torch.equal(rgb, want[0]) and torch.equal(depth, want[1]), (apc, parts)
    batch.destroy()


def test_boxes_across_the_eye_plane(oracle):
    """Boxes across the eye plane that are off to one side go to no tile, those that reach into the view to all: beside, above and
    below the eye, touching the view's edge from outside and inside, around the eye, long ones that cross the view, and some of
    infinite extent, at narrow and wide angles."""
    from helpers import box_rows
    rng = np.random.default_rng(4)
    E, nb, gx = 12, 40, 24
    g = np.zeros((E, 16, gx, gx), np.uint8)
    g[:, 0] = 1
    eye = np.array([12.3, 8.2, 12.6])
    cams, boxes = [], []
    for e in range(E):
        yaw, pitch = rng.uniform(0, 6.28), rng.uniform(-0.9, 0.9)
        cams.append(cam_row(*eye, yaw, pitch))
        fwd = np.array([np.cos(pitch) * np.sin(yaw), np.sin(pitch), np.cos(pitch) * np.cos(yaw)])
        right = np.array([np.cos(yaw), 0, -np.sin(yaw)])
        up = np.cross(fwd, right)
        items = []
        for n in range(nb):
            side = (right, -right, up, -up)[n % 4] * rng.uniform(0.3, 7) + fwd * rng.uniform(-1.0, 1.5)
            half = rng.uniform(0.05, 1.5, 3)
            if n % 10 == 9:
                half[n // 10 % 3] = 9.0                        # a long one
            c = eye + side
            if n == 5:
                c, half = eye + fwd * 0.2, np.array([0.4, 0.3, 0.5])   # around the eye
            lo, hi = c - half, c + half
            if n == 7:
                lo[1] = -np.inf
            if n == 11:
                hi[0] = np.inf
            items.append((lo, hi, 1 + n % 5))
        boxes.append(box_rows(items))
    for hfov in (0.5, 1.5707964, 2.6):
        for only in (range(nb), [5, 7, 11], [n for n in range(nb) if n not in (5, 7, 11)]):
            some = np.stack([b[list(only)] for b in boxes])
            rgb, depth, status, st = _render_custom(oracle, g, _pal(E, 6), np.stack(cams), 64, 36, some, np.full(E, len(list(only)), np.int32), 1,
                                                    some.shape[1], hfov_rad=hfov)
            assert status == 0
            parity.assert_parity(st, f"across the eye plane {hfov}")


def test_a_tall_world_is_uploaded_by_as_many_ctas_as_low_ones():
    """One world of 1024 heights takes about as long as 32 of 32 heights, the same bytes.  With a column's 32 tiles one behind the
    other in a CTA it was 12 times as long (74 us); three times is well beyond what runs differ by."""
    B = _binding()
    times = {}
    for E, gy in ((1, 1024), (32, 32)):
        grid = torch.randint(0, 3, (E, gy, 16, 16), dtype=torch.uint8, device="cuda")
        batch = B.Batch(B.make_desc(E, 1, (16, gy, 16), 0, 64, 36, 3))
        runs = []
        for _ in range(8):
            begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            begin.record()
            for _ in range(50):
                batch.upload_worlds(0, E, grid)
            end.record()
            end.synchronize()
            runs.append(begin.elapsed_time(end))
        times[gy] = min(runs)
        batch.destroy()
    assert times[1024] < 3 * times[32], times


@pytest.mark.parametrize("grid,size,boxes,envs,in_global", [
    ((64, 16, 64), (640, 360), 32, 300, False), ((64, 16, 64), (480, 272), 36, 1000, False), ((16, 8, 16), (640, 360), 0, 200, False),
    ((192, 32, 192), (128, 72), 0, 220, False), ((192, 32, 192), (128, 72), 0, 1000, True), ((128, 48, 128), (128, 72), 0, 600, True),
    ((96, 32, 96), (480, 272), 16, 1000, False), ((160, 32, 160), (128, 72), 0, 2048, False), ((192, 48, 192), (128, 72), 0, 1, True)])
def test_where_the_occupancy_is_read(grid, size, boxes, envs, in_global):
    """Left in global memory only where that makes room for three CTAs on an SM instead of one and there are more observations than
    those hold: not under images whose tables fill the SM anyway, nor in a batch that is resident at once."""
    B = _binding()
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the numbers of observations are for 148 SMs")
    batch = B.Batch(B.make_desc(envs, 1, grid, boxes, *size, 4))
    assert batch.debug_occupancy_in_global(None) == in_global
    batch.destroy()


def test_staging_that_does_not_fit_beside_all_agents_is_refused():
    """More observations than are resident at once, several agents and a block near the limit: the library reads the occupancy
    from global memory and lets a CTA render all ten agents, beside whom the block would not fit.  The hook says so, the batch
    renders on, and with a CTA per observation it stages the block; the same bytes each time."""
    B = _binding()
    A, envs, grid, boxes = 10, 450, (224, 12, 224), 40
    batch = B.Batch(B.make_desc(envs, A, grid, boxes, 64, 36, 4))
    worlds = torch.zeros(envs, grid[1], grid[2], grid[0], dtype=torch.uint8, device="cuda")
    worlds[:, 0] = 1
    worlds[:, :5, ::9, ::7] = 2
    batch.upload_worlds(0, envs, worlds, torch.zeros(envs, boxes, 8, dtype=torch.int32, device="cuda"),
                        torch.zeros(envs, dtype=torch.int32, device="cuda"), torch.full((envs, 4, 3), 90, dtype=torch.uint8, device="cuda"))
    rng = np.random.default_rng(2)
    cams = np.stack([cam_row(*rng.uniform(20, 200, 1), 3.5, *rng.uniform(20, 200, 1), rng.uniform(0, 6.28), -0.1) for _ in range(envs * A)])
    batch.set_cameras(torch.from_numpy(cams).cuda())
    frames = []

    def render():
        out = batch.alloc_outputs()
        batch.render_batch(*out)
        assert batch.query_status() == 0
        frames.append(out)

    assert batch.debug_occupancy_in_global(None) and batch.debug_agents_per_cta(0) <= envs
    render()
    with pytest.raises(B.MvError) as refused:
        batch.debug_occupancy_in_global(False)
    assert refused.value.code == -6
    render()
    batch.debug_agents_per_cta(1)
    assert not batch.debug_occupancy_in_global(False)
    render()
    assert batch.debug_agents_per_cta(A) > 0 and batch.debug_occupancy_in_global(None)
    render()
    for rgb, depth in frames[1:]:
        assert torch.equal(rgb, frames[0][0]) and torch.equal(depth, frames[0][1])
    batch.destroy()


@pytest.mark.parametrize("agents", [1, 2])
def test_many_small_images_of_tall_grids(oracle, agents):
    """The CTAs of six warps that small images get in a large batch, on a grid of two planes: staged and with the occupancy in
    global memory the same bytes, and some of them against the oracle."""
    from gpu_util import scene_to_numpy
    from paper_2107_08170_b200 import scenes
    B = _binding()
    cfg = scenes.config("rooms", num_envs=1000, agents=agents, grid=(16, 36, 16), width=64, height=36, movable_boxes=4, extra={"n_lines": 1})
    sc = scenes.make_scene(cfg, device="cuda")
    for e in range(0, 1000, 3):                                   # every third world filled only low down
        sc["grid"][e, 6:] = 0
    batch = B.Batch(B.desc_from_config(cfg, 0))
    batch.upload_worlds(0, 1000, sc["grid"], sc["boxes"], sc["box_count"], sc["palette"])
    batch.set_cameras(sc["cams"])
    out = []
    for in_global in (False, True):
        assert batch.debug_occupancy_in_global(in_global) == in_global
        rgb, depth = batch.alloc_outputs()
        rgb.fill_(9); depth.fill_(-3.0)
        batch.render_batch(rgb, depth)
        out.append((rgb, depth))
    assert batch.query_status() == 0
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    some = [0, 1, 2, 333 * agents, 500 * agents, cfg.num_obs - 1]
    st = parity.compare_scene(oracle, cfg, scene_to_numpy(sc), some, out[0][0][some].cpu().numpy(), out[0][1][some].cpu().numpy())
    parity.assert_parity(st, f"small images {agents}")
    batch.destroy()


def test_more_observations_than_staged_blocks(oracle):
    """A batch that the library renders with the occupancy in global memory although the block would fit: the bytes that the same
    worlds and cameras have in a small batch, whose blocks are staged, and some against the oracle."""
    from gpu_util import scene_to_numpy
    from paper_2107_08170_b200 import scenes
    B = _binding()
    cfg = scenes.config("rooms", num_envs=460, agents=1, grid=(192, 12, 192), width=64, height=36, movable_boxes=0, extra={"n_lines": 8})
    sc = scenes.make_scene(cfg, device="cuda")
    frames = {}
    for n in (460, 40):
        batch = B.Batch(B.make_desc(n, 1, cfg.grid, 0, 64, 36, cfg.palette_size))
        assert batch.debug_occupancy_in_global(None) == (n == 460)
        batch.upload_worlds(0, n, sc["grid"][:n].contiguous(), palette=sc["palette"][:n].contiguous())
        batch.set_cameras(sc["cams"][:n].contiguous())
        rgb, depth = batch.alloc_outputs()
        batch.render_batch(rgb, depth)
        assert batch.query_status() == 0
        frames[n] = rgb, depth
        batch.destroy()
    assert torch.equal(frames[460][0][:40], frames[40][0]) and torch.equal(frames[460][1][:40], frames[40][1])
    some = [0, 39, 230, 459]
    st = parity.compare_scene(oracle, cfg, scene_to_numpy(sc), some, frames[460][0][some].cpu().numpy(), frames[460][1][some].cpu().numpy())
    parity.assert_parity(st, "from global memory")


def test_the_height_of_a_grid_does_not_limit_the_image():
    """An image whose tables fill shared memory to the last hundred bytes fits whatever the grid's height, as what a CTA keeps of
    the planes has one size."""
    B = _binding()
    accepted = {}
    for gy in (4, 64, 1024):
        for palette in range(60, 120, 4):
            try:
                B.Batch(B.make_desc(1, 1, (4, gy, 4), 0, 480, 764, palette)).destroy()
                accepted.setdefault(gy, []).append(palette)
            except B.MvError as e:
                assert e.code == -6
    assert accepted[4] and accepted[4][-1] < 116 and accepted[64] == accepted[4] and accepted[1024] == accepted[4], accepted
