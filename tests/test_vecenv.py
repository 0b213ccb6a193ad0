"""The vectorised step() wrapper: bookkeeping on CPU, whole loop on the GPU against the oracle."""
import numpy as np
import pytest
import torch

from paper_2107_08170_b200 import scenes, vecenv


def test_time_bar_rects_layout():
    rec = vecenv.time_bar_rects([10, 5, 0], [10, 10, 4], 128, 2)
    assert rec.shape == (6, 1, 4) and rec.dtype == torch.int32
    raw = rec.numpy().view(np.int16).reshape(6, 8)
    assert raw[:, 0].tolist() == [0] * 6 and raw[:, 1].tolist() == [0] * 6          # x0, y0
    assert raw[:, 2].tolist() == [128, 128, 64, 64, 0, 0]                             # x1 = W * left / len
    assert (raw[:, 3] == vecenv.BAR_ROWS).all()                                       # y1
    assert (rec.numpy().view(np.uint8).reshape(6, 16)[:, 8:11] == np.array(vecenv.BAR_RGB, np.uint8)).all()


@pytest.mark.gpu
def test_step_loop_with_auto_reset_matches_oracle(oracle):
    import parity
    from gpu_util import scene_to_numpy
    cfg = scenes.config("rooms_boxes", num_envs=4)
    lens = [3, 4, 5, 50]
    env = vecenv.VecRenderEnv(cfg, lens)
    env.reset()
    A, E = cfg.agents, cfg.num_envs
    # CPU mirror of the state
    state = [scene_to_numpy(scenes.make_scene(cfg, e, 1)) for e in range(E)]
    t = np.zeros(E, int); ep = np.zeros(E, int)
    rng = np.random.default_rng(3)
    dones = []
    for step in range(7):
        moves = np.stack([rng.uniform(-0.4, 0.4, cfg.num_obs), rng.uniform(-0.2, 0.2, cfg.num_obs),
                          rng.normal(0, 0.3, cfg.num_obs), rng.normal(0, 0.05, cfg.num_obs)], 1).astype(np.float32)
        rgb, depth, done = env.step(torch.from_numpy(moves).cuda())
        dones.append(done.tolist())
        for e in range(E):
            s = state[e]
            for a in range(A):
                f = s["cams"][a, :5].view(np.float32)
                new, _ = oracle.move_agent(s["grid"][0], f, moves[e * A + a], (0.25, 0.75, 0.25), 1.0)
                s["cams"][a, :5] = new.view(np.int32)
                sb = s["cams"][a, 5]
                s["boxes"][0, sb, :3] = (new[:3] - np.float32([0.25, 0.75, 0.25])).view(np.int32)
                s["boxes"][0, sb, 3:6] = (new[:3] + np.float32([0.25, 0.25, 0.25])).view(np.int32)
            t[e] += 1
            if t[e] >= lens[e]:
                ep[e] += 1; t[e] = 0
                state[e] = scene_to_numpy(scenes.make_scene(cfg, e + ep[e] * E, 1))
    assert dones[2] == [True, False, False, False] and dones[3] == [False, True, False, False]
    assert dones[5] == [True, False, False, False] and not any(d[3] for d in dones)
    # final frames: 3D view per the oracle, then the time bar on top
    g_rgb, g_depth = rgb.cpu().numpy(), depth.cpu().numpy()
    bars = vecenv.time_bar_rects(np.array(lens) - t, lens, cfg.width, A).numpy()
    desc = oracle.desc_from_config(cfg)
    total = None
    for e in range(E):
        s = state[e]
        for a in range(A):
            o = e * A + a
            o_rgb, o_depth, o_ids = oracle.render_obs(desc, s["grid"][0], s["boxes"][0], s["box_count"][0],
                                                      s["palette"][0], s["cams"][a])
            rect = bars[o].view(oracle.RECT_DTYPE).reshape(-1)
            o_rgb = oracle.overlay(np.ascontiguousarray(o_rgb), rect, 1)
            # the bar hides the 3D pixels under it on both sides, so the parity rule applies as is
            st = parity.compare_obs(oracle, desc, s["grid"][0], s["boxes"][0], int(s["box_count"][0]),
                                    s["palette"][0], s["cams"][a], g_rgb[o], g_depth[o], o_rgb, o_depth, o_ids)
            total = st if total is None else {k: total[k] + st[k] for k in st}
    parity.assert_parity(total, "vecenv")
    bar_len = int(bars[0].view(np.int16).reshape(-1)[2])
    assert (g_rgb[0, :2, :bar_len] == np.array(vecenv.BAR_RGB, np.uint8)).all()
    env.close()


@pytest.mark.parametrize("inference", [False, True])
def test_host_copy_of_a_clock_follows_every_change(inference):
    with torch.inference_mode(inference):
        clock = vecenv._Clock(torch.arange(6), "cpu")
        assert not clock.tensor.is_inference()

        def follows():
            clock.refresh()
            return clock.host.tolist() == clock.tensor.tolist()

        assert follows()
        quiet = clock.host
        clock.refresh()
        assert clock.host is quiet                                     # nothing changed: nothing is read
        for change in (lambda t: t.__setitem__(2, 40), lambda t: t.fill_(3), lambda t: t[1:4].add_(2),
                       lambda t: t.masked_fill_(t > 4, 0), lambda t: torch.add(t, 1, out=t), lambda t: t.view(2, 3).zero_()):
            before = clock.tensor.tolist()
            change(clock.tensor)
            assert clock.tensor.tolist() != before and follows()
            assert clock.host is not quiet
        mine = torch.arange(6) * 7                                     # (under inference mode one that counts no changes)
        clock.assign(mine)
        assert follows() and clock.host.tolist() == [0, 7, 14, 21, 28, 35]
        mine[0] = 9
        assert clock.tensor[0] == 9 and follows()                      # taken as it is, not copied
        clock.assign(5)
        assert clock.tensor.tolist() == [5] * 6 and clock.tensor.dtype == torch.int64 and follows()
        clock.host += 1                                                # the host's own step leaves the device's tensor alone
        assert clock.tensor.tolist() == [5] * 6


@pytest.mark.gpu
@pytest.mark.parametrize("inference", [False, True])
def test_clocks_set_by_the_caller_end_episodes(inference):
    """t, episode and episode_len belong to the caller too: whatever is put there between steps decides which
    environments the next step resets, and to which world."""
    from gpu_util import render_scene
    cfg = scenes.config("rooms_boxes", num_envs=4, agents=2)
    E, A = cfg.num_envs, cfg.agents
    first = lambda scene_id: [torch.from_numpy(v) for v in render_scene(scenes.config("rooms_boxes", num_envs=1, agents=2),
                                                                       scenes.make_scene(cfg, scene_id, 1))[:2]]
    still = torch.zeros(cfg.num_obs, 4, device="cuda")
    with torch.inference_mode(inference):
        env = vecenv.VecRenderEnv(cfg, 10, time_bar=False)
        env.reset()

        def step(ended):
            rgb, depth, done = env.step(still)
            assert done.tolist() == [e in ended for e in range(E)]
            for e, k in ended.items():
                want = first(e + k * E)
                assert torch.equal(rgb[e * A:e * A + A].cpu(), want[0]) and torch.equal(depth[e * A:e * A + A].cpu(), want[1])
                assert int(env.episode[e]) == k and int(env.t[e]) == 0
            env._refresh()
            assert all(c.host.tolist() == c.tensor.tolist() for c in env._clocks.values())

        step({})
        env.t[1] = 9                                                   # early termination
        step({1: 1})
        step({})
        env.episode[2] = 5
        env.t[2:4] = 100
        step({2: 6, 3: 1})
        env.episode_len[0] = int(env.t[0]) + 1
        step({0: 1})
        env.episode_len = 1
        env.t = torch.zeros(E, dtype=torch.int64, device="cuda")
        step({0: 2, 1: 2, 2: 7, 3: 2})
        env.t.data[0] = -1                                             # not seen by torch, so said by hand
        env.t = env.t
        step({1: 3, 2: 8, 3: 3})
    env.close()


@pytest.mark.gpu
@pytest.mark.parametrize("change", [{"extra": {"n_lines": 1, "n_pillars": 200}}, {"world": "columns", "extra": {"n_rects": 30}}, {"seed": 77}, {},
                                    {"movable_boxes": 0}, {"movable_boxes": 40}])
def test_worlds_follow_a_changed_configuration(change):
    """A configuration changed between steps (a curriculum): the episodes that begin then have its grids and palettes; boxes and cameras
    are dealt out over those as the object was made to."""
    from paper_2107_08170_b200 import binding as B
    make = lambda **over: scenes.config("rooms_boxes", num_envs=3, agents=2, **over)
    cfg, A = make(), 2
    desc = scenes.native_desc(cfg)
    env = vecenv.VecRenderEnv(cfg, 2, time_bar=False)
    env.reset()
    still = torch.zeros(cfg.num_obs, 4, device="cuda")
    env.step(still)
    for name, value in change.items():
        setattr(cfg, name, value)
    rgb, depth, done = env.step(still)
    assert done.all()
    ids = torch.arange(3, 6, device="cuda")
    w = scenes.make_worlds(make(**change), device="cuda", env_ids=ids)
    e = scenes.native_entities(make(), desc, ids, w["height"])
    batch = B.Batch(B.desc_from_config(make()))
    batch.upload_worlds(0, 3, w["grid"], e["boxes"], e["box_count"], w["palette"])
    batch.set_cameras(e["cams"])
    want = batch.alloc_outputs()
    batch.render_batch(*want)
    assert torch.equal(env.cams, e["cams"]) and torch.equal(rgb, want[0]) and torch.equal(depth, want[1])
    batch.destroy()
    env.close()


@pytest.mark.gpu
@pytest.mark.parametrize("change,refused", [({"grid": (64, 16, 60)}, ValueError), ({"palette_size": 63}, ValueError), ({"world": "maze"}, ValueError)])
def test_configurations_the_batch_was_not_made_for_are_refused(change, refused):
    cfg = scenes.config("rooms_boxes", num_envs=3, agents=2)
    env = vecenv.VecRenderEnv(cfg, 1, time_bar=False)
    env.reset()
    for name, value in change.items():
        setattr(cfg, name, value)
    with pytest.raises(refused):
        env.step(torch.zeros(cfg.num_obs, 4, device="cuda"))
    env.close()


@pytest.mark.gpu
def test_resets_send_what_they_need(monkeypatch):
    """To new episodes that go straight into the batch one id each; elsewhere their destinations, too."""
    cfg = scenes.config("rooms_boxes", num_envs=5, agents=2)
    env = vecenv.VecRenderEnv(cfg, 4, time_bar=False, phase=torch.tensor([3, 0, 3, 3, 0]))
    env.reset()
    still, sent, real = torch.zeros(cfg.num_obs, 4, device="cuda"), [], torch.from_numpy
    monkeypatch.setattr(torch, "from_numpy", lambda a: (sent.append(a.nbytes), real(a))[1])
    env.step(still)
    assert sent == [3 * 8]
    cfg.seed = 8
    env.t.fill_(3)
    env.step(still)
    assert sent == [3 * 8, 2 * 5 * 8]
    env.close()


def test_recipe_sees_every_change_of_the_scenes():
    """Whatever the library's generator is told, changes in place included."""
    make = lambda: scenes.config("rooms", extra={"n_lines": 2})
    made = vecenv._recipe(make())
    assert vecenv._recipe(make()) == made
    for name, value in dict(world="columns", seed=9, grid=(64, 20, 64), palette_size=9, agents=1, movable_boxes=3, body_boxes=True, cam_y_fixed=0.5).items():
        cfg = make()
        before = bytes(scenes.native_desc(cfg))
        setattr(cfg, name, value)
        desc = scenes.native_desc(cfg)
        assert desc is None or bytes(desc) != before
        assert vecenv._recipe(cfg) != made
    cfg = make()
    made = vecenv._recipe(cfg)
    cfg.extra["n_lines"] = 3
    assert vecenv._recipe(cfg) != made
