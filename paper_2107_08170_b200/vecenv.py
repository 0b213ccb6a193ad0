"""Vectorised step() interface over the C ABI (paper Appendix A.1): one call advances N
environments x M agents and returns N x M observations and N termination flags; finished
environments are reset automatically, so the last frame of an episode is never rendered.

Scenario logic, rewards and object physics are outside this library: an "episode" here is a
fixed number of steps, after which the environment gets a freshly generated world.  The
time-left bar of Appendix A.2 is drawn through the GUI overlay.  Observations are zero-copy CUDA
tensors owned by this object (Section 3.2: frames exposed directly as GPU-side tensors).

Built for thousands of environments: episode clocks, time-left bars, agent state and the generation of new worlds
all run on the GPU.  The host keeps its own copy of the clocks and so knows which environments end without asking: a step
enqueues its work and reads nothing back, unless the caller has changed a clock since the last one."""
from __future__ import annotations

import numpy as np
import torch

from . import binding, scenes

BAR_RGB = (250, 240, 30)
BAR_ROWS = 2
_GEN_CHUNK = 512            # environments generated per scene-generator call


def time_bar_rects(steps_left, episode_len, width, agents):
    """int32 [E*agents][1][4] overlay records: a bar of BAR_ROWS rows whose length is the share of
    the episode that is left, rounded down to whole pixels.  Runs on the device of its inputs."""
    steps_left = torch.as_tensor(steps_left, dtype=torch.int64)
    episode_len = torch.as_tensor(episode_len, dtype=torch.int64).to(steps_left.device)
    x1 = (width * steps_left) // episode_len.clamp(min=1)
    x1 = x1.clamp(0, width).repeat_interleave(agents)
    n = x1.numel()
    rec = torch.zeros(n, 1, 4, dtype=torch.int32, device=steps_left.device)
    rec[:, 0, 1] = x1.to(torch.int32) | (BAR_ROWS << 16)   # x1 (low half), y1 (high half); x0 = y0 = 0
    rec[:, 0, 2] = BAR_RGB[0] | (BAR_RGB[1] << 8) | (BAR_RGB[2] << 16)
    return rec


class _Clock:
    """A per-env counter on the device that callers may change, and the host's copy of it."""

    def __init__(self, values: torch.Tensor, device):
        with torch.inference_mode(False):           # (an inference tensor does not count its changes)
            self._take(values.to(device, copy=True))
        self.refresh()

    def _take(self, tensor):
        self.tensor, self._counts, self._seen = tensor, not tensor.is_inference(), None

    def assign(self, value):
        """`value` (a tensor of the right kind is taken as it is, not copied) instead of the present tensor."""
        like = self.tensor
        self._take(torch.as_tensor(value, dtype=like.dtype, device=like.device).expand(like.shape).contiguous())

    def refresh(self):
        """Brings the host's copy up to date if the tensor was changed since it was read."""
        if self._counts and self.tensor._version == self._seen:
            return
        self.host = self.tensor.cpu().numpy().copy()
        self._seen = self.tensor._version if self._counts else None


def _clock_property(name, doc):
    return property(lambda self: self._clocks[name].tensor, lambda self, value: self._clocks[name].assign(value), doc=doc)


def _recipe(cfg: scenes.SceneConfig):
    """What the scenes of a configuration depend on."""
    return (cfg.world, cfg.seed, tuple(cfg.grid), cfg.palette_size, cfg.agents, cfg.movable_boxes, cfg.body_boxes, cfg.cam_y_fixed, dict(cfg.extra))


class VecRenderEnv:
    """The clocks t, episode and episode_len (CUDA int64 [num_envs]) may be changed between steps, in place by torch
    operations or by assignment, for instance t[i] = episode_len[i] - 1 to end an episode with the next step; that step then
    reads them back once.  (A write that torch does not see, through `.data` or another library's pointer, is made known
    by assigning the tensor to its own name: env.t = env.t.)
    cfg may be changed between steps as far as the batch's sizes allow: the grids and palettes of episodes that begin later
    follow it; boxes and cameras are drawn as the object was made to."""

    t = _clock_property("t", "steps taken in the present episode")
    episode = _clock_property("episode", "episodes finished; env e in its k-th episode shows the seeded scene e + k * num_envs")
    episode_len = _clock_property("episode_len", "steps per episode")

    def __init__(self, cfg: scenes.SceneConfig, episode_len, device: int = 0, time_bar: bool = True, phase=None):
        """episode_len: steps per episode (scalar or one per env).  phase: optional initial value of each
        env's step clock (so that episodes end at different times from the start)."""
        self.cfg, self.device = cfg, torch.device("cuda", device)
        E = cfg.num_envs
        host = lambda v: torch.as_tensor(v, dtype=torch.int64).expand(E).cpu().clone()
        self._clocks = {"t": _Clock(host(0 if phase is None else phase), self.device),
                        "episode": _Clock(torch.zeros(E, dtype=torch.int64), self.device),
                        "episode_len": _Clock(host(episode_len), self.device)}
        self.time_bar = time_bar
        self.batch = binding.Batch(binding.desc_from_config(cfg, device, max_overlay_rects=1 if time_bar else 0))
        self.cams = torch.zeros(cfg.num_obs, 6, dtype=torch.int32, device=self.device)
        self.rgb, self.depth = self.batch.alloc_outputs()
        self._native = scenes.native_desc(cfg)
        self._made_by = _recipe(cfg)
        self._started = False

    def _load_envs(self, envs):
        """Fresh worlds for the env indices in `envs` (sorted int64 array), each in its current episode: env e in its
        k-th episode uses the seeded scene id e + k * num_envs."""
        A = self.cfg.agents
        # straight into the batch while the scenes' configuration is the one that this object was made with
        direct = self._native is not None and _recipe(self.cfg) == self._made_by
        made = self.batch.desc
        if not direct and (tuple(self.cfg.grid), self.cfg.palette_size) != ((made.grid_x, made.grid_y, made.grid_z), made.palette_size):
            raise ValueError("the grid's size and the number of colours are fixed when the environment is made")
        if self._native is None and (self.cfg.agents, self.cfg.max_boxes) != (made.agents_per_env, made.max_boxes):
            raise ValueError("the numbers of agents and boxes are fixed when the environment is made")
        for c0 in range(0, len(envs), _GEN_CHUNK):
            chunk = envs[c0:c0 + _GEN_CHUNK]
            # ids, and destinations (as int32) where an upload does not bring them, in one pinned copy that nothing waits for
            host = np.empty((1 if direct else 2, len(chunk)), np.int64)
            host[0] = chunk + self._clocks["episode"].host[chunk] * self.cfg.num_envs
            if not direct:
                host[1].view(np.int32)[:len(chunk)] = chunk
            sent = torch.from_numpy(host).pin_memory().to(self.device, non_blocking=True)
            ids = sent[0]
            if direct:
                scenes.native_upload(self.cfg, self._native, ids, self.batch, chunk.astype(np.int32), self.cams)
                continue
            dst = sent[1].view(torch.int32)[:len(chunk)]
            w = scenes.make_worlds(self.cfg, device=self.device, env_ids=ids)
            if self._native is not None:
                e = scenes.native_entities(self.cfg, self._native, ids, w["height"], self.cams, dst)
            else:
                e = scenes.make_boxes_and_cameras(self.cfg, w)
                self.cams.view(-1, A, 6)[dst.long()] = e["cams"].view(-1, A, 6)
            boxes = count = None
            if made.max_boxes > 0:
                boxes, count = e["boxes"], e["box_count"]
            self.batch.upload_worlds_at(chunk.astype(np.int32), w["grid"], boxes, count, w["palette"])

    def _refresh(self):
        for clock in self._clocks.values():
            clock.refresh()

    def _advance(self, done=None):
        """Advance the clocks (with `done`) and draw the time-left bars."""
        if done is not None or self.time_bar:
            self.batch.advance_episodes(self.t, self.episode, self.episode_len, done, BAR_ROWS if self.time_bar else 0, BAR_RGB)

    def reset(self):
        """Only needed once, right after construction."""
        self._refresh()
        self._load_envs(np.arange(self.cfg.num_envs))
        self.batch.set_cameras(self.cams)
        self._started = True
        self._advance()
        self.batch.render_batch(self.rgb, self.depth)
        return self.rgb, self.depth

    def step(self, moves: torch.Tensor):
        """moves: CUDA float32 [num_obs][4] = (forward, strafe, dyaw, dpitch).  Returns
        (rgb [O][H][W][3] uint8, depth [O][H][W] float32, done [E] bool on the GPU); for a finished env
        the frames already show the first view of its next episode."""
        assert self._started, "call reset() once before step()"
        self.batch.move_agents(self.cams, moves.contiguous())
        done = torch.empty(self.cfg.num_envs, dtype=torch.bool, device=self.device)
        self._refresh()
        self._advance(done)
        t = self._clocks["t"].host
        t += 1
        finished = np.flatnonzero(t >= self._clocks["episode_len"].host)
        if len(finished):
            self._clocks["episode"].host[finished] += 1
            t[finished] = 0
            self._load_envs(finished)
            self.batch.set_cameras(self.cams)
        self.batch.render_batch(self.rgb, self.depth)
        return self.rgb, self.depth, done

    def close(self):
        self.batch.destroy()
