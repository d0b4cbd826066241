"""Performance cases of the streaming global-attention step, over the calls a user of the package makes.

A case is one pass of a program that already has its cache handle, its weights and its inputs on the GPU:

  kind "step"        one frame through one layer (layer_step), the cache at its budget: the steady state of a stream
  kind "host"        the same frame with its tensors in pinned host memory (layer_step_host)
  kind "start"       a new scene on a used handle: reset, then the first frames, while the cache fills and first evicts
  kind "camera"      the camera head's caches: one token per frame through every layer (layer_attend, camera_compress)
  kind "stack"       one frame through a stack of global-attention layers with their projections (ProjectionStack)
  kind "aggregator"  one frame through alternating frame- and global-attention blocks with MLPs; all layers are
                     compressed together at the end of the frame (Aggregator: layer_attend, layers_compress)

Inputs are drawn on the GPU: q, k, v ~ N(0, 1), residual rows N(0, I) times a lognormal gain per token, confidence and
coverage ~ U(0, 1): the distributions of the package's own workloads.  Every pass is one more frame of the stream.
"""
from __future__ import annotations

import math

import torch

from paper_2603_05959_b200 import binding as B
from paper_2603_05959_b200 import harness as H
from paper_2603_05959_b200 import inputs as gen

MODES = {"hybrid": B.SCORE_HYBRID, "stored": B.SCORE_RESIDUAL_STORED, "random": B.SCORE_RANDOM, "qk": B.SCORE_QK}
LAYOUTS = {"holes": B.COMPACT_FILL_HOLES, "stable": B.COMPACT_STABLE_GATHER}
DTYPES = {"f32": B.DTYPE_F32, "bf16": B.DTYPE_BF16}


def _case(kind, **kw):
    c = dict(kind=kind, layers=1, heads=16, grid_h=37, grid_w=37, budget=16384, anchor_tokens=64, anchor_interval=100,
             mode="hybrid", layout="holes", dtype="bf16", sigma=0.75, frames=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest stream of the package's configurations: 69 tokens a frame, 256 rows, fp32, anchors every 4 frames
        _case("step", name="tiny_step_f32", heads=4, grid_h=8, grid_w=8, budget=256, anchor_tokens=8, anchor_interval=4,
              sigma=0.5, dtype="f32"),
        # the camera head beside an aggregator: four refinement layers, one token each, 144 frames remembered
        _case("camera", name="camera_head_bf16", layers=4, grid_h=0, grid_w=0, budget=144, anchor_tokens=0),
        # a smaller backbone (12 heads) on an odd frame and an odd budget
        _case("step", name="ragged_step_bf16", heads=12, grid_h=23, grid_w=31, budget=5003, anchor_tokens=37),
        # the memory-lean end of the long streams: 4096 rows, no historical anchors, rows ranked by their stored scores
        _case("step", name="lean_step_stored_bf16", budget=4096, anchor_tokens=0, mode="stored"),
        # the ordinary step: one layer of 16 heads, 1374 tokens a frame, 16384 rows
        _case("step", name="layer_step_bf16", budget=16384),
        # the same step for a program whose tensors are in host memory
        _case("host", name="layer_step_host_bf16", budget=16384),
        # the same step with rows kept in token order on the device
        _case("step", name="layer_step_stable_bf16", budget=16384, layout="stable"),
        # the large end of the long streams
        _case("step", name="long_budget_step_bf16", budget=32768, anchor_tokens=256),
        # a full-width layer run in fp32, as one checks a bf16 run against
        _case("step", name="layer_step_f32", budget=4096, dtype="f32"),
        # the first frames of a scene: short clips never leave this regime
        _case("start", name="scene_start_bf16", budget=8192, frames=8),
        # 24 global-attention layers with their projections, one cache each
        _case("stack", name="stack24_frame_bf16", layers=24, budget=8192),
        # the full alternating aggregator on 518 x 392 frames: 24 + 24 blocks with MLPs
        _case("aggregator", name="aggregator24_frame_bf16", layers=24, grid_h=28, grid_w=37, budget=12288),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["host", "start", "camera", "stack", "aggregator"])
    if kind == "camera":
        return _case("camera", layers=rng.randint(1, 8), heads=rng.choice([8, 12, 16]), grid_h=0, grid_w=0,
                     budget=_log_int(rng, 16, 512), anchor_tokens=0, mode=rng.choice(["hybrid", "stored"]))
    dtype = rng.choice(["bf16"] * 4 + ["f32"]) if kind in ("step", "start", "host") else "bf16"
    heads = rng.randint(4, 16) if kind in ("step", "start", "host") else rng.choice([8, 12, 16])
    c = _case(kind, heads=heads, grid_h=rng.randint(8, 37), grid_w=rng.randint(8, 37), dtype=dtype,
              sigma=rng.choice([0.5, 0.75]), anchor_interval=rng.choice([4, 20, 100]))
    M = 5 + c["grid_h"] * c["grid_w"]
    c["anchor_tokens"] = rng.randint(0, min(256, M // 5))
    # the budget holds the first frame and three anchors at least, and a few frames as a rule
    c["budget"] = _log_int(rng, 2 * M, 32768 if dtype == "bf16" and kind in ("step", "host") else max(4 * M, 8192))
    if kind in ("step", "start"):
        c["mode"] = rng.choice(["hybrid"] * 4 + ["stored", "random", "qk"])
        c["layout"] = rng.choice(["holes"] * 4 + ["stable"])
    if kind == "start":
        c["frames"] = rng.randint(2, 10)
    if kind in ("stack", "aggregator"):
        c["layers"] = rng.randint(2, 24)
        c["budget"] = min(c["budget"], 12288)
    return c


def _tokens(c):
    return (1 if c["kind"] == "camera" else 5) + c["grid_h"] * c["grid_w"]


def _rand_frame(c, g, shape):
    """One frame's [q, k, v, resid] on the device."""
    dt = B.torch_dtype(DTYPES[c["dtype"]])
    x = torch.randn((4,) + shape, generator=g, device="cuda")
    gain = torch.randn(shape[:-1] + (1,), generator=g, device="cuda").mul_(c["sigma"]).exp_()
    x[3] *= gain
    return x.to(dt)


def _stream_config(c, seed):
    return gen.StreamConfig(name=c["kind"], n_layers=c["layers"], n_heads=c["heads"], grid_h=c["grid_h"],
                            grid_w=c["grid_w"], budget=c["budget"], anchor_tokens=c["anchor_tokens"],
                            min_anchor_interval=c["anchor_interval"], score_mode=MODES[c["mode"]],
                            dtype=DTYPES[c["dtype"]], gain_sigma=c["sigma"], seed=seed)


class _State:
    """What the program keeps between frames: the handle, a pool of input frames, the number of the next frame."""

    def __init__(self, c, seed):
        self.c = c
        self.t = 0
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        self.M, self.C = _tokens(c), 64 * c["heads"]

    def side_inputs(self, count):
        """Confidence map and coverage ratio of each pool frame."""
        n_p = self.M - 5
        self.conf = [torch.rand(n_p, generator=self.g, device="cuda") for _ in range(count)]
        self.rho = torch.rand(count, generator=self.g, device="cuda").tolist()


def prepare(case, seed):
    c, s = case, _State(case, seed)
    if c["kind"] == "camera":
        s.cache = B.OvggtCache.camera(n_layers=c["layers"], n_heads=c["heads"], budget=c["budget"],
                                      score_mode=MODES[c["mode"]], dtype=DTYPES[c["dtype"]])
        s.pool = [_rand_frame(c, s.g, (61, 1, s.C)) for _ in range(c["layers"])]
        s.out = [torch.empty_like(s.pool[0][0][0]) for _ in range(c["layers"])]
        s.anchors = []
        fill = c["budget"] + 2
    elif c["kind"] in ("stack", "aggregator"):
        cfg = _stream_config(c, seed)
        s.model = (H.ProjectionStack if c["kind"] == "stack" else H.Aggregator)(cfg, torch.device("cuda"))
        s.pool = [torch.randn((s.M, s.C), generator=s.g, device="cuda").to(torch.bfloat16) for _ in range(5)]
        s.side_inputs(5)
        if c["kind"] == "stack":
            s.resid = [_rand_frame(c, s.g, (s.M, s.C))[3].clone() for _ in range(c["layers"])]
        s.stream = torch.cuda.current_stream()
        fill = -(-c["budget"] // s.M) + 2
    else:
        s.cache = B.OvggtCache.from_stream(_stream_config(c, seed), compaction=LAYOUTS[c["layout"]])
        s.pool = [_rand_frame(c, s.g, (s.M, s.C)) for _ in range(7 if c["kind"] == "host" else 13)]
        s.side_inputs(len(s.pool))
        s.out = [torch.empty_like(s.pool[0][0]) for _ in range(c["frames"])]
        fill = -(-c["budget"] // s.M) + 2
        if c["kind"] == "host":
            s.pool = [p.cpu().pin_memory() for p in s.pool]        # one block [q | k | v | resid] a frame
            s.conf = [x.cpu().pin_memory() for x in s.conf]
            s.out = [torch.empty_like(s.pool[0][0]).pin_memory() for _ in range(2)]
        if c["kind"] == "start":
            fill = 1
    for _ in range(fill):          # the stream up to its steady state
        run(s)
    torch.cuda.synchronize()
    return s


def _camera_frame(s):
    """One token through the camera head's layers; its anchor flags follow the aggregator's decisions: here a
    registration every 100 frames, the oldest of four released."""
    i = s.t % 61
    registered, demoted = s.t > 0 and s.t % 100 == 0, -1
    if registered:
        s.anchors.append(s.t)
        if len(s.anchors) > 3:
            demoted = s.anchors.pop(0)
    for l, x in enumerate(s.pool):
        s.cache.layer_attend(l, s.t, x[0, i], x[1, i], x[2, i], out=s.out[l])
        s.cache.camera_compress(l, s.t, x[3, i], registered, demoted)
    s.t += 1
    return s.out


def run(state):
    s, kind = state, state.c["kind"]
    if kind == "camera":
        return _camera_frame(s)
    if kind == "start":
        s.cache.reset()
        for t in range(s.c["frames"]):
            x = s.pool[t]
            s.cache.layer_step(0, t, x[0], x[1], x[2], x[3], s.conf[t], s.rho[t], out=s.out[t])
        return s.out
    i = s.t % len(s.pool)
    x, t = s.pool[i], s.t
    s.t += 1
    if kind == "stack":
        return s.model.frame(t, x, s.resid, s.conf[i], s.rho[i], s.stream)
    if kind == "aggregator":
        return s.model.frame(t, x, s.conf[i], s.rho[i], s.stream)
    if kind == "host":
        out = s.out[t % 2]
        s.cache.layer_step_host(0, t, x[0], x[1], x[2], x[3], s.conf[i], s.rho[i], out)
        return out
    return s.cache.layer_step(0, t, x[0], x[1], x[2], x[3], s.conf[i], s.rho[i], out=s.out[0])


def _layer_work(c, M, C, n):
    """One layer, one frame, n rows cached before it: inputs, output and cache once; attention and key diversity."""
    e = 4 if c["dtype"] == "f32" else 2
    diversity = 4.0 * n * C if c["mode"] in ("hybrid", "qk") else 0.0
    return e * C * (4 * M + M + 2 * n + 2 * M), 4.0 * M * (n + M) * C + diversity + 2.0 * M * C


def work(case):
    c, M, C, L = case, _tokens(case), 64 * case["heads"], case["layers"]
    if c["kind"] == "start":
        per = [_layer_work(c, M, C, min(t * M, c["budget"])) for t in range(c["frames"])]
        return {"bytes": sum(p[0] for p in per), "flops": sum(p[1] for p in per)}
    b, f = _layer_work(c, M, C, c["budget"])
    b, f = b * L, f * L
    if c["kind"] == "stack":                  # QKV and output projections: 4 C^2 weights a layer
        b += L * 2 * 4 * C * C
        f += L * 2.0 * M * 4 * C * C
    if c["kind"] == "aggregator":             # two blocks a layer with 12 C^2 weights each, and the frame attention
        b += L * 2 * (24 * C * C)
        f += L * (2.0 * M * 24 * C * C + 4.0 * M * M * C)
    return {"bytes": b, "flops": f}


def tolerance(case):
    # bf16: probabilities and outputs are rounded to 8 bits.  fp32: sums of up to some ten thousand terms.
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2}
