"""The work that is measured: what a program that tracks with this library has it do, through its public calls.

Three kinds of call:
  frames  one session tracks depth frames (trk_track_frame from host memory, one frame per pass, or
          trk_track_frame_device over a clip that is on the device already, read back at its end);
  group   many sessions step together (a fused batch, a schedule of batches, or the frame server fed from
          host memory), every session's results read back;
  rows    the contraction [J r]^T [J r] of a caller's own residual rows on its device buffers.

A tracking pass carries on from the state the last one left, as a live loop does: the frames of a short clip
are taken forwards, then backwards, so the motion between two passes is always one frame's.  The "acquire"
pass starts over each time (trk_set_pose, then the frame), as a program does that (re)finds its subject.
"""
import functools

import numpy as np
import torch

from paper_1711_07999_gb300 import synth, trk

PRECISIONS = {"fp32": trk.PRECISION_FP32, "bf16x3": trk.PRECISION_BF16X3, "tf32x3": trk.PRECISION_TF32X3}
FPS = 30.0


def _frames(name, how, config, V, width, height, **over):
    c = dict(name=name, kind="frames", how=how, config=config, V=V, width=width, height=height, clip=4,
             precision="fp32", association=0, shape_solver=0, shape_sweeps=1, pose_iters=10, shape_iters=2)
    c.update(over)
    return c


def _group(name, how, sessions, config, V, width, height, **over):
    c = dict(name=name, kind="group", how=how, sessions=sessions, first=0, config=config, V=V, width=width,
             height=height, clip=2, precision="fp32", association=0)
    c.update(over)
    return c


def _rows(name, how, n, nc, ld):
    return dict(name=name, kind="rows", how=how, n=n, nc=nc, ld=ld)


def listed():
    return [
        # a small model found in one 160x120 image from a pose 10 degrees off per joint: the smallest frame there
        # is, launches and latency
        _frames("acquire_5k_160x120", "acquire", 1, 5000, 160, 120, clip=1),
        # one live camera: the 50k-vertex humanoid at 640x480, host depth in, joints and offsets out
        _frames("live_50k_640x480", "live", 2, 50000, 640, 480),
        # the high-resolution stream, its normal equations on the tensor cores
        _frames("live_200k_1280x720_tf32x3", "live", 3, 200000, 1280, 720, precision="tf32x3"),
        # the template size and camera of the paper, with the O(1) association and the coupled shape solve
        _frames("live_55k_512x424_rid_pcg", "live", 2, 55474, 512, 424, association=1, shape_solver=1, shape_sweeps=8),
        # a recorded clip that is on the device already, tracked offline: odd sizes, split-BF16 normal equations
        _frames("clip_17k_357x269_bf16x3", "clip", 2, 17000, 357, 269, precision="bf16x3", clip=6),
        # sixteen equal cameras in step: a fused batch over device depth, four frames between two readings
        _group("batch_16x50k_640x480", "batch", 16, 2, 50000, 640, 480, clip=4),
        # sessions of uneven size (5k-200k vertices, 12-40 bones, 320x240 to 1280x720): a fused batch
        _group("batch_8_uneven", "batch", 8, 4, 0, 0, 0, clip=4),
        # twelve small cameras under a schedule of two concurrent groups
        _group("schedule_12x9k_320x240", "schedule", 12, 2, 9000, 320, 240, clip=4),
        # the frame server: twelve streams of mixed sizes submit host depth and collect their results
        _group("serve_12_mixed", "serve", 12, 2, 12000, 320, 240),
        # a caller's own rows: a small problem without allocation, a large one in FP32, a session-sized one
        # on the tensor cores
        _rows("rows_3k_x31_noalloc", "noalloc", 3001, 31, 31),
        _rows("rows_1m_x73", "fp32", 1_000_003, 73, 76),
        _rows("rows_50k_x56_bf16x3", "bf16x3", 50010, 56, 56),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["frames", "frames", "group", "rows"])
    if kind == "rows":
        nc = rng.randint(1, 80)
        return {k: v for k, v in _rows("", rng.choice(["fp32", "noalloc", "bf16x3", "tf32x3"]),
                                       _log_uniform(rng, 500, 1_000_000), nc, nc + rng.choice([0, 0, 1, 4, 7])).items()
                if k != "name"}
    width = _log_uniform(rng, 120, 1280)
    height = max(90, min(720, int(width * rng.choice([0.75, 0.5625, 0.83]))))
    precision = rng.choice(["fp32", "fp32", "tf32x3", "bf16x3"])
    if kind == "frames":
        solver = rng.choice([0, 0, 1])
        c = _frames("", rng.choice(["live", "clip", "acquire"]), 2, _log_uniform(rng, 3000, 200000), width, height,
                    precision=precision, association=rng.choice([0, 0, 1]), shape_solver=solver,
                    shape_sweeps=rng.randint(4, 10) if solver else rng.choice([1, 1, 3]),
                    pose_iters=rng.randint(8, 15), clip=rng.randint(2, 4))
        if c["how"] == "acquire":
            c.update(config=1, V=min(c["V"], 60000), clip=1)
    else:
        n = rng.randint(2, 12)
        c = _group("", rng.choice(["batch", "schedule", "serve"]), n, rng.choice([2, 4]),
                   min(_log_uniform(rng, 3000, 60000), 400000 // n), width, height, precision=precision,
                   association=rng.choice([0, 0, 1]))
        c["first"] = rng.randint(0, 50)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=32)
def _template(config, session, V, width, height, **over):
    """The template a program loads once: mesh, weights, skeleton, camera and parameters."""
    if not V:  # the size class of the uneven batch
        return synth.make_model(4, session=session, **over)
    return synth.make_model(config, session=session, V=V, width=width, height=height, **over)


def _models(case):
    over = dict(precision=PRECISIONS[case["precision"]], association=case["association"])
    if case["kind"] == "frames":
        over.update(shape_solver=case["shape_solver"], shape_sweeps=case["shape_sweeps"],
                    pose_iters=case["pose_iters"], shape_iters=case["shape_iters"])
        return [_template(case["config"], 0, case["V"], case["width"], case["height"], **over)]
    if case["config"] == 4 and not case["V"]:
        return [_template(4, case["first"] + k, 0, 0, 0, **over) for k in range(case["sessions"])]
    if case["how"] == "serve":  # mixed sizes: three model sizes, two cameras
        return [_template(case["config"], case["first"] if case["config"] == 2 else case["first"] + k,
                          case["V"] * (2 + k % 3) // 3, case["width"] * (1 + k % 2), case["height"] * (1 + k % 2), **over)
                for k in range(case["sessions"])]
    return [_template(case["config"], case["first"] if case["config"] == 2 else case["first"] + k, case["V"],
                      case["width"], case["height"], **over) for k in range(case["sessions"])]


def _sensor(depth, config, gen):
    """A rendered depth image as a camera delivers it: noise growing with depth and dropped pixels (or a static
    scene's noise, quantised to 1 mm), 0 where nothing returns."""
    d = torch.from_numpy(depth).cuda()
    hit = d > 0
    noise = torch.randn(d.shape, generator=gen, device="cuda")
    if config == 1:
        d = torch.where(hit, torch.round((d + 0.001 * noise) * 1000) / 1000, torch.zeros_like(d))
    else:
        d = torch.where(hit, d + noise * 0.0015 * (d / 3) ** 2, torch.zeros_like(d))
        d[torch.rand(d.shape, generator=gen, device="cuda") < 0.02] = 0
    return d.clamp_(min=0).contiguous()


def _start(session, model, case, seed, k):
    """The session's clip of depth frames (device tensors) and its start: the pose and offsets before the first."""
    gen = torch.Generator(device="cuda").manual_seed(1000 * seed + k)
    rng = np.random.default_rng([seed, k])
    config = model["motion"]["config"]
    t0 = float(rng.uniform(0, 8))
    clip = []
    for f in range(case["clip"]):
        t = t0 + f / FPS
        clip.append(_sensor(session.render_depth(synth.gt_theta(model, t), synth.gt_offsets(model, t)), config, gen))
    theta = synth.gt_theta(model, t0)
    if config == 1:  # found from a pose up to 10 degrees off at each hinge
        theta = theta + model["motion"]["start_pert"] * rng.uniform(0.5, 1.0, len(theta))
    session.set_pose(theta)
    return clip, theta


def prepare(case, seed):
    if case["kind"] == "rows":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        # Jacobian entries of very different sizes, most of a row zero (the links above its bones), the residual last
        scale = 0.01 + torch.rand(case["nc"], generator=gen, device="cuda")
        rows = torch.randn((case["n"], case["ld"]), generator=gen, device="cuda")
        rows[:, :case["nc"]] *= scale
        rows[:, :max(case["nc"] - 1, 0)] *= torch.rand((case["n"], max(case["nc"] - 1, 0)), generator=gen, device="cuda") < 0.4
        return dict(case=case, rows=rows, out=torch.empty((case["nc"], case["nc"]), dtype=torch.float64, device="cuda"))
    models = _models(case)
    sessions = [trk.Session(m) for m in models]
    made = [_start(s, m, case, seed, k) for k, (s, m) in enumerate(zip(sessions, models))]
    st = dict(case=case, sessions=sessions, pos=0, step=1, start=made[0][1])
    if case["how"] in ("clip", "batch", "schedule"):
        st["clips"] = [c for c, _ in made]
    else:
        st["clips"] = [[d.cpu().numpy() for d in c] for c, _ in made]
    st["stream"] = torch.cuda.Stream()
    if case["how"] == "batch":
        st["batch"] = trk.Batch(sessions)
    elif case["how"] == "schedule":
        st["schedule"] = trk.Schedule(sessions, config=dict(groups=2, assoc_blocks=608, tail_blocks=304))
    elif case["how"] == "serve":
        st["server"] = trk.Server(8 * sum(s.info()["device_bytes"] for s in sessions) + (1 << 30),
                                  max_inflight=len(sessions))
        for s in sessions:
            st["server"].attach(s)
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------------------
def _next(st):
    """The index of the next frame of the clip: forwards, then backwards."""
    f, n = st["pos"], st["case"]["clip"]
    if n > 1:
        if not 0 <= f + st["step"] < n:
            st["step"] = -st["step"]
        st["pos"] = f + st["step"]
    return f


def _together(results):
    return dict(theta=[r["theta"] for r in results], offsets=[r["offsets"] for r in results],
                energy=[r["energy"] for r in results],
                counts=[np.array([[r["n_assoc_px"], r["n_assoc_verts"]] for r in results])])


def run(st):
    case = st["case"]
    if case["kind"] == "rows":
        args = (st["rows"].data_ptr(), case["n"], case["nc"], case["ld"])
        if case["how"] == "fp32":
            trk.jtj_rows(*args, st["out"].data_ptr())
        elif case["how"] == "noalloc":
            trk.jtj_rows_noalloc(*args, st["out"].data_ptr())
        else:
            trk.jtj_rows_tc(*args, PRECISIONS[case["how"]], st["out"].data_ptr())
        return st["out"]
    sessions, clips = st["sessions"], st["clips"]
    if case["how"] == "acquire":
        sessions[0].set_pose(st["start"])
        return sessions[0].track_frame(clips[0][0])
    if case["how"] == "live":
        return sessions[0].track_frame(clips[0][_next(st)])
    if case["how"] == "clip":
        for _ in range(case["clip"]):
            sessions[0].track_frame_device(clips[0][_next(st)].data_ptr(), st["stream"].cuda_stream)
        return sessions[0].read_result()
    if case["how"] == "serve":
        tickets = []
        for _ in range(case["clip"]):
            f = _next(st)
            tickets.append([st["server"].submit(s, c[f]) for s, c in zip(sessions, clips)])
        for waiting in tickets:  # every stream's frames, in order; the last one's results are the pass's
            results = [st["server"].wait(s, t) for s, t in zip(sessions, waiting)]
        return _together(results)
    many = st["batch"] if case["how"] == "batch" else st["schedule"]
    for _ in range(case["clip"]):
        f = _next(st)
        many.track_device([c[f].data_ptr() for c in clips], st["stream"].cuda_stream)
    return _together([s.read_result() for s in sessions])


# ---------------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------------------
def _frame_work(model, case):
    V, F = len(model["mesh"]["verts"]), len(model["mesh"]["tris"])
    npx = model["camera"]["width"] * model["camera"]["height"]
    P, n = len(model["skeleton"]["parent"]), len(model["skeleton"]["parent"]) + 1
    pose, shape = model["params"]["pose_iters"], model["params"]["shape_iters"]
    rows, px = V / 3, npx / 12  # about a third of the vertices collect a pixel; the body fills about a twelfth of the image
    # per vertex: positions, weights and bones, four neighbours, offsets in and out; per triangle its corners
    per_frame = V * (12 + 16 + 4 + 16 + 2 * 12) + 12 * F + 4 * npx
    per_iter = V * 160 + F * 60 + px * 9 * 9
    per_pose = rows * (n * (n + 1) + 12 * P) + 6 * (P ** 3 / 3 + 2 * P * P) + 2 * rows * 110
    return per_frame, (pose + shape) * per_iter + pose * per_pose + shape * V * 120


def work(case):
    if case["kind"] == "rows":
        n, nc = case["n"], case["nc"]
        return {"bytes": 4 * n * nc + 8 * nc * nc, "flops": n * nc * (nc + 1)}
    frames = case["clip"] if case["how"] not in ("live", "acquire") else 1
    each = [_frame_work(m, case) for m in _models(case)]
    return {"bytes": frames * sum(b for b, _ in each), "flops": frames * sum(f for _, f in each)}


def exact(case, seed):
    # A tracked frame has no value of its own in 64 bits: its correspondences are an argmin whose ties rounding
    # decides, and each later iteration starts from what was chosen.
    if case["kind"] != "rows":
        return None
    st = prepare(case, seed)
    x = st["rows"][:, :case["nc"]].double()
    return x.T @ x
