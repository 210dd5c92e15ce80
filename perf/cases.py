"""The measured work of this framework: what a program that tracks a depth camera, builds its map and trains
and runs the learned proposal has the library do, through its public calls.

Six kinds of call, each over the range it is used in (frames of 80 x 60 to 640 x 480, maps of 64^3 to 512^3 voxels
in the three storage types, 256 to 20,000 particles):

  track     one frame of Algorithm 1 (pfo_track_frame_ex_async) against a map fused at known poses
  sequence  the online loop: a map started at frame 0, then frames from pinned host memory, a host pose for each
  batch     several uneven sequences stepped together (rf_batch_*), as a CUDA graph
  fitness   fitness_eval: scoring a swarm on a frame's overlap points
  fuse      a map rebuilt from posed frames (reset, tsdf_integrate_dev per frame), then scored or exported
  propose   the learned proposal of one frame: features, network, (c_0, r_0)
  train     one batch of the proposal network's training: forward, loss, backward

The scenes, trajectories and depth noise are those of paper_2105_05600_gb300.synth; the seed picks the room, the
path, the noise, the template and the network.
"""
import math

import numpy as np
import torch

from paper_2105_05600_gb300 import _native as nat
from paper_2105_05600_gb300 import synth

ROOM = 5.12          # metres, the extent of the 512^3 map at 1 cm voxels
SMALL_ROOM = 2.56    # metres, the extent of the 64^3 map at 4 cm voxels
R_FIRST = [0.05, 0.05, 0.05, 0.15, 0.15, 0.15]  # axis lengths of a first frame
MAP_FRAMES = 6       # frames fused into the map before the frame that is tracked or scored
FLAGS = {"default": 0, "l1": nat.RF_L1, "nearest": nat.RF_NEAREST, "right_mult": nat.RF_RIGHT_MULT}


def listed():
    return [
        # the smallest frame: the 64^3 workload, where the iteration's fixed cost counts
        dict(name="track_tiny", kind="track", dims=64, dtype="f32", width=80, height=60, stride=1, n=1024, k_max=10,
             speed=3.0),
        # the short run that refines a learned proposal (10,000 particles, at most 5 iterations)
        dict(name="track_short", kind="track", dims=512, dtype="i16", width=640, height=480, stride=4, n=10000,
             k_max=5, speed=4.0),
        # the paper-scale frame: 20,000 particles, 160 x 120 points, up to 20 iterations
        dict(name="track_paper", kind="track", dims=512, dtype="i16", width=640, height=480, stride=4, n=20000,
             k_max=20, speed=3.0),
        # the online loop of a live camera with the multi-resolution schedule: tracking, fusion and the copies
        dict(name="sequence_multires", kind="sequence", dims=512, dtype="i16", width=640, height=480, frames=4,
             levels="1024:3,3072:4,10240:6", k_max=20, speed=1.68),
        # offline processing of several recordings at once, uneven in frame size, map size and swarm
        dict(name="batch_uneven", kind="batch", dtype="i16", k_max=20, speed=3.0,
             specs="80x60:256:10240,160x120:384:17111,120x90:256:20000,200x150:512:12345"),
        # one swarm of a few hundred particles on a small frame: the smallest scoring call, ragged sizes
        dict(name="fitness_small", kind="fitness", dims=64, dtype="f16", width=61, height=45, stride=2, n=257,
             flags="default", spread=1.0),
        # the paper-scale swarm and frame in half storage
        dict(name="fitness_paper_f16", kind="fitness", dims=512, dtype="f16", width=640, height=480, stride=4,
             n=20000, flags="default", spread=1.0),
        # a float map, odd sizes throughout
        dict(name="fitness_f32_odd", kind="fitness", dims=328, dtype="f32", width=321, height=243, stride=3, n=9973,
             flags="default", spread=0.5),
        # a map rebuilt at paper scale from posed frames and scored at the last pose
        dict(name="fuse_paper", kind="fuse", dx=512, dy=512, dz=512, dtype="i16", width=640, height=480, frames=8,
             export=False, speed=3.0),
        # a small non-cubic float map rebuilt from a window of keyframes and exported to the host
        dict(name="fuse_export_f32", kind="fuse", dx=128, dy=96, dz=112, dtype="f32", width=161, height=119,
             frames=48, export=True, speed=1.68),
        # the learned proposal's latency per frame
        dict(name="propose", kind="propose", width=640, height=480, speed=4.0),
        # the training batch of the proposal network
        dict(name="train_512", kind="train", batch=512, rows=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _frame(rng, lo=60, hi=640):
    w = _log_int(rng, lo, hi)
    return w, max(45, int(w * rng.choice([0.75, 0.5625, 0.7])))


def _stride(w, h, most):
    s = 1
    while -(-w // s) * -(-h // s) > most:
        s += 1
    return s


def draw(rng):
    kind = rng.choice(["track", "track", "sequence", "batch", "fitness", "fitness", "fuse", "fuse", "propose", "train"])
    dtype = rng.choice(["i16", "i16", "f16", "f32"])
    dims = 8 * _log_int(rng, 8, 64)
    speed = round(rng.uniform(1.0, 4.0), 2)
    w, h = _frame(rng)
    if kind == "track":
        n, k = _log_int(rng, 500, 20000), rng.randint(3, 20)
        return dict(kind=kind, dims=dims, dtype=dtype, width=w, height=h, stride=_stride(w, h, rng.randint(2000, 19200)),
                    n=n, k_max=k, speed=speed)
    if kind == "sequence":
        a = _log_int(rng, 600, 2000)
        s = _stride(w, h, 30000)
        return dict(kind=kind, dims=dims, dtype=dtype, width=w, height=h, frames=rng.randint(2, 5),
                    levels="%d:%d,%d:%d,%d:%d" % (a, s, 3 * a, s + 1, 5 * a, s + 3), k_max=rng.randint(6, 20), speed=speed)
    if kind == "batch":
        specs = []
        for _ in range(rng.randint(2, 4)):
            bw, bh = _frame(rng, 60, 200)
            specs.append("%dx%d:%d:%d" % (bw, bh, 8 * _log_int(rng, 16, 48), _log_int(rng, 2000, 17000)))
        return dict(kind=kind, dtype=dtype, k_max=rng.randint(5, 20), speed=speed, specs=",".join(specs))
    if kind == "fitness":
        return dict(kind=kind, dims=dims, dtype=dtype, width=w, height=h, stride=_stride(w, h, rng.randint(500, 19200)),
                    n=_log_int(rng, 200, 20000), flags=rng.choice(["default", "default", "l1", "nearest", "right_mult"]),
                    spread=round(rng.uniform(0.05, 2.0), 3))
    if kind == "fuse":
        export = rng.random() < 0.5
        top = 128 if export else 512
        d = [8 * _log_int(rng, 8, top // 8)] * 3
        if export:  # odd boxes: each side at least 0.6 of the longest
            d = [8 * max(8, int(d[0] // 8 * rng.uniform(0.6, 1.0))) for _ in range(2)] + [d[0]]
            rng.shuffle(d)
        return dict(kind=kind, dx=d[0], dy=d[1], dz=d[2], dtype=dtype, width=w, height=h,
                    frames=rng.randint(4, 32) if export else rng.randint(2, 10), export=export, speed=speed)
    if kind == "propose":
        return dict(kind=kind, width=w, height=h, speed=speed)
    return dict(kind="train", batch=8 * _log_int(rng, 8, 128), rows=_log_int(rng, 1500, 50000))


# ----------------------------------------------------------------------------------------------- inputs
def _scene(extent, seed, frames, width, height, speed):
    """A room, a path through it, the camera and the path's noisy depth frames (on the GPU)."""
    scene = synth.make_scene(extent, 0.30 if extent < 4.0 else 0.20, seed)
    traj = synth.make_trajectory(scene, frames, speed, 0.75 * speed, seed)
    K = synth.intrinsics(width, height)
    depth = synth.render_depth_batch(scene, traj, K, seed=1000 + seed)
    poses = torch.from_numpy(traj.astype(np.float32)).cuda()
    return K, depth, poses


def _extent(dims):
    return SMALL_ROOM if dims <= 96 else ROOM


def _voxel(dims):
    return _extent(dims) / dims


def _trunc(dims):
    return (3 if dims <= 96 else 6) * _voxel(dims)


def _map_inputs(case, seed):
    return _scene(_extent(case["dims"]), seed, MAP_FRAMES + 1, case["width"], case["height"], case.get("speed", 3.0))


def _map(case, K, depth, poses):
    vol = nat.Volume(case["dims"], _voxel(case["dims"]), _trunc(case["dims"]), (0, 0, 0), case["dtype"])
    for f in range(MAP_FRAMES):
        nat.tsdf_integrate_dev(vol, depth[f], K, poses[f])
    return vol


def _levels(case):
    return [[int(v) for v in part.split(":")] for part in case["levels"].split(",")]


def _specs(case):
    got = []
    for part in case["specs"].split(","):
        size, dims, n = part.split(":")
        w, h = size.split("x")
        got.append(dict(width=int(w), height=int(h), dims=int(dims), n=int(n)))
    return got


def _network_inputs(rows, seed):
    """Network parameters (He-scaled hidden layers, a small output layer) and a dataset with the proposal's statistics."""
    g = torch.Generator(device="cuda")
    g.manual_seed(7000 + seed)
    theta, shapes = [], [(256, 832), (256, 256), (256, 256), (16, 256)]
    for l, (o, i) in enumerate(shapes):
        W = torch.randn(o, i, generator=g, device="cuda") * (math.sqrt(2.0 / i) if l < 3 else 0.05)
        b = torch.randn(o, generator=g, device="cuda") * 0.02
        if l == 0:
            W[:, 774:] = 0
        if l == 3:
            W[12:], b[12:] = 0, 0
        theta += [W.reshape(-1), b]
    x = torch.zeros(rows, 832, device="cuda")
    x[:, :768] = (torch.randn(rows, 768, generator=g, device="cuda") * 0.7).clamp(-8, 8)
    x[:, 768:774] = torch.randn(rows, 6, generator=g, device="cuda")
    y = x[:, 768:774] + 0.5 * torch.randn(rows, 6, generator=g, device="cuda")
    return torch.cat(theta), x.to(torch.bfloat16), y.contiguous(), g


def _row_floats(stats):
    """The float fields of the first iteration's row of a frame-statistics buffer, as a view."""
    off = nat.rf_frame_stats.it.offset + nat.rf_iter_stats.rho_ref.offset
    end = nat.rf_frame_stats.it.offset + nat.rf_iter_stats.offset.offset + nat.rf_iter_stats.offset.size
    return stats[off:end].view(torch.float32)


# ---------------------------------------------------------------------------------------------- prepare
def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed % 100003)


def run(state):
    return state["run"](state)


def _prepare_track(case, seed):
    K, depth, poses = _map_inputs(case, seed)
    vol = _map(case, K, depth, poses)
    pst = nat.pst_create(case["n"], seed=1 + seed)
    tr = nat.Tracker(vol, pst, nat.make_params(k_max=case["k_max"], stride=case["stride"]), case["width"], case["height"])
    stats = nat.new_stats_buffer()
    return dict(run=_run_track, K=K, tr=tr, depth=depth[MAP_FRAMES], prev=depth[MAP_FRAMES - 1], pose=poses[MAP_FRAMES - 1],
                out=torch.zeros(7, device="cuda"), r0=torch.tensor(R_FIRST, device="cuda"),
                r=torch.zeros(6, device="cuda"), stats=stats, row=_row_floats(stats))


def _run_track(s):
    s["r"].copy_(s["r0"])
    nat.pfo_track_frame_ex_async(s["tr"], s["depth"], s["prev"], s["K"], s["pose"], s["out"], s["stats"],
                                 scale_dev=s["r"])
    return dict(pose=s["out"], r1=s["r"], first=s["row"])


def _prepare_sequence(case, seed):
    K, depth, poses = _scene(_extent(case["dims"]), seed, case["frames"] + 1, case["width"], case["height"], case["speed"])
    vol = nat.Volume(case["dims"], _voxel(case["dims"]), _trunc(case["dims"]), (0, 0, 0), case["dtype"])
    levels = _levels(case)
    pst = nat.pst_create(max(n for n, _ in levels), seed=1 + seed)
    tr = nat.Tracker(vol, pst, nat.make_params(k_max=case["k_max"], stride=levels[0][1]), case["width"], case["height"])
    tr.set_schedule([n for n, _ in levels], [t for _, t in levels])
    host = [d.cpu().pin_memory() for d in depth]
    return dict(run=_run_sequence, K=K, vol=vol, tr=tr, host=host, pose0=poses[0].cpu().numpy())


def _run_sequence(s):
    s["vol"].reset()
    s["tr"].set_scale(R_FIRST)
    nat.rf_sequence_start(s["tr"], s["host"][0], s["K"], s["pose0"])
    return [nat.rf_sequence_step(s["tr"], d, s["K"])[0] for d in s["host"][1:]]


def _prepare_batch(case, seed):
    vols, trs, Ks, frames, start = [], [], [], [], []
    for i, p in enumerate(_specs(case)):
        K, depth, poses = _scene(ROOM, seed + 11 * i, 3, p["width"], p["height"], case["speed"])
        vol = nat.Volume(p["dims"], ROOM / p["dims"], 6 * ROOM / p["dims"], (0, 0, 0), case["dtype"])
        pst = nat.pst_create(p["n"], seed=1 + seed + i)
        trs.append(nat.Tracker(vol, pst, nat.make_params(k_max=case["k_max"]), p["width"], p["height"]))
        vols.append(vol)
        Ks.append(K)
        frames.append(depth)
        start.append(poses[0].cpu().numpy())
    b = nat.Batch(trs, Ks)
    slots = [[b.depth_slot(i, q) for q in (0, 1)] for i in range(len(trs))]
    rings = [[b.pose_dev(i, q) for i in range(len(trs))] for q in (0, 1)]
    return dict(run=_run_batch, b=b, vols=vols, trs=trs, frames=frames, start=start, slots=slots, rings=rings,
                out=torch.zeros(2, len(trs), 7, device="cuda"))


def _run_batch(s):
    for v, t in zip(s["vols"], s["trs"]):
        v.reset()
        t.set_scale(R_FIRST)
    for slot, d in zip(s["slots"], s["frames"]):
        slot[0].copy_(d[0])
        slot[1].copy_(d[1])
    s["b"].start(s["start"])
    s["b"].step(1, use_graph=True)
    torch.stack(s["rings"][1], out=s["out"][0])  # the rings belong to the trackers: a path is kept in the program's own memory
    for slot, d in zip(s["slots"], s["frames"]):
        slot[0].copy_(d[2])
    s["b"].step(0, use_graph=True)
    torch.stack(s["rings"][0], out=s["out"][1])
    return s["out"]


def _fitness_scale(case):
    return [0.03 * case["spread"]] * 3 + [0.05 * case["spread"]] * 3


def _prepare_fitness(case, seed):
    K, depth, poses = _map_inputs(case, seed)
    vol = _map(case, K, depth, poses)
    cur, prev = poses[MAP_FRAMES].cpu().numpy(), poses[MAP_FRAMES - 1].cpu().numpy()
    pts = nat.rf_depth_to_points(depth[MAP_FRAMES], K, case["stride"])
    mask, _ = nat.rf_overlap_mask(pts, depth[MAP_FRAMES - 1], K, cur, prev, math.sqrt(3.0) * _voxel(case["dims"]))
    pts = pts[mask.bool()].contiguous()
    if pts.shape[0] == 0:  # a view without overlap: score every valid point
        pts = nat.rf_depth_to_points(depth[MAP_FRAMES], K, case["stride"])
    return dict(run=_run_fitness, vol=vol, pts=pts, pst=nat.pst_create(case["n"], seed=1 + seed), centre=cur,
                scale=_fitness_scale(case), params=nat.make_params(flags=nat.RF_DEFAULT_FLAGS | FLAGS[case["flags"]]))


def _run_fitness(s):
    rho, S, valid = nat.fitness_eval(s["vol"], s["pts"], s["pst"], s["centre"], s["scale"], s["params"])
    return dict(rho=rho, sumsq=S, valid=valid)


def _fuse_geometry(case):
    """Dims, room extent, voxel and the origin that centres the map in the room."""
    dims = (case["dx"], case["dy"], case["dz"])
    extent = ROOM if max(dims) > 96 else SMALL_ROOM
    voxel = extent / max(dims)
    return dims, extent, voxel, [0.5 * (extent - d * voxel) for d in dims]


def _prepare_fuse(case, seed):
    dims, extent, voxel, origin = _fuse_geometry(case)
    K, depth, poses = _scene(extent, seed, case["frames"], case["width"], case["height"], case["speed"])
    vol = nat.Volume(dims, voxel, 4 * voxel, origin, case["dtype"])
    s = dict(run=_run_export if case["export"] else _run_fuse, K=K, vol=vol, depth=depth, poses=poses)
    if not case["export"]:
        pts = nat.rf_depth_to_points(depth[-1], K, _stride(case["width"], case["height"], 20000))
        s.update(pts=pts[pts[:, 3] > 0].contiguous(), pst=nat.pst_create(256, seed=1 + seed),
                 centre=poses[-1].cpu().numpy(), params=nat.make_params())
    return s


def _fuse_frames(s):
    s["vol"].reset()
    for d, p in zip(s["depth"], s["poses"]):
        nat.tsdf_integrate_dev(s["vol"], d, s["K"], p)


def _run_fuse(s):
    _fuse_frames(s)
    rho, S, valid = nat.fitness_eval(s["vol"], s["pts"], s["pst"], s["centre"], [0.03] * 3 + [0.05] * 3, s["params"])
    return dict(rho=rho, sumsq=S, valid=valid)


def _run_export(s):
    _fuse_frames(s)
    values, weights = s["vol"].download()
    return dict(values=values, weights=weights)


def _propose_inputs(case, seed):
    K, depth, poses = _scene(ROOM, seed, 3, case["width"], case["height"], case["speed"])
    theta, _, _, _ = _network_inputs(8, seed)
    return K, depth, poses, theta


def _prepare_propose(case, seed):
    K, depth, poses, theta = _propose_inputs(case, seed)
    net = nat.MLP(8)
    net.set_params(theta.cpu().numpy())
    return dict(run=_run_propose, K=K, depth=depth, poses=poses, net=net, params=nat.proposal_params())


def _run_propose(s):
    x = nat.rf_proposal_features(s["depth"][2], s["depth"][1], s["K"], s["poses"][0], s["poses"][1])
    o = s["net"].forward(x.view(1, -1))
    c0, r0 = nat.rf_proposal_apply(o, x, s["poses"][1], s["params"])
    return dict(x=x, o=o, c0=c0, r0=r0)


def _train_inputs(case, seed):
    theta, x, y, g = _network_inputs(case["rows"], seed)
    idx = torch.randint(0, case["rows"], (case["batch"],), generator=g, device="cuda", dtype=torch.int32)
    return theta, x, y, idx


def _prepare_train(case, seed):
    theta, x, y, idx = _train_inputs(case, seed)
    net = nat.MLP(case["batch"])
    net.set_params(theta.cpu().numpy())
    return dict(run=_run_train, net=net, x=x, y=y, idx=idx, batch=case["batch"])


def _run_train(s):
    grad, loss, out = s["net"].gradient(s["x"], s["y"], s["batch"], s["idx"])
    return dict(grad=grad, loss=loss, out=out)


# ------------------------------------------------------------------------------------- work and tolerance
_BYTES = {"i16": 2, "f16": 2, "f32": 4}
_LOOKUP_FLOPS = 47  # transform 18, floor and fraction 6, eight-corner interpolation 21, square and sum 2


def _points(w, h, stride):
    return -(-w // stride) * -(-h // stride)


def _score_work(n, m, es):
    """One swarm on one frame: points and template read once, each point's cell at least once, three results a particle."""
    return dict(bytes=16 * m + 8 * es * m + 24 * n + 16 * n, flops=float(n) * m * _LOOKUP_FLOPS)


def _fuse_bytes(case, voxels, frames):
    """A frame's voxels: about a seventh of a paper-scale map is in view; value and weight read and written, depth read."""
    return frames * (0.14 * voxels * 2 * (_BYTES[case["dtype"]] + 1) + 4 * case["width"] * case["height"])


def work(case):
    kind = case["kind"]
    if kind in ("track", "fitness"):
        m = _points(case["width"], case["height"], case["stride"])
        one = _score_work(case["n"], m, _BYTES[case["dtype"]])
        if kind == "fitness":
            return one
        return dict(bytes=one["bytes"] + 8 * case["width"] * case["height"], flops=case["k_max"] * one["flops"])
    if kind == "sequence":
        each = [n * _points(case["width"], case["height"], t) for n, t in _levels(case)]
        lookups = sum(each[k % len(each)] for k in range(case["k_max"])) * case["frames"]
        frame = 4 * case["width"] * case["height"]
        return dict(bytes=case["dims"] ** 3 * (9 * _BYTES[case["dtype"]] + 1) + (case["frames"] + 1) * 2 * frame
                    + _fuse_bytes(case, case["dims"] ** 3, case["frames"] + 1), flops=float(lookups) * _LOOKUP_FLOPS)
    if kind == "batch":
        got = dict(bytes=0.0, flops=0.0)
        for p in _specs(case):
            one = _score_work(p["n"], p["width"] * p["height"], _BYTES[case["dtype"]])
            got["bytes"] += 2 * one["bytes"] + p["dims"] ** 3 * (9 * _BYTES[case["dtype"]] + 1)
            got["bytes"] += _fuse_bytes(dict(case, **p), p["dims"] ** 3, 3)
            got["flops"] += 2 * case["k_max"] * one["flops"]
        return got
    if kind == "fuse":
        voxels, es = case["dx"] * case["dy"] * case["dz"], _BYTES[case["dtype"]]
        # the reset writes values, weights and the eight corners of every cell; the read-out reads the map once more
        b = voxels * (9 * es + 1) + _fuse_bytes(case, voxels, case["frames"])
        if case["export"]:
            return dict(bytes=b + voxels * (es + 1), flops=30.0 * 0.14 * voxels * case["frames"])
        one = _score_work(256, min(20000, case["width"] * case["height"]), es)
        return dict(bytes=b + one["bytes"], flops=30.0 * 0.14 * voxels * case["frames"] + one["flops"])
    macs = 832 * 256 + 2 * 256 * 256 + 256 * 16
    if kind == "propose":
        return dict(bytes=8 * case["width"] * case["height"] + 2 * macs, flops=2.0 * macs + 4 * case["width"] * case["height"])
    return dict(bytes=2 * macs + 4 * macs + case["batch"] * (2 * 832 + 24 + 64), flops=2.0 * case["batch"] * (3 * macs - 832 * 256))


def tolerance(case):
    kind = case["kind"]
    if kind in ("track", "sequence", "batch"):
        # whole runs of Algorithm 1: a difference in the last bit of one fitness changes which particles beat the
        # threshold by a hair, and up to 20 iterations a frame carry that into the pose, each frame into the next.
        # Sums in other orders (three work splits and lookup groups): up to 7e-5 on one frame, 2.4e-3 on sequences
        return dict(rel=4e-4, max=0.02) if kind == "track" else dict(rel=0.01, max=0.05)
    if kind == "fitness":
        # FP32 sums of up to 19,200 terms, and samples on the edge between a known and an unknown cell that may count
        # either way: up to 9e-5 from 64 bits
        return dict(rel=3e-4, max=2e-2, differ=0.01)
    if kind == "fuse":
        # a voxel whose pixel or truncation decision lies within FP32 rounding may go either way: 5e-5 from 64 bits
        return dict(rel=2e-4, max=0.05, differ=1e-3)
    return dict(rel=4e-3, max=0.2, differ=0.01)  # bfloat16 activations and gradients: up to 8e-4 from 64 bits


# ------------------------------------------------------------------------------------------- 64-bit values
_D = torch.float64


def _rot64(q):
    w, x, y, z = q.unbind(-1)
    rows = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]
    return torch.stack(rows, -1).reshape(*q.shape[:-1], 3, 3)


def _f32(v):
    return float(np.float32(v))


def _valid64(z, K):
    return (z > _f32(K["z_min"])) & (z <= _f32(K["z_max"]))


def _store64(F, dtype):
    if dtype == "f32":
        return F.float().double()
    if dtype == "f16":
        return F.half().double()
    return (F * 32767).round().clamp(-32767, 32767) / 32767


def _fuse64(dims, voxel, trunc, dtype, K, depth, poses, origin=(0.0, 0.0, 0.0)):
    """The map (values, NaN where unobserved, and weights), shaped (dz, dy, dx), in 64 bits with the storage's rounding."""
    dx, dy, dz = dims
    voxel, trunc = _f32(voxel), _f32(trunc)
    F = torch.full((dz, dy, dx), float("nan"), dtype=_D, device="cuda")
    W = torch.zeros((dz, dy, dx), dtype=_D, device="cuda")
    ax = [_f32(o) + (torch.arange(n, dtype=_D, device="cuda") + 0.5) * voxel for o, n in zip(origin, dims)]
    for f in range(len(poses)):
        p = poses[f].double()
        R, t = _rot64(p[:4]), p[4:]
        for z0 in range(0, dz, 64):
            gx, gy, gz = (ax[0] - t[0])[None, None, :], (ax[1] - t[1])[None, :, None], (ax[2][z0:z0 + 64] - t[2])[:, None, None]
            c = [R[0, a] * gx + R[1, a] * gy + R[2, a] * gz for a in range(3)]
            u = torch.floor(_f32(K["fx"]) * c[0] / c[2] + _f32(K["cx"]) + 0.5)
            v = torch.floor(_f32(K["fy"]) * c[1] / c[2] + _f32(K["cy"]) + 0.5)
            ok = (c[2] > 0) & (u >= 0) & (u < K["width"]) & (v >= 0) & (v < K["height"])
            pix = torch.where(ok, v * K["width"] + u, torch.zeros_like(u)).long()
            D = depth[f].reshape(-1).double()[pix]
            sdf = D - c[2]
            ok &= _valid64(D, K) & (sdf >= -trunc)
            new = (sdf / trunc).clamp(max=1.0)
            Fs, Ws = F[z0:z0 + 64], W[z0:z0 + 64]
            seen = ~torch.isnan(Fs)
            w = torch.where(seen, Ws, torch.zeros_like(Ws))
            got = _store64((w * torch.nan_to_num(Fs) + new) / (w + 1), dtype)
            F[z0:z0 + 64] = torch.where(ok, got, Fs)
            W[z0:z0 + 64] = torch.where(ok, (w + 1).clamp(max=255), Ws)
    return F, W


def _unproject64(depth, K, stride):
    z = depth[::stride, ::stride].double()
    v, u = torch.meshgrid(torch.arange(0, depth.shape[0], stride, device="cuda", dtype=_D),
                          torch.arange(0, depth.shape[1], stride, device="cuda", dtype=_D), indexing="ij")
    p = torch.stack([(u - _f32(K["cx"])) * z / _f32(K["fx"]), (v - _f32(K["cy"])) * z / _f32(K["fy"]), z], -1)
    return p[_valid64(z, K)]


def _overlap64(pts, prev_depth, K, cur, prev, cell):
    g = pts @ _rot64(cur[:4]).T + cur[4:] - prev[4:]
    c = g @ _rot64(prev[:4])
    u, v = _f32(K["fx"]) * c[:, 0] / c[:, 2] + _f32(K["cx"]), _f32(K["fy"]) * c[:, 1] / c[:, 2] + _f32(K["cy"])
    mu, mv = _f32(K["fx"]) * cell / c[:, 2], _f32(K["fy"]) * cell / c[:, 2]
    ok = (c[:, 2] > 0) & (u >= mu - 0.5) & (u < K["width"] - 0.5 - mu) & (v >= mv - 0.5) & (v < K["height"] - 0.5 - mv)
    iu, iv = (u + 0.5).floor().clamp(0, K["width"] - 1).long(), (v + 0.5).floor().clamp(0, K["height"] - 1).long()
    return pts[ok & _valid64(prev_depth.double()[iv, iu], K)]


def _compose64(c, d, right):
    """MovePST: poses (n, 7) of the offsets d (n, 6) from the pose c (7)."""
    dq = d[:, :3]
    n2 = (dq * dq).sum(-1, keepdim=True)
    dq = torch.where(n2 > 1, dq / n2.clamp(min=1e-300).sqrt(), dq)
    a = torch.cat([(1 - n2).clamp(min=0).sqrt(), dq], -1)
    b = c[:4].expand_as(a)
    t = c[4:] + (d[:, 3:] @ _rot64(c[:4]).T if right else d[:, 3:])
    if right:
        a, b = b, a
    q = torch.stack([a[:, 0] * b[:, 0] - a[:, 1] * b[:, 1] - a[:, 2] * b[:, 2] - a[:, 3] * b[:, 3],
                     a[:, 0] * b[:, 1] + a[:, 1] * b[:, 0] + a[:, 2] * b[:, 3] - a[:, 3] * b[:, 2],
                     a[:, 0] * b[:, 2] - a[:, 1] * b[:, 3] + a[:, 2] * b[:, 0] + a[:, 3] * b[:, 1],
                     a[:, 0] * b[:, 3] + a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1] + a[:, 3] * b[:, 0]], -1)
    q = q / q.norm(dim=-1, keepdim=True)
    return torch.cat([torch.where(q[:, :1] < 0, -q, q), t], -1)


def _score64(F, voxel, pts, poses, flags):
    """(sum of psi^2 or |psi|, valid samples) of every pose over the points."""
    dz, dy, dx = F.shape
    F = F.reshape(-1)
    voxel, S, V = _f32(voxel), [], []
    step = max(1, 6_000_000 // max(1, pts.shape[0]))
    for i in range(0, poses.shape[0], step):
        p = poses[i:i + step]
        g = (torch.einsum("nij,mj->nmi", _rot64(p[:, :4]), pts) + p[:, None, 4:]) / voxel - 0.5
        if flags == "nearest":
            k = (g + 0.5).floor().long()
            x, y, z = k.unbind(-1)
            ok = (x >= 0) & (x < dx) & (y >= 0) & (y < dy) & (z >= 0) & (z < dz)
            psi = F[torch.where(ok, x + dx * (y + dy * z), torch.zeros_like(x))]
        else:
            k = g.floor()
            a = g - k
            x, y, z = k.long().unbind(-1)
            ok = (x >= 0) & (x < dx - 1) & (y >= 0) & (y < dy - 1) & (z >= 0) & (z < dz - 1)
            at = torch.where(ok, x + dx * (y + dy * z), torch.zeros_like(x))
            psi = 0
            for c in range(8):
                wgt = 1
                for d in range(3):
                    wgt = wgt * (a[..., d] if c >> d & 1 else 1 - a[..., d])
                psi = psi + wgt * F[at + (c & 1) + dx * ((c >> 1 & 1) + dy * (c >> 2))]
        ok &= ~torch.isnan(psi)
        psi = torch.where(ok, psi, torch.ones_like(psi))
        S.append((psi.abs() if flags == "l1" else psi * psi).sum(-1))
        V.append(ok.sum(-1))
    return torch.cat(S), torch.cat(V)


def exact(case, seed):
    return globals()["_exact_" + case["kind"]](case, seed % 100003)


def _map64(case, K, depth, poses):
    return _fuse64((case["dims"],) * 3, _voxel(case["dims"]), _trunc(case["dims"]), case["dtype"], K, depth[:MAP_FRAMES],
                   poses[:MAP_FRAMES])[0]


def _exact_track(case, seed):
    """The first iteration of Algorithm 1; the pose after several has no 64-bit value (see tolerance)."""
    K, depth, poses = _map_inputs(case, seed)
    F = _map64(case, K, depth, poses)
    voxel, prev = _voxel(case["dims"]), poses[MAP_FRAMES - 1].double()
    pts = _unproject64(depth[MAP_FRAMES], K, case["stride"])
    pts = _overlap64(pts, depth[MAP_FRAMES - 1], K, prev, prev, 1.7320508 * _f32(voxel))
    r0 = torch.tensor(R_FIRST, device="cuda").double()
    offsets = nat.pst_create(case["n"], seed=1 + seed).double().T * r0
    if pts.shape[0] == 0:
        return None
    S, V = _score64(F, voxel, pts, _compose64(prev, offsets, False), "default")
    rho = torch.exp(-S / pts.shape[0])
    ref, eps, beta = rho[0], _f32(1e-3), _f32(0.1)
    wgt = torch.where(rho > ref, rho - ref, torch.zeros_like(rho))
    wgt[0] = 0
    dbar, tilde = torch.zeros(6, dtype=_D, device="cuda"), ref
    if int(V.sum()) == 0:
        tilde, rhat = torch.tensor(0.5, dtype=_D, device="cuda"), torch.full((6,), 0.5 + eps, dtype=_D, device="cuda")
    elif float(wgt.sum()) > 0:
        dbar, tilde = (wgt[:, None] * offsets).sum(0) / wgt.sum(), (wgt * rho).sum() / wgt.sum()
        rhat = (1 - tilde) * dbar.abs() / dbar.norm() + eps
    else:
        rhat = (2 * (1 - ref) / math.sqrt(6.0) + eps).expand(6)
    r1 = beta * r0 + (1 - beta) * rhat
    best = torch.topk(rho, 2).values
    pose = _compose64(prev, dbar[None], False)[0]
    return dict(pose=None, r1=r1, first=torch.cat([torch.stack([ref, tilde, best[0], best[1]]), pose, r1, dbar]))


def _exact_sequence(case, seed):
    return None


def _exact_batch(case, seed):
    return None


def _exact_fitness(case, seed):
    K, depth, poses = _map_inputs(case, seed)
    F = _map64(case, K, depth, poses)
    voxel, cur, prev = _voxel(case["dims"]), poses[MAP_FRAMES].double(), poses[MAP_FRAMES - 1].double()
    pts = _unproject64(depth[MAP_FRAMES], K, case["stride"])
    pts = _overlap64(pts, depth[MAP_FRAMES - 1], K, cur, prev, _f32(math.sqrt(3.0) * voxel))
    if pts.shape[0] == 0:
        return None
    scale = torch.tensor(_fitness_scale(case), device="cuda").double()
    offsets = nat.pst_create(case["n"], seed=1 + seed).double().T * scale
    S, _ = _score64(F, voxel, pts, _compose64(cur, offsets, case["flags"] == "right_mult"), case["flags"])
    return dict(rho=torch.exp(-S / pts.shape[0]), sumsq=S, valid=None)


def _exact_fuse(case, seed):
    dims, extent, voxel, origin = _fuse_geometry(case)
    K, depth, poses = _scene(extent, seed, case["frames"], case["width"], case["height"], case["speed"])
    F, W = _fuse64(dims, voxel, 4 * voxel, case["dtype"], K, depth, poses, origin)
    if case["export"]:
        return dict(values=None if case["dtype"] == "i16" else F, weights=None)
    pts = _unproject64(depth[-1], K, _stride(case["width"], case["height"], 20000))
    offsets = nat.pst_create(256, seed=1 + seed).double().T * torch.tensor([0.03] * 3 + [0.05] * 3, device="cuda").double()
    S, _ = _score64(F, voxel, pts, _compose64(poses[-1].double(), offsets, False), "default")
    return dict(rho=torch.exp(-S / pts.shape[0]), sumsq=S, valid=None)


def _layers64(theta):
    got, at = [], 0
    for o, i in [(256, 832), (256, 256), (256, 256), (16, 256)]:
        got.append((theta[at:at + o * i].reshape(o, i), theta[at + o * i:at + o * i + o]))
        at += o * i + o
    return [(W.to(torch.bfloat16).double(), b.double()) for W, b in got]


def _forward64(theta, x):
    """Activations of every layer, in 64 bits between the network's own roundings to bfloat16."""
    layers, h = _layers64(theta), [x.double()]
    for l, (W, b) in enumerate(layers):
        v = h[-1] @ W.T + b
        h.append(v.clamp(min=0).to(torch.bfloat16).double() if l < 3 else v)
    return layers, h


def _exact_propose(case, seed):
    K, depth, poses, theta = _propose_inputs(case, seed)
    H, W = depth.shape[1:]
    x = torch.zeros(832, dtype=_D, device="cuda")
    mean = []
    for f in (2, 1):
        z = depth[f].double()
        ok = _valid64(z, K)
        cs = [torch.zeros(H + 1, W + 1, dtype=_D, device="cuda") for _ in range(2)]
        cs[0][1:, 1:] = torch.where(ok, z, torch.zeros_like(z)).cumsum(0).cumsum(1)
        cs[1][1:, 1:] = ok.double().cumsum(0).cumsum(1)
        c = torch.arange(33, device="cuda") * W // 32
        r = torch.arange(25, device="cuda") * H // 24
        box = [(v[r][:, c][1:, 1:] - v[r][:, c][:-1, 1:] - v[r][:, c][1:, :-1] + v[r][:, c][:-1, :-1]) for v in cs]
        mean.append((box[0] / box[1].clamp(min=1), box[1] > 0))
    x[:768] = torch.where(mean[0][1] & mean[1][1], ((mean[0][0] - mean[1][0]) / 0.1).clamp(-8, 8), torch.zeros_like(mean[0][0])).reshape(-1)
    units = torch.tensor([0.05] * 3 + [0.1] * 3, dtype=_D, device="cuda")
    a, b = poses[0].double(), poses[1].double()
    inv = torch.cat([a[:4] * torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=_D, device="cuda") / (a[:4] ** 2).sum(), a[4:]])
    q = _compose64(inv, torch.cat([b[1:4], b[1:4]])[None], False)[0, :4]  # q_b q_a^-1, scalar part >= 0
    x[768:774] = torch.cat([q[1:], b[4:] - a[4:]]) / units
    xr = x.to(torch.bfloat16).double()
    o = _forward64(theta, xr[None])[1][-1]
    d = (xr[768:774] + o[0, :6]) * units
    p = nat.proposal_params()
    lo, hi = (torch.tensor(list(v), dtype=_D, device="cuda") for v in (p.r_min, p.r_max))
    r0 = (p.kappa * torch.exp(o[0, 6:12].clamp(-6, 6)) * units).clamp(lo, hi)
    return dict(x=x, o=o, c0=_compose64(b, d[None], False)[0], r0=r0)


def _exact_train(case, seed):
    theta, xs, ys, idx = _train_inputs(case, seed)
    x, y = xs[idx.long()], ys[idx.long()].double()
    layers, h = _forward64(theta, x)
    B, out = case["batch"], h[-1]
    mu, s = out[:, :6] + h[0][:, 768:774], out[:, 6:12].clamp(-6, 6)
    r, ex = y - mu, torch.exp(-2 * s)
    loss = (0.5 * r * r * (1 + ex) + s).sum(-1).mean()
    inside = (out[:, 6:12] > -6) & (out[:, 6:12] < 6)
    g = torch.zeros(B, 16, dtype=_D, device="cuda")
    g[:, :6], g[:, 6:12] = -r * (1 + ex) / B, torch.where(inside, (1 - r * r * ex) / B, torch.zeros_like(r))
    grads = []
    for l in (3, 2, 1, 0):
        g = g.to(torch.bfloat16).double()
        grads[:0] = [(g.T @ h[l]).reshape(-1), g.sum(0)]
        g = (g @ layers[l][0]) * (h[l] > 0)
    return dict(grad=torch.cat(grads), loss=loss.reshape(1), out=out)
