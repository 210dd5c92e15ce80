"""GPU PST sampling, depth preprocessing, overlap set and TSDF fusion against the
FP64 oracle and closed forms, through the C ABI."""
import math

import numpy as np
import pytest

from paper_2105_05600_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_2105_05600_gb300 import build

    build.build()
    from paper_2105_05600_gb300 import _native

    return _native


# ----------------------------------------------------------------------------- PST
@pytest.mark.parametrize("n,seed", [(1, 1), (2, 1), (1000, 1), (20000, 1), (777, 2 ** 40 + 5)])
def test_pst_uniform_bit_exact(oracle, nat, n, seed):
    gpu = nat.pst_create(n, seed=seed).cpu().numpy()
    np.testing.assert_array_equal(gpu, oracle.pst_uniform(n, seed))


def test_pst_poisson_invariants(nat):
    n = 512
    P = nat.pst_create(n, seed=3, method=1).cpu().numpy().astype(np.float64)
    U = nat.pst_create(n, seed=3, method=0).cpu().numpy().astype(np.float64)
    assert np.all(P[:, 0] == 0)
    assert np.linalg.norm(P, axis=0).max() <= 1.0 + 1e-6

    def min_dist(X):
        d = np.linalg.norm(X[:, :, None] - X[:, None, :], axis=0)
        d[np.diag_indices(X.shape[1])] = np.inf
        return d.min()

    # blue noise: the closest pair is far further apart than in a uniform sample
    assert min_dist(P) > 2.0 * min_dist(U)


# ----------------------------------------------------------------------------- points
@pytest.mark.parametrize("W,H,stride", [(80, 60, 1), (640, 480, 4), (97, 61, 3), (5, 3, 8)])
def test_depth_to_points_parity(oracle, nat, W, H, stride):
    import torch

    K = synth.intrinsics(W, H)
    rng = np.random.default_rng(W * H)
    depth = rng.uniform(0.2, 6.0, size=(H, W)).astype(np.float32)
    depth[rng.random((H, W)) < 0.1] = 0.0
    depth[rng.random((H, W)) < 0.02] = 9.5
    depth[rng.random((H, W)) < 0.02] = np.nan
    ref = oracle.unproject(depth, K, stride)
    got = nat.rf_depth_to_points(torch.from_numpy(depth).cuda(), K, stride).cpu().numpy().astype(np.float64)
    assert got.shape == ref.shape
    np.testing.assert_array_equal(got[:, 3], ref[:, 3])
    np.testing.assert_allclose(got[:, :3], ref[:, :3], rtol=1e-6, atol=1e-7)


@pytest.mark.parametrize("cell", [0.0, 0.01 * 3 ** 0.5])
def test_overlap_parity(oracle, nat, cell):
    import torch

    cfg = synth.CONFIGS["paper"]
    scene = synth.make_scene(cfg["dims"] * cfg["voxel"], cfg["wall_inset"], 0)
    traj = synth.make_trajectory(scene, 3, 3.0, 3.0, 0)
    K = synth.intrinsics(640, 480)
    d0 = synth.render_depth(scene, traj[0], K)
    d1 = synth.render_depth(scene, traj[1], K)
    pts = oracle.unproject(d1, K, 4).astype(np.float32).astype(np.float64)
    cur = traj[1].astype(np.float32).astype(np.float64)
    prev = traj[0].astype(np.float32).astype(np.float64)
    mask, margin, n = oracle.overlap(pts, d0, K, cur, prev, cell_m=cell)
    gmask, gcount = nat.rf_overlap_mask(torch.from_numpy(pts.astype(np.float32)).cuda(), torch.from_numpy(d0).cuda(),
                                        K, cur, prev, cell_extent=cell)
    gmask = gmask.cpu().numpy().astype(np.int32)
    sure = margin > 1e-3  # decisions more than 1e-3 px from a rounding boundary are unique
    assert sure.mean() > 0.99
    np.testing.assert_array_equal(gmask[sure], mask[sure])
    assert int(gcount.cpu()[0]) == int(gmask.sum())
    assert abs(int(gmask.sum()) - n) <= int((~sure).sum())


# ----------------------------------------------------------------------------- fusion
def test_integrate_fronto_parallel_plane(nat):
    import torch

    K = dict(fx=8.0, fy=8.0, cx=15.5, cy=11.5, z_min=0.1, z_max=8.0, width=32, height=24)
    v = nat.Volume(16, 0.1, 0.3, (-0.8, -0.8, 0.0), "f32")
    nat.tsdf_integrate(v, torch.full((24, 32), 1.0, device="cuda"), K, [1, 0, 0, 0, 0, 0, 0])
    F, W = v.download()
    k, j, i = np.meshgrid(np.arange(16), np.arange(16), np.arange(16), indexing="ij")
    x, y, z = -0.8 + 0.1 * (i + 0.5), -0.8 + 0.1 * (j + 0.5), 0.1 * (k + 0.5)
    inside = (z >= 0.45) & (np.abs(x) <= 0.75) & (np.abs(y) <= 0.6)
    band = inside & (1.0 - z >= -0.3)
    # FP32: z = origin + voxel (k + 0.5) carries ~2 ulp(1.6) = 2.4e-7, / trunc 0.3 -> ~8e-7
    np.testing.assert_allclose(F[band], np.minimum(1.0, (1.0 - z) / 0.3)[band], atol=1e-6)
    assert np.all(W[band] == 1)
    assert np.all(np.isnan(F[inside & (1.0 - z < -0.3)]))


@pytest.mark.parametrize("dtype", ["f32", "f16", "i16"])
def test_integrate_parity_sequence(oracle, nat, dtype):
    import torch

    cfg = dict(synth.CONFIGS["tiny"])
    dims, voxel, trunc = cfg["dims"], cfg["voxel"], cfg["trunc"]
    scene = synth.make_scene(dims * voxel, cfg["wall_inset"], 0)
    traj = synth.make_trajectory(scene, 4, 3.0, 3.0, 0)
    K = synth.intrinsics(cfg["width"], cfg["height"])
    gv = nat.Volume(dims, voxel, trunc, (0, 0, 0), dtype)
    ov = oracle.Volume((dims,) * 3, voxel, (0, 0, 0), trunc, qmode=dtype)
    amb = np.zeros(dims ** 3, bool)
    rng = np.random.default_rng(3)
    for f in range(4):
        depth = synth.render_depth(scene, traj[f], K, rng)
        pose = traj[f].astype(np.float32).astype(np.float64)
        amb |= ov.integrate_ambiguity(depth, K, pose, tol=1e-4).astype(bool)
        ov.integrate(depth, K, pose)
        nat.tsdf_integrate(gv, torch.from_numpy(depth).cuda(), K, pose)
    codes, W = gv.download()
    Fg = synth.decode_values(codes).reshape(-1)
    Wg = W.reshape(-1).astype(np.int32)
    sure = ~amb
    assert sure.mean() > 0.99
    np.testing.assert_array_equal(Wg[sure], ov.W[sure])
    both = sure & np.isfinite(Fg) & np.isfinite(ov.F)
    assert np.array_equal(np.isfinite(Fg[sure]), np.isfinite(ov.F[sure]))
    # FP32 running average vs FP64, then the storage rounding of each dtype.  In FP32
    # the camera-frame depth carries ~2 ulp(2.5 m) = 5e-7 m, i.e. 4e-6 after / trunc (0.12 m).
    atol = {"f32": 5e-6, "f16": 2e-3, "i16": 4.0 / 32767}[dtype]
    np.testing.assert_allclose(Fg[both], ov.F[both], atol=atol)
    if dtype == "i16":
        # the FP32 depth error above is up to 0.14 code steps (4e-6 * 32767), so a voxel whose
        # FP64 average lies that close to a rounding boundary may store the neighbouring code,
        # and the step then persists through the later averages: most codes agree exactly
        assert np.mean(np.abs(Fg[both] - ov.F[both]) < 0.5 / 32767 + 1e-9) > 0.98


def test_integrate_parity_many_bricks(oracle, nat):
    """A 256^3 int16 volume (32,768 bricks) whose visible bricks outnumber the
    persistent fusion grid, so every CTA walks several list entries; values and
    weights match the oracle, and the fusion counters agree with the result:
    on a fresh volume every updated voxel ends with weight 1, and the bricks that
    passed the frustum test include every brick holding an updated voxel."""
    import torch

    dims, voxel, trunc = 256, 0.02, 0.06
    scene = synth.make_scene(dims * voxel, 0.3, 5)
    traj = synth.make_trajectory(scene, 3, 3.0, 3.0, 5)
    K = synth.intrinsics(160, 120)
    gv = nat.Volume(dims, voxel, trunc, (0, 0, 0), "i16")
    ov = oracle.Volume((dims,) * 3, voxel, (0, 0, 0), trunc, qmode="i16")
    amb = np.zeros(dims ** 3, bool)
    rng = np.random.default_rng(7)
    for f in range(3):
        depth = synth.render_depth(scene, traj[f], K, rng)
        pose = traj[f].astype(np.float32).astype(np.float64)
        amb |= ov.integrate_ambiguity(depth, K, pose, tol=1e-4).astype(bool)
        ov.integrate(depth, K, pose, threads=8)
        gv.counters(reset=True)
        nat.tsdf_integrate(gv, torch.from_numpy(depth).cuda(), K, pose)
        c = gv.counters(reset=True)
        if f == 0:
            _, W0 = gv.download()
            w = W0.reshape(dims // 8, 8, dims // 8, 8, dims // 8, 8)
            bricks_touched = int((w.max(axis=(1, 3, 5)) > 0).sum())
            assert c["voxels_updated"] == int((W0 > 0).sum())
            assert bricks_touched <= c["bricks_visited"] < (dims // 8) ** 3
            assert c["bricks_visited"] > 2 * 152 * 4  # more list entries than CTAs in the grid
            assert 0 < c["bricks_repacked"] <= 8 * bricks_touched
    codes, W = gv.download()
    Fg = synth.decode_values(codes).reshape(-1)
    Wg = W.reshape(-1).astype(np.int32)
    sure = ~amb
    assert sure.mean() > 0.99
    np.testing.assert_array_equal(Wg[sure], ov.W[sure])
    assert np.array_equal(np.isfinite(Fg[sure]), np.isfinite(ov.F[sure]))
    both = sure & np.isfinite(Fg) & np.isfinite(ov.F)
    np.testing.assert_allclose(Fg[both], ov.F[both], atol=4.0 / 32767)


@pytest.mark.parametrize("dtype", ["f32", "f16", "i16"])
@pytest.mark.parametrize("dims", [(304, 296, 288), (96, 104, 88)])
def test_integrate_free_space_bricks(oracle, nat, dtype, dims):
    """Volumes on both sides of the brick count from which whole bricks are fused as free space, a frame that ends
    inside a pixel tile, with unequal focal lengths and clustered holes, and a map that already holds weights up to
    their limit, unobserved voxels and values other than +1 in front of the surface: values and weights against the
    oracle after three frames, in which many bricks of the large map went the free-space way."""
    import torch

    voxel, trunc = 5.12 / max(dims), 4 * 5.12 / max(dims)
    scene = synth.make_scene(5.12, 0.3, 11)
    traj = synth.make_trajectory(scene, 3, 2.0, 2.0, 11)
    K = synth.intrinsics(197, 131)
    K["fy"] *= 1.2
    rng = np.random.default_rng(3)
    shape = dims[::-1]
    F0 = np.where(rng.random(shape) < 0.02, rng.uniform(-1, 1, shape), 1.0)
    F0[:, : dims[1] // 4] = np.where(rng.random((shape[0], dims[1] // 4, shape[2])) < 0.5, np.nan, 1.0)
    codes0 = synth.encode_values(F0, dtype)
    W0 = np.where(np.isnan(F0), 0, rng.integers(1, 256, shape)).astype(np.uint8)
    gv = nat.Volume(dims, voxel, trunc, (0, 0, 0), dtype)
    gv.upload(codes0, W0)
    ov = oracle.Volume(dims, voxel, (0, 0, 0), trunc, qmode=dtype)
    ov.F[:] = synth.decode_values(codes0).reshape(-1)
    ov.W[:] = W0.reshape(-1)
    amb = np.zeros(F0.size, bool)
    for f in range(3):
        depth = synth.render_depth(scene, traj[f], K, rng)
        depth[20:37, 60:90] = 0.0
        depth[100:, 150:][rng.random((31, 47)) < 0.1] = np.nan
        pose = traj[f].astype(np.float32).astype(np.float64)
        amb |= ov.integrate_ambiguity(depth, K, pose, tol=1e-4).astype(bool)
        ov.integrate(depth, K, pose, threads=8)
        nat.tsdf_integrate(gv, torch.from_numpy(depth).cuda(), K, pose)
        projected, free = gv.fusion_lists()
        assert projected > 100 and (free > 100 if np.prod(dims) // 512 >= 49152 else free == 0)
    codes, W = gv.download()
    Fg = synth.decode_values(codes).reshape(-1)
    sure = ~amb
    assert sure.mean() > 0.98
    np.testing.assert_array_equal(W.reshape(-1).astype(np.int32)[sure], ov.W[sure])
    assert np.array_equal(np.isfinite(Fg[sure]), np.isfinite(ov.F[sure]))
    both = sure & np.isfinite(Fg) & np.isfinite(ov.F)
    # one rounding step of the storage per frame, FP32 arithmetic (1e-5 of the truncation) below it
    atol = {"f32": 2e-5, "f16": 3 * 2.0**-11, "i16": 4.0 / 32767}[dtype]
    np.testing.assert_allclose(Fg[both], ov.F[both], atol=atol)


@pytest.mark.parametrize("sx,sy", [(1, -1), (-1, 1), (-1, -1)])
@pytest.mark.parametrize("dims", [(304, 296, 288), (96, 104, 88)])
def test_integrate_negative_focal_length(oracle, nat, dims, sx, sy):
    """A focal length may have either sign (some datasets publish fy = -480): a fresh map on both sides of the brick
    count from which whole bricks are fused as free space, unequal focal lengths, two frames, against the oracle."""
    import torch

    voxel, trunc = 5.12 / max(dims), 4 * 5.12 / max(dims)
    scene = synth.make_scene(5.12, 0.3, 12)
    traj = synth.make_trajectory(scene, 2, 2.0, 2.0, 12)
    K = synth.intrinsics(161, 119)
    K["fx"], K["fy"] = sx * K["fx"], sy * 1.25 * K["fy"]
    rng = np.random.default_rng(4)
    gv = nat.Volume(dims, voxel, trunc, (0, 0, 0), "i16")
    ov = oracle.Volume(dims, voxel, (0, 0, 0), trunc, qmode="i16")
    amb = np.zeros(ov.F.size, bool)
    for f in range(2):
        depth = synth.render_depth(scene, traj[f], K, rng)
        depth[7:19, 90:101] = 0.0
        pose = traj[f].astype(np.float32).astype(np.float64)
        amb |= ov.integrate_ambiguity(depth, K, pose, tol=1e-4).astype(bool)
        ov.integrate(depth, K, pose, threads=8)
        nat.tsdf_integrate(gv, torch.from_numpy(depth).cuda(), K, pose)
        assert (gv.fusion_lists()[1] > 100) == (np.prod(dims) // 512 >= 49152)
    codes, W = gv.download()
    Fg = synth.decode_values(codes).reshape(-1)
    sure = ~amb
    assert sure.mean() > 0.98 and ov.W.max() == 2
    np.testing.assert_array_equal(W.reshape(-1).astype(np.int32)[sure], ov.W[sure])
    both = sure & np.isfinite(ov.F)
    assert np.array_equal(np.isfinite(Fg[sure]), np.isfinite(ov.F[sure]))
    np.testing.assert_allclose(Fg[both], ov.F[both], atol=4.0 / 32767)  # a storage step a frame, FP32 below it


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("dims", [(304, 296, 288), (96, 104, 88)])
def test_integrate_keeps_infinities(nat, dtype, dims):
    """Values that a float or half map can hold but no frame produces: the running average (W F + 1) / (W + 1) as IEEE
    arithmetic gives it, in free bricks, in bricks next to invalid pixels and on small maps."""
    import torch

    voxel = 5.12 / max(dims)
    np_t = np.float32 if dtype == "f32" else np.float16
    special = [np.inf, -np.inf] + ([3e38, -3e38, 1e-40, -1e-45, 1e31] if dtype == "f32" else [65504, -65504, 6e-8])
    rng = np.random.default_rng(5)
    shape = dims[::-1]
    F0 = np.ones(shape, np_t)
    at = rng.random(shape) < 0.01
    F0[at] = rng.choice(np.array(special, np_t), at.sum())
    W0 = rng.integers(1, 200, shape).astype(np.uint8)
    gv = nat.Volume(dims, voxel, 3 * voxel, (0, 0, 0), dtype)
    gv.upload(F0, W0)
    K = synth.intrinsics(160, 120, z_max=9.0)
    depth = np.full((120, 160), 8.5, np.float32)  # beyond the map: f = 1 in every voxel in view
    depth[50:60, 70:75] = 0.0
    nat.tsdf_integrate(gv, torch.from_numpy(depth).cuda(), K, [1, 0, 0, 0, 2.5, 2.5, -1.0])
    assert gv.fusion_lists()[0] > 20 and (gv.fusion_lists()[1] > 100) == (np.prod(dims) // 512 >= 49152)
    F1, W1 = gv.download()
    F1, W1 = F1.reshape(shape), W1.reshape(shape)
    up = W1 == W0 + 1
    assert np.array_equal(W1[~up], W0[~up]) and up.mean() > 0.3 and up[at].sum() > 1000
    np.testing.assert_array_equal(F1[~up], F0[~up])
    w, one = W0[up].astype(np.float32), np.float32(1)
    with np.errstate(over="ignore"):
        # one rounding of W F + 1 to FP32, as fma does: W F is exact in FP64, and where the 1 lies below its last bit
        # the next FP64 number stands for it (it decides ties of the FP32 rounding)
        total = w.astype(np.float64) * F0[up].astype(np.float64)
        total = np.where(np.isfinite(total) & (np.abs(total) > 2.0**53), np.nextafter(total, np.inf), total + 1.0)
        total = total.astype(np.float32)
        want = (total / (w + one)).astype(np_t)
    np.testing.assert_array_equal(F1[up], want)


def _hard_quotients(n, rng):
    """Pairs (a, b) of 24-bit integers whose quotient lies next to a midpoint of two floats: a 2^k = b m + c with m an
    odd 25-bit integer and c a few units, k = 24 or 25."""
    A, B = [], []
    while sum(map(len, A)) < n:
        b = (rng.integers(1 << 23, 1 << 24, 1 << 20) | 1).astype(np.uint64)
        b[::8] = (1 << 24) - 1 - 2 * rng.integers(0, 64, len(b[::8])).astype(np.uint64)
        c = rng.choice(np.array([-4, -3, -2, -1, 1, 2, 3, 4]), b.size)
        k = rng.integers(24, 26, b.size).astype(np.uint64)
        mod = np.uint64(1) << k
        inv = np.ones_like(b)
        for _ in range(6):
            inv = inv * (np.uint64(2) - b * inv)  # the inverse of an odd b modulo 2^64, by Newton
        m = ((-c).astype(np.uint64) * inv) & (mod - np.uint64(1))
        m = np.where(m < 1 << 24, m + mod, m)
        a2 = b * m + c.astype(np.uint64)
        a = a2 >> k
        ok = (m & np.uint64(1) == 1) & (m < 1 << 25) & (a << k == a2) & (a >= 1 << 23) & (a < 1 << 24)
        A.append(a[ok])
        B.append(b[ok])
    return np.concatenate(A)[:n].astype(np.float32), np.concatenate(B)[:n].astype(np.float32)


def test_fusion_quotients_are_those_of_ieee_division(nat):
    """Every significand's reciprocal, and quotients that a last-bit error anywhere would round the wrong way:
    next to midpoints, the running average's divisors 1 .. 256, depths over a wide range."""
    import torch

    rng = np.random.default_rng(8)
    b = (np.arange(1 << 23, dtype=np.uint32) | np.uint32(127 << 23)).view(np.float32)
    scale = np.float32(2.0) ** rng.integers(-29, 30, b.size).astype(np.float32)
    dev = lambda x: torch.from_numpy(x).cuda()
    for bs in (b, b * scale):
        out = torch.empty(b.size, device="cuda")
        nat.rf_quotient_probe(None, dev(bs), out)
        np.testing.assert_array_equal(out.cpu().numpy(), np.float32(1) / bs)
    hard = _hard_quotients(1 << 20, rng)
    div = np.repeat(np.arange(1, 257, dtype=np.float32), 4096)
    avg = ((div - 1) * rng.uniform(-1, 1, div.size) + rng.uniform(-1, 1, div.size)).astype(np.float32)
    z = np.exp(rng.uniform(np.log(1e-8), np.log(1e4), 1 << 20)).astype(np.float32)
    nu = (rng.normal(size=z.size) * z * 500).astype(np.float32)
    for a, d in (hard, (hard[0] * np.float32(2.0**-9), hard[1] * np.float32(2.0**-22)), (avg, div), (nu, z)):
        out = torch.empty(a.size, device="cuda")
        nat.rf_quotient_probe(dev(a), dev(d), out)
        np.testing.assert_array_equal(out.cpu().numpy(), a / d)


def test_dirty_brick_repacking_matches_full_pack(nat):
    """Fusion repacks only the trilinear cells of bricks it touched; a volume that
    receives the same values by upload (full repack) must score identically."""
    import torch

    cfg = dict(synth.CONFIGS["tiny"])
    dims, voxel, trunc = cfg["dims"], cfg["voxel"], cfg["trunc"]
    scene = synth.make_scene(dims * voxel, cfg["wall_inset"], 0)
    traj = synth.make_trajectory(scene, 4, 3.0, 3.0, 0)
    K = synth.intrinsics(cfg["width"], cfg["height"])
    for dtype in ("i16", "f16", "f32"):
        a = nat.Volume(dims, voxel, trunc, (0, 0, 0), dtype)
        for f in range(4):
            nat.tsdf_integrate(a, torch.from_numpy(synth.render_depth(scene, traj[f], K)).cuda(), K, traj[f])
        codes, w = a.download()
        b = nat.Volume(dims, voxel, trunc, (0, 0, 0), dtype)
        b.upload(codes, w)
        d = torch.from_numpy(synth.render_depth(scene, traj[2], K)).cuda()
        pts = nat.rf_depth_to_points(d, K, 1)
        pts = pts[pts[:, 3] > 0].contiguous()
        pst = nat.pst_create(512, seed=4)
        ra = nat.fitness_eval(a, pts, pst, traj[1], [0.05] * 6, nat.make_params())
        rb = nat.fitness_eval(b, pts, pst, traj[1], [0.05] * 6, nat.make_params())
        for x, y in zip(ra, rb):
            np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy())


def test_integrate_skips_invalid_depth(nat):
    import torch

    K = synth.intrinsics(80, 60)
    v = nat.Volume(64, 0.04, 0.12, (0, 0, 0), "i16")
    d = torch.zeros((60, 80), device="cuda")
    d[10, 10] = float("nan")
    nat.tsdf_integrate(v, d, K, [1, 0, 0, 0, 1.28, 1.28, 1.28])
    codes, W = v.download()
    assert W.max() == 0 and np.all(codes == -32768)
