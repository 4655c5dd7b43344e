"""GPU parity of the Q-Render hot path against the FP64 oracle, through the C ABI.

Tolerances (derived in the design notes):
  * selected ids: bit-exact on every pixel the oracle does not flag as a near
    tie; flagged pixels must stay a small fraction and are reported;
  * FP32 features: mixed relative error (oracle/compare.py) <= FEAT_TOL;
  * dense Eq. 1: same metric <= DENSE_TOL (longer FP32 products).
"""
import numpy as np
import pytest

import oracle
from oracle import compare
from paper_2512_20927_gb300 import scenes

import gpu_harness as H

pytestmark = pytest.mark.gpu

FEAT_TOL = 1e-5     # blend of fixed ids/weights and end-to-end Q-Render features
DENSE_TOL = 2e-5    # Eq. 1 over the whole list (up to a few hundred FP32 factors)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_20927_gb300 import qrender
    qrender.load()


def test_tiny_config_end_to_end():
    g, f = scenes.tiny_scene()
    cam = scenes.tiny_camera()
    gpu = H.run_gpu(g, f, cam, K=8)
    pr, pix, ref = H.run_oracle(g, f, cam, 8)
    rep = H.check_frame(gpu, ref, pix, cam.width, f, FEAT_TOL, DENSE_TOL, label="tiny")
    print("tiny", rep)


def test_projection_matches_oracle():
    g, f = H.small_room(n=20000, channels=16)
    cam = scenes.room_camera(320, 240)
    from paper_2512_20927_gb300 import qrender as q
    import torch
    gdev = q.gaussians_to_device(g)
    fr = q.frame_create(g.n, cam, q.default_params(8), 1 << 22)
    q.qr_project(fr, *gdev)
    v = q.qr_frame_view_get(fr)
    torch.cuda.synchronize()
    n = g.n
    rec_m = _device_copy(v.mean2d_hi_lo, n * 4, torch.float32).view(n, 4).cpu().numpy()
    axes = _device_copy(v.axes, n * 4, torch.float32).view(n, 4).cpu().numpy().astype(np.float64)
    opac = _device_copy(v.opacity, n, torch.float32).cpu().numpy()
    dkey = _device_copy(v.depth_key, n, torch.int32).cpu().numpy().view(np.uint32)
    pr = oracle.project(g, cam.as_array())
    vis = dkey != 0xFFFFFFFF
    assert vis.sum() > 100
    # every Gaussian the GPU keeps is in front of the near plane in FP64
    assert (pr.valid[vis] == 1).all()
    m2 = rec_m[vis, 0:2].astype(np.float64) + rec_m[vis, 2:4].astype(np.float64)
    np.testing.assert_allclose(m2, pr.mean2d[vis], rtol=0, atol=1e-6)
    # conic rebuilt from the principal axes: A = 2 (w1 w1^T + w2 w2^T)
    w1, w2 = axes[vis, 0:2], axes[vis, 2:4]
    A = 2.0 * np.stack([w1[:, 0] ** 2 + w2[:, 0] ** 2, w1[:, 0] * w1[:, 1] + w2[:, 0] * w2[:, 1],
                        w1[:, 1] ** 2 + w2[:, 1] ** 2], axis=1)
    scale = np.abs(pr.conic[vis]).max(axis=1, keepdims=True)
    assert (np.abs(A - pr.conic[vis]) <= 1e-6 * scale).all(), np.abs(A - pr.conic[vis]).max()
    # the axes are orthogonal
    assert (np.abs((w1 * w2).sum(axis=1)) <= 1e-6 * np.linalg.norm(w1, axis=1) *
            np.linalg.norm(w2, axis=1)).all()
    depth32 = dkey[vis].view(np.float32).astype(np.float64)
    assert (np.abs(depth32 - pr.depth[vis]) <= 2.0 ** -23 * pr.depth[vis]).all()
    np.testing.assert_array_equal(opac[vis], g.opacity[vis])
    # Gaussians with any visible pixel are kept (checked on the oracle's members)
    ref = oracle.render(pr, None, 8, oracle.all_pixels(cam.width, cam.height), want_q=False,
                        want_dense=False, max_members=64)
    members = np.unique(ref.members[ref.members >= 0])
    assert vis[members].all()


def _device_copy(ptr, count, dtype):
    """Copy `count` elements at a raw device pointer into a new torch tensor."""
    import torch
    typestr = {torch.float32: "<f4", torch.int32: "<i4", torch.uint8: "|u1"}[dtype]

    class _View:
        __cuda_array_interface__ = {"shape": (count,), "typestr": typestr,
                                    "data": (int(ptr), False), "version": 3, "strides": None}
    return torch.as_tensor(_View(), device="cuda").clone()


def test_tile_lists_sorted_and_conservative():
    g, f = scenes.tiny_scene()
    cam = scenes.tiny_camera()
    gpu = H.run_gpu(g, None, cam, K=8, dense=False)
    fr = gpu["frame"]
    from paper_2512_20927_gb300 import qrender as q
    import torch
    v = q.qr_frame_view_get(fr)
    nis = gpu["n_isect"]
    tiles = fr.frame.tiles_x * fr.frame.tiles_y
    cnt = _device_copy(v.counters, 8, torch.int32).cpu().numpy()
    n_kept = int(cnt[2])
    assert int(cnt[1]) == nis
    gkey = _device_copy(v.depth_key, g.n, torch.int32).cpu().numpy().view(np.uint32)
    tcount = _device_copy(v.tile_count, g.n, torch.int32).cpu().numpy()
    kid = _device_copy(v.kept_gid, n_kept, torch.int32).cpu().numpy()
    koff = _device_copy(v.kept_offset, n_kept, torch.int32).cpu().numpy()
    gids = _device_copy(v.isect_gid, nis, torch.int32).cpu().numpy()
    rng = _device_copy(v.tile_range, 2 * tiles, torch.int32).cpu().numpy().reshape(tiles, 2)
    # kept set: finite depth key <=> non-empty footprint, compacted in id order
    kept = np.nonzero(gkey != 0xFFFFFFFF)[0]
    np.testing.assert_array_equal(kid, kept)
    assert (tcount[kept] > 0).all() and (tcount[gkey == 0xFFFFFFFF] == 0).all()
    np.testing.assert_array_equal(koff, np.concatenate([[0], np.cumsum(tcount[kid])[:-1]]))
    assert koff[-1] + tcount[kid[-1]] == nis
    # ranges tile the list; every kept Gaussian appears once per touched tile
    assert rng[0, 0] == 0 and rng[-1, 1] == nis and (rng[1:, 0] == rng[:-1, 1]).all()
    np.testing.assert_array_equal(np.bincount(gids, minlength=g.n), tcount)
    # each tile's list is ordered by (FP32 depth key, id)
    depth32 = gkey.view(np.float32)
    for t in range(tiles):
        a, b = rng[t]
        assert len(set(gids[a:b].tolist())) == b - a
        order = np.lexsort((gids[a:b], depth32[gids[a:b]]))
        np.testing.assert_array_equal(order, np.arange(b - a))
    # every member of a pixel (FP64 oracle) appears in its tile's list
    pr = oracle.project(g, cam.as_array())
    ref = oracle.render(pr, None, 8, oracle.all_pixels(cam.width, cam.height), want_q=False,
                        want_dense=False, max_members=64)
    assert ref.n_members.max() <= 64
    for p in range(cam.width * cam.height):
        x, y = p % cam.width, p // cam.width
        t = (y // 16) * fr.frame.tiles_x + x // 16
        a, b = rng[t]
        mem = ref.members[p][ref.members[p] >= 0]
        assert np.isin(mem, gids[a:b]).all()


def test_large_tile_lists_use_the_merge_path():
    """Tiles with more than 8192 Gaussians are sorted in chunks and merged."""
    rng = np.random.default_rng(11)
    n = 30000
    # a thin slab of small Gaussians right in front of a 48x48 camera: every
    # tile sees thousands of them
    mean = np.stack([rng.uniform(-0.2, 0.2, n), rng.uniform(-0.2, 0.2, n),
                     rng.uniform(-0.5, 0.5, n)], 1).astype(np.float32)
    g = scenes.Gaussians(mean, np.full((n, 3), -2.0, np.float32),
                         np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1)),
                         np.full(n, 0.05, np.float32))
    f = rng.normal(size=(n, 16)).astype(np.float32)
    cam = scenes.tiny_camera(48, 48)
    gpu = H.run_gpu(g, f, cam, K=8)
    fr = gpu["frame"]
    from paper_2512_20927_gb300 import qrender as q
    import torch
    v = q.qr_frame_view_get(fr)
    tiles = fr.frame.tiles_x * fr.frame.tiles_y
    rngs = _device_copy(v.tile_range, 2 * tiles, torch.int32).cpu().numpy().reshape(tiles, 2)
    sizes = rngs[:, 1] - rngs[:, 0]
    assert sizes.max() > 8192, sizes.max()
    gkey = _device_copy(v.depth_key, n, torch.int32).cpu().numpy().view(np.uint32)
    gids = _device_copy(v.isect_gid, gpu["n_isect"], torch.int32).cpu().numpy()
    for t in range(tiles):
        a, b = rngs[t]
        order = np.lexsort((gids[a:b], gkey.view(np.float32)[gids[a:b]]))
        np.testing.assert_array_equal(order, np.arange(b - a))
    pix = H.sample_pixels(48, 48, 200, seed=3)
    pr, pix, ref = H.run_oracle(g, f, cam, 8, pixels=pix)
    # 30,000 Gaussians within 1 m of depth: the FP32 depth keys of neighbours
    # in a pixel's list collide often, and the oracle flags 90 of these 204
    # pixels (44 %; deterministic for this seed)
    H.check_frame(gpu, ref, pix, cam.width, f, FEAT_TOL, DENSE_TOL, max_tie_frac=0.46,
                  label="big tiles")


def _slab_scene(n, seed=11):
    """A thin slab of small Gaussians right in front of a 48x48 camera: the
    central tiles see nearly all of them."""
    rng = np.random.default_rng(seed)
    mean = np.stack([rng.uniform(-0.2, 0.2, n), rng.uniform(-0.2, 0.2, n),
                     rng.uniform(-0.5, 0.5, n)], 1).astype(np.float32)
    g = scenes.Gaussians(mean, np.full((n, 3), -2.0, np.float32),
                         np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1)),
                         np.full(n, 0.05, np.float32))
    return g, rng.normal(size=(n, 16)).astype(np.float32)


@pytest.mark.parametrize("n,lo,hi", [(200, 1, 256), (420, 257, 512), (900, 513, 1024),
                                     (1800, 1025, 2048), (5000, 2049, 8192)])
def test_tile_sort_size_classes(n, lo, hi):
    """Each size class of the per-tile sort (registers with 1, 2, 4, 8 keys
    per thread; shared memory up to 8192 keys) orders its bucket by
    (FP32 depth, id) and keeps every intersection exactly once."""
    g, f = _slab_scene(n)
    cam = scenes.tiny_camera(48, 48)
    gpu = H.run_gpu(g, f, cam, K=8)
    fr = gpu["frame"]
    from paper_2512_20927_gb300 import qrender as q
    import torch
    v = q.qr_frame_view_get(fr)
    tiles = fr.frame.tiles_x * fr.frame.tiles_y
    rngs = _device_copy(v.tile_range, 2 * tiles, torch.int32).cpu().numpy().reshape(tiles, 2)
    sizes = rngs[:, 1] - rngs[:, 0]
    assert lo <= sizes.max() <= hi, sizes
    gkey = _device_copy(v.depth_key, n, torch.int32).cpu().numpy().view(np.uint32)
    tcount = _device_copy(v.tile_count, n, torch.int32).cpu().numpy()
    gids = _device_copy(v.isect_gid, gpu["n_isect"], torch.int32).cpu().numpy()
    np.testing.assert_array_equal(np.bincount(gids, minlength=n), tcount)
    for t in range(tiles):
        a, b = rngs[t]
        assert len(set(gids[a:b].tolist())) == b - a
        order = np.lexsort((gids[a:b], gkey.view(np.float32)[gids[a:b]]))
        np.testing.assert_array_equal(order, np.arange(b - a))
    pix = H.sample_pixels(48, 48, 120, seed=5)
    pr, pix, ref = H.run_oracle(g, f, cam, 8, pixels=pix)
    # the oracle flags at most 6 of these 124 pixels (4.8 %, n = 1800)
    H.check_frame(gpu, ref, pix, cam.width, f, FEAT_TOL, DENSE_TOL, max_tie_frac=0.05,
                  label=f"slab {n}")


@pytest.mark.parametrize("n", [1, 2, 256, 300, 1025, 2048, 2049, 5000, 9000])
@pytest.mark.parametrize("depths", ["equal", "few", "narrow", "clusters"])
def test_tile_sort_equal_and_narrow_depths(n, depths):
    """Buckets whose 32-bit sort keys tie: one depth, a few, a range of a few
    ulps beside a far Gaussian, clusters.  The lists are in (depth, id) order."""
    import torch
    from paper_2512_20927_gb300 import qrender as q
    g, _ = _slab_scene(n)
    rng = np.random.default_rng(n)
    z = {"equal": np.zeros(n), "few": rng.integers(0, 7, n) * 0.05, "narrow": rng.integers(0, 40, n) * 2.0 ** -21,
         "clusters": rng.integers(0, 5, n) * 0.1 + rng.normal(0, 1e-5, n)}[depths]
    if depths == "narrow" and n > 2:
        z[n // 2] = -50.0
    g.mean[:, 2] = z
    fr = H.run_gpu(g, None, scenes.tiny_camera(48, 48), K=8, dense=False)["frame"]
    v = q.qr_frame_view_get(fr)
    tiles = fr.frame.tiles_x * fr.frame.tiles_y
    rngs = _device_copy(v.tile_range, 2 * tiles, torch.int32).cpu().numpy().reshape(tiles, 2)
    gkey = _device_copy(v.depth_key, n, torch.int32).cpu().numpy().view(np.uint32)
    gids = _device_copy(v.isect_gid, int(rngs[-1, 1]), torch.int32).cpu().numpy()
    assert (rngs[:, 1] - rngs[:, 0]).max() >= 0.9 * n - 1
    for a, b in rngs:
        order = np.lexsort((gids[a:b], gkey.view(np.float32)[gids[a:b]]))
        np.testing.assert_array_equal(order, np.arange(b - a))
        assert len(set(gids[a:b].tolist())) == b - a


@pytest.mark.parametrize("n", [300, 2048, 2049, 8192, 9000])
@pytest.mark.parametrize("run", [2, 256, 257, 258])
@pytest.mark.parametrize("ulps", [1, 16])
def test_tile_sort_runs_of_close_depths(n, run, ulps):
    """One run of keys whose leading bits agree, at the longest length that is
    placed by rank and beside it, among distinct depths: equal depths, or 16
    values that a far Gaussian leaves the 32-bit keys no bits for."""
    import torch
    from paper_2512_20927_gb300 import qrender as q
    g, _ = _slab_scene(n)
    rng = np.random.default_rng(n + run)
    z = rng.permutation(n) * (1.0 / n) + 0.25
    at = rng.choice(n, run, replace=False)
    z[at] = rng.integers(0, ulps, run) * 2.0 ** -21
    if ulps > 1:
        z[np.setdiff1d(np.arange(n), at)[0]] = -50.0
    g.mean[:, 2] = z
    fr = H.run_gpu(g, None, scenes.tiny_camera(48, 48), K=8, dense=False)["frame"]
    v = q.qr_frame_view_get(fr)
    tiles = fr.frame.tiles_x * fr.frame.tiles_y
    rngs = _device_copy(v.tile_range, 2 * tiles, torch.int32).cpu().numpy().reshape(tiles, 2)
    gkey = _device_copy(v.depth_key, n, torch.int32).cpu().numpy().view(np.float32)
    gids = _device_copy(v.isect_gid, int(rngs[-1, 1]), torch.int32).cpu().numpy()
    assert (rngs[:, 1] - rngs[:, 0]).max() >= 0.9 * n - 1
    assert len(np.unique(gkey[at])) <= ulps
    for a, b in rngs:
        np.testing.assert_array_equal(np.lexsort((gids[a:b], gkey[gids[a:b]])), np.arange(b - a))
        assert len(set(gids[a:b].tolist())) == b - a


@pytest.mark.parametrize("C", [16, 64, 512])
def test_blend_stage_matches_definition(C):
    import torch
    from paper_2512_20927_gb300 import qrender as q
    rng = np.random.default_rng(C)
    n, P, K = 5000, 3000, 8
    f = rng.normal(size=(n, C)).astype(np.float32)
    ids, w, cnt = scenes.random_selection(seed=C, pixels=P, k=K, n=n)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    out = torch.empty((P, C), dtype=torch.float32, device="cuda")
    q.qr_blend(dev(f), None, dev(ids), dev(w), dev(cnt), out)
    torch.cuda.synchronize()
    ref = compare.blend(ids, w, cnt, f)
    err = compare.feature_error(out.cpu().numpy(), ref, compare.blend_scale(ids, w, cnt, f))
    assert err.max() <= FEAT_TOL, err.max()
    assert (out.cpu().numpy()[cnt == 0] == 0).all()


@pytest.mark.parametrize("K", [4, 8, 16])
def test_room_small_ragged(K):
    g, f = H.small_room(n=20000, channels=64)
    cam = scenes.room_camera(150, 110)        # ragged: neither side a multiple of 16
    gpu = H.run_gpu(g, f, cam, K=K)
    pr, pix, ref = H.run_oracle(g, f, cam, K)
    rep = H.check_frame(gpu, ref, pix, cam.width, f, FEAT_TOL, DENSE_TOL, label=f"room K={K}")
    print(f"room-small K={K}", rep)


def test_room_tiles_8x32():
    g, f = H.small_room(n=20000, channels=64)
    cam = scenes.room_camera(150, 110)
    gpu = H.run_gpu(g, f, cam, K=8, params_kw={"tile_w": 8, "tile_h": 32})
    pr, pix, ref = H.run_oracle(g, f, cam, 8)
    H.check_frame(gpu, ref, pix, cam.width, f, FEAT_TOL, DENSE_TOL, label="8x32")


@pytest.mark.parametrize("K", [1, 32])
def test_extreme_k(K):
    g, f = scenes.tiny_scene(seed=2)
    cam = scenes.tiny_camera(96, 80)
    gpu = H.run_gpu(g, f, cam, K=K)
    pr, pix, ref = H.run_oracle(g, f, cam, K)
    H.check_frame(gpu, ref, pix, cam.width, f, FEAT_TOL, DENSE_TOL, label=f"K={K}")


def test_dense_without_early_stop():
    g, f = scenes.tiny_scene(seed=4)
    cam = scenes.tiny_camera(64, 64)
    gpu = H.run_gpu(g, f, cam, K=8, params_kw={"T_min": 0.0})
    pr, pix, ref = H.run_oracle(g, f, cam, 8, T_min=0.0)
    H.check_frame(gpu, ref, pix, cam.width, f, FEAT_TOL, DENSE_TOL, label="T_min=0")


@pytest.mark.parametrize("C,T_min,size", [(64, 1e-4, (33, 50)), (128, 0.0, (48, 48)), (256, 1e-4, (41, 23)),
                                          (512, 0.0, (17, 9))])
def test_dense_long_lists(C, T_min, size):
    """Blocks that keep hundreds of entries (every ring of the block kernel
    wraps around), images smaller than a tile and with cut blocks."""
    rng = np.random.default_rng(11)
    n = 2000
    mean = np.stack([rng.uniform(-0.2, 0.2, n), rng.uniform(-0.2, 0.2, n),
                     rng.uniform(-1.5, 1.5, n)], 1).astype(np.float32)
    g = scenes.Gaussians(mean, np.full((n, 3), -2.0, np.float32),
                         np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1)),
                         np.full(n, 0.02, np.float32))
    f = rng.normal(size=(n, C)).astype(np.float32)
    cam = scenes.tiny_camera(*size)
    gpu = H.run_gpu(g, f, cam, K=8, dense=True, params_kw={"T_min": T_min})
    pr, pix, ref = H.run_oracle(g, f, cam, 8, T_min=float(np.float32(T_min)))
    assert ref.n_dense.max() > 300
    ok = (ref.tie & compare.DENSE_TIE_BITS) == 0
    err = compare.feature_error(np.asarray(gpu["dense"]), ref.out_dense, ref.scale_dense)[ok]
    # every factor of T and every sum rounds once: 2^-23 per entry of the longest walk
    assert err.max() <= DENSE_TOL + 2.0 ** -23 * ref.n_dense.max(), err.max()


def test_indoor_full_size_sampled():
    """The 500k-Gaussian 640x480 512-D workload in the benchmark's launch
    configuration, checked on sampled pixels the oracle computes one by one."""
    g, f = scenes.room_scene(seed=0, n=500_000, channels=512)
    cam = scenes.room_camera(640, 480)
    gpu = H.run_gpu(g, f, cam, K=8, dense=True)
    pix = H.sample_pixels(640, 480, 300, seed=1)
    pr, pix, ref = H.run_oracle(g, f, cam, 8, pixels=pix)
    rep = H.check_frame(gpu, ref, pix, cam.width, f, FEAT_TOL, DENSE_TOL, label="indoor")
    print("indoor sampled", rep, "n_isect", gpu["n_isect"])


def test_empty_and_culled_scenes():
    import torch
    from paper_2512_20927_gb300 import qrender as q
    cam = scenes.tiny_camera(40, 24)
    # all Gaussians behind the camera
    g, f = scenes.tiny_scene(n=300)
    g.mean[:, 2] = 10.0      # camera at z=3 looking down -z: these are behind it
    gpu = H.run_gpu(g, f, cam, K=8)
    assert (gpu["counts"] == 0).all() and (gpu["out"] == 0).all() and (gpu["dense"] == 0).all()
    assert gpu["n_isect"] == 0
    # zero Gaussians
    g0 = scenes.Gaussians(np.zeros((0, 3), np.float32), np.zeros((0, 3), np.float32),
                          np.zeros((0, 4), np.float32), np.zeros(0, np.float32))
    fr = q.frame_create(0, cam, q.default_params(8), 1024)
    P = fr.pixels
    ids = torch.full((P, 8), 7, dtype=torch.int32, device="cuda")
    w = torch.full((P, 8), 3.0, device="cuda")
    cnt = torch.full((P,), 9, dtype=torch.uint8, device="cuda")
    e = torch.empty(0, device="cuda")
    q.qr_project(fr, e, e, e, e)
    q.qr_sort(fr)
    q.qr_select(fr, ids, w, cnt)
    torch.cuda.synchronize()
    assert (cnt == 0).all() and (ids == -1).all() and (w == 0).all()
    del g0


def test_capacity_overflow_is_reported_and_outputs_are_zero():
    import torch
    from paper_2512_20927_gb300 import qrender as q
    g, f = scenes.tiny_scene()
    cam = scenes.tiny_camera()
    gdev = q.gaussians_to_device(g)
    fr = q.frame_create(g.n, cam, q.default_params(8), 100)     # far too small
    P = fr.pixels
    ids = torch.empty((P, 8), dtype=torch.int32, device="cuda")
    w = torch.empty((P, 8), device="cuda")
    cnt = torch.empty(P, dtype=torch.uint8, device="cuda")
    q.qr_project(fr, *gdev)
    q.qr_sort(fr)
    q.qr_select(fr, ids, w, cnt)
    code, nis = q.qr_frame_status(fr)
    assert code == q.QR_ERR_CAPACITY
    assert nis > 100
    assert (cnt == 0).all()
    # retry with the reported size succeeds
    fr2 = q.frame_create(g.n, cam, q.default_params(8), nis)
    q.qr_project(fr2, *gdev)
    q.qr_sort(fr2)
    assert q.qr_frame_status(fr2) == (q.QR_OK, nis)


def test_host_buffer_render_matches_device_render():
    import torch
    from paper_2512_20927_gb300 import qrender as q
    g, f = scenes.tiny_scene()
    cam = scenes.tiny_camera()
    K, C = 8, f.shape[1]
    dev_res = H.run_gpu(g, f, cam, K=K, dense=False)
    fr = q.frame_create(g.n, cam, q.default_params(K), 1 << 20)
    nin, nout = q.qr_render_host_bytes(g.n, cam.width, cam.height, K, C, q.QR_F32)
    din = torch.empty(nin + 256, dtype=torch.uint8, device="cuda")
    dout = torch.empty(nout + 256, dtype=torch.uint8, device="cuda")
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).pin_memory()  # noqa: E731
    out_h = torch.empty((cam.width * cam.height, C), dtype=torch.float32).pin_memory()
    q.qr_render_host(fr, pin(g.mean), pin(g.log_scale), pin(g.quat), pin(g.opacity), pin(f), None,
                     q.QR_F32, C, _aligned(din), _aligned(dout), out_h)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out_h.numpy(), dev_res["out"])


def _aligned(t):
    class _A:
        def __init__(self, p):
            self._p = p

        def data_ptr(self):
            return self._p
    return _A((t.data_ptr() + 255) // 256 * 256)


def test_launch_counter_advances():
    from paper_2512_20927_gb300 import qrender as q
    before = q.qr_launch_count()
    g, f = scenes.tiny_scene(n=200)
    H.run_gpu(g, f, scenes.tiny_camera(32, 32), K=4)
    assert q.qr_launch_count() > before


@pytest.mark.parametrize("C,kind,tile", [(512, "f32", (16, 16)), (256, "f32", (8, 32)),
                                         (128, "bf16", (32, 8)), (512, "fp8", (16, 16))])
def test_dense_subtile_kernel(C, kind, tile):
    """The sub-tile dense kernel (rows of 128-512 channels; 16x4, 8x8 or 32x2
    sub-tiles, one walk per pixel, culled and skipped entries) against the
    oracle's Eq. 1, and its work counter against the oracle's walk lengths."""
    import torch
    from paper_2512_20927_gb300 import qrender as q
    g, f = H.small_room(n=20000, channels=C)
    cam = scenes.room_camera(150, 110)
    fdev = torch.from_numpy(f).cuda()
    table, scale, fdec = fdev, None, f
    if kind == "bf16":
        table = q.qr_quantize_bf16(fdev)
        fdec = oracle.bf16_decode(oracle.bf16_encode(f))
    elif kind == "fp8":
        table, scale = q.qr_quantize_fp8(fdev)
        c8, s8 = oracle.fp8_quantize_rows(f)
        fdec = oracle.fp8_dequantize_rows(c8, s8)
    params = q.default_params(8, tile_w=tile[0], tile_h=tile[1])
    res = q.render_frame(q.gaussians_to_device(g), None, cam, K=8, params=params)
    fr = res["frame"]
    P = cam.width * cam.height
    out = torch.empty((P, C), device="cuda")
    tf = torch.empty(P, device="cuda")
    counts = q.qr_dense_work(fr, table, scale, out, tf)
    torch.cuda.synchronize()
    pr, pix, ref = H.run_oracle(g, fdec, cam, 8)
    dtie = (ref.tie & compare.DENSE_TIE_BITS) != 0
    err = compare.feature_error(out.cpu().numpy(), ref.out_dense, ref.scale_dense)[~dtie]
    assert err.max() <= DENSE_TOL, err.max()
    tf_err = np.abs(tf.cpu().numpy() - ref.t_final)[~dtie]
    assert tf_err.max() <= 1e-5, tf_err.max()
    blended, executed = (int(x) for x in counts.cpu().numpy())
    want = int(ref.n_dense.sum())
    slack = int(ref.n_dense[dtie].sum()) + int(dtie.sum())
    assert abs(blended - want) <= slack, (blended, want, slack)
    assert executed >= blended * C
    print(f"dense sub-tile C={C} {kind} tile {tile}: err {err.max():.2e}, blended {blended} "
          f"(oracle {want}), executed/useful FMA {executed / max(blended * C, 1):.2f}")


@pytest.mark.parametrize("C,kind,tile", [(64, "f32", (8, 32)), (64, "bf16", (16, 16)), (64, "fp8", (32, 8)),
                                         (128, "f32", (16, 16)), (128, "fp8", (16, 16)),
                                         (256, "bf16", (32, 8)), (256, "fp8", (8, 32)),
                                         (512, "bf16", (16, 16))])
def test_dense_block_kernel_other_widths(C, kind, tile):
    """The widths and formats of the block kernel that the test above leaves out."""
    test_dense_subtile_kernel(C, kind, tile)


@pytest.mark.parametrize("kind", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("scene", ["deep", "room"])
def test_dense_kernels_agree_bit_for_bit(kind, scene):
    """Rows of 64, 128, 256 and 512 channels on the block kernel and of 192 on
    the slice kernel: the same sums and transmittances for the channels they
    share, on lists of thousands of entries too, and no timeout."""
    import torch
    from paper_2512_20927_gb300 import qrender as q
    if scene == "deep":
        g, _ = _slab_scene(6000)
        cam = scenes.tiny_camera(53, 47)
    else:
        g, _ = H.small_room(n=20000, channels=16)
        cam = scenes.room_camera(150, 110)
    x = torch.randn((g.n, 512), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    table, scale = x, None
    if kind == "bf16":
        table = q.qr_quantize_bf16(x)
    elif kind == "fp8":
        table, scale = q.qr_quantize_fp8(x)
    fr = q.render_frame(q.gaussians_to_device(g), None, cam, K=8)["frame"]

    def dense(C):
        out = torch.full((fr.pixels, C), float("nan"), device="cuda")
        T = torch.full((fr.pixels,), float("nan"), device="cuda")
        q.qr_dense(fr, table[:, :C].contiguous(), scale, out, T)
        assert q.qr_frame_status(fr)[0] == q.QR_OK
        return out, T
    want, T = dense(192)
    assert bool((T < 0.5).any()) and bool(torch.isfinite(want).all())
    for C in (64, 128, 256, 512):
        got, Tc = dense(C)
        n = min(C, 192)
        assert torch.equal(got[:, :n], want[:, :n]), C
        assert torch.equal(Tc, T) and bool(torch.isfinite(got).all()), C


@pytest.mark.parametrize("dtype,C", [("f32", 512), ("bf16", 512), ("bf16", 1024), ("fp8", 1024),
                                     ("fp8", 512)])
def test_blend_channel_chunks_bit_identical(dtype, C):
    """Splitting the rows into channel chunks across warps changes neither the
    terms nor their order per channel: every chunk count gives the same bits,
    in both pixel orders, with ragged P and counts (0 .. K)."""
    import torch
    from paper_2512_20927_gb300 import qrender as q
    rng = np.random.default_rng(C + len(dtype))
    n, W, H_, K = 4000, 53, 37, 8
    P = W * H_
    f = torch.from_numpy(rng.normal(size=(n, C)).astype(np.float32)).cuda()
    table, sc = f, None
    if dtype == "bf16":
        table = q.qr_quantize_bf16(f)
    elif dtype == "fp8":
        table, sc = q.qr_quantize_fp8(f)
    ids, w, cnt = scenes.random_selection(seed=C, pixels=P, k=K, n=n)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    ids, w, cnt = dev(ids), dev(w), dev(cnt)
    try:
        for width in (0, W):
            outs = []
            for chunks in (0, 1, 2, 4):
                q.qr_set_blend_chunks(chunks)
                o = torch.full((P, C), float("nan"), dtype=torch.float32, device="cuda")
                q.qr_blend(table, sc, ids, w, cnt, o, width=width)
                outs.append(o)
            torch.cuda.synchronize()
            for o in outs[1:]:
                assert torch.equal(o, outs[0]), (width, dtype, C)
            assert not torch.isnan(outs[0]).any()
    finally:
        q.qr_set_blend_chunks(0)
    with pytest.raises(q.QRError):
        q.qr_set_blend_chunks(3)


@pytest.mark.parametrize("K,C,dtype,width", [(8, 512, "f32", 67), (9, 512, "bf16", 67), (16, 128, "f32", 0),
                                             (16, 512, "fp8", 67), (17, 256, "f32", 67), (32, 512, "f32", 0)])
def test_blend_of_many_entries_per_group(K, C, dtype, width):
    """Pixel groups whose entries fill one, two and four sets of a warp's lanes,
    partly listed, on an image with cut groups and as consecutive pixels."""
    import torch
    from paper_2512_20927_gb300 import qrender as q
    rng = np.random.default_rng(K + C)
    n, P = 60, 67 * 35
    f = rng.normal(size=(n, C)).astype(np.float32)
    ids, w, cnt = scenes.random_selection(seed=K, pixels=P, k=K, n=n)
    fdev = torch.from_numpy(f).cuda()
    table, scale, fdec = fdev, None, f.astype(np.float64)
    if dtype == "bf16":
        table, fdec = q.qr_quantize_bf16(fdev), oracle.bf16_decode(oracle.bf16_encode(f))
    elif dtype == "fp8":
        (table, scale), fdec = q.qr_quantize_fp8(fdev), oracle.fp8_dequantize_rows(*oracle.fp8_quantize_rows(f))
    out = torch.full((P, C), float("nan"), device="cuda")
    q.qr_blend(table, scale, *(torch.from_numpy(a).cuda() for a in (ids, w, cnt)), out, width=width)
    torch.cuda.synchronize()
    want = compare.blend(ids, w, cnt, fdec)
    mag = compare.blend(ids, np.abs(w), cnt, np.abs(fdec))
    # K products and sums in FP32 (and the FP8 scale folded into the weight)
    assert (np.abs(out.cpu().numpy() - want) <= (K + 2) * 2.0 ** -23 * mag + 1e-30).all()


@pytest.mark.parametrize("w,h,K,tile", [(1, 1, 8, (16, 16)), (7, 9, 3, (16, 16)),
                                        (9, 17, 4, (32, 8)), (33, 8, 12, (8, 32)),
                                        (16, 31, 32, (32, 8)), (50, 23, 8, (8, 32))])
def test_selection_block_edges(w, h, K, tile):
    """8 x 8 blocks cut by the image's edge, every tile shape, vector and
    scalar stores (K % 4, 4-byte aligned outputs)."""
    import torch
    from paper_2512_20927_gb300 import qrender as q
    g, f = scenes.tiny_scene(seed=11, n=1500, channels=16)
    cam = scenes.tiny_camera(w, h)
    gpu = H.run_gpu(g, f, cam, K, dense=False, params_kw={"tile_w": tile[0], "tile_h": tile[1]})
    _, pix, ref = H.run_oracle(g, f, cam, K)
    H.check_frame(gpu, ref, pix, w, f, 1e-5, max_tie_frac=0.05, label=f"{w}x{h}")
    P = w * h
    ids = torch.full((P * K + 2,), -7, dtype=torch.int32, device="cuda")
    wts = torch.full((P * K + 2,), -7.0, device="cuda")
    cnt = torch.empty(P, dtype=torch.uint8, device="cuda")
    q.qr_select(gpu["frame"], ids[1:-1].view(P, K), wts[1:-1].view(P, K), cnt)
    torch.cuda.synchronize()
    assert (ids[1:-1].cpu().numpy().reshape(P, K) == gpu["ids"]).all()
    assert (wts[1:-1].cpu().numpy().reshape(P, K) == gpu["weights"]).all()
    assert (cnt.cpu().numpy() == gpu["counts"]).all()
    assert ids[0] == -7 and ids[-1] == -7 and wts[0] == -7 and wts[-1] == -7


@pytest.mark.parametrize("K,tile", [(8, (16, 16)), (5, (32, 8)), (32, (8, 32))])
def test_selection_whole_and_half_blocks_agree(K, tile):
    """The two block sizes of the selection (by the capacity of the lists per
    tile) keep the same Gaussians with the same weights on a ragged image."""
    import torch
    from paper_2512_20927_gb300 import qrender as q
    g, f = H.small_room(n=20000, channels=16)
    cam = scenes.room_camera(517, 389)
    gdev = q.gaussians_to_device(g)
    params = q.default_params(K, tile_w=tile[0], tile_h=tile[1])
    tiles = -(-517 // tile[0]) * -(-389 // tile[1])
    for rule in (q.QR_RULE_QUANTILE, q.QR_RULE_RIEMANN):
        outs = []
        for per_tile in (500, 2048):
            res = q.render_frame(gdev, None, cam, K=K, params=params, max_isect=per_tile * tiles, rule=rule)
            torch.cuda.synchronize()
            assert res["frame"].frame.max_isect == per_tile * tiles and res["n_isect"] > 0
            outs.append(res)
        for k in ("ids", "weights", "counts"):
            assert torch.equal(outs[0][k], outs[1][k]), (rule, k)
        assert int(outs[0]["counts"].max()) > 1
