"""Kernels at the sizes where their splits change: tile lists around the sort's register, warp and CTA
limits, the chain rule around its faces per warp, the forward's pixel lists, the photometric loss's
strips (needs a GB300)."""
import numpy as np
import pytest

from harness import assert_grad, assert_images, assert_pose_grad, gpu_run, oracle_run, params_pair
from ts_synth.scenes import Scene, noise_targets, random_triangles_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 32, 33, 64, 65, 128, 129, 256, 257, 511, 512, 513, 1025, 4095, 4096, 4097, 8193])
def test_tile_sort_list_lengths(n):
    """One 8 x 8 tile that all n faces cover, at 37 depths in a random order: ascending (depth, face)."""
    rng = np.random.default_rng(n)
    z = 1.0 + 0.01 * rng.integers(0, 37, n)
    tri = np.array([[-10.0, -10.0], [10.0, -10.0], [0.0, 20.0]])
    pos = np.concatenate([np.repeat(tri[None], n, 0) * z[:, None, None], np.repeat(z[:, None, None], 3, 1)], 2)
    sc = Scene(pos.reshape(-1, 3).astype(np.float32), np.full((3 * n, 3), 0.5, np.float32),
               np.full(3 * n, 0.01, np.float32), None, np.array([[8.0, 8.0, 4.0, 4.0, 8, 8]]),
               np.array([[1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0]], np.float32))
    p, _ = params_pair(tile_w=8, tile_h=8)
    rast = gpu_run(sc, p, backward=False)["rast"]
    zb = rast.debug("zbits").cpu().numpy().view(np.uint32)
    order = np.lexsort((np.arange(n), zb))
    assert np.array_equal(rast.debug("ids").cpu().numpy().view(np.uint32)[:n], order)
    assert np.array_equal(rast.debug("keys").cpu().numpy().view(np.uint64)[:n], zb[order].astype(np.uint64))


@pytest.mark.parametrize("n_faces,n_wide", [(1, 0), (33, 33), (1025, 3), (2049, 600), (9000, 300)])
@pytest.mark.parametrize("n_views", [1, 3])
def test_tile_lists_of_wide_faces(n_faces, n_wide, n_views):
    """Binning around its rounds of faces and its queue of wide rectangles (256 a block), with rectangles on
    both sides of 128 tiles: every tile's list holds exactly the faces whose rectangle covers it, by depth."""
    rng = np.random.default_rng(n_faces + n_views)
    z = rng.uniform(1.0, 2.0, n_faces)
    size = np.where(np.arange(n_faces) < n_wide, rng.uniform(20.0, 400.0, n_faces), rng.uniform(1.0, 12.0, n_faces))
    centre = rng.uniform([0.0, 0.0], [300.0, 200.0], (n_faces, 2)) - [150.0, 100.0]
    tri = np.array([[-0.5, -0.5], [0.5, -0.5], [0.0, 0.5]])
    xy = (centre[:, None] + tri[None] * size[:, None, None]) * (z / 100.0)[:, None, None]
    pos = np.concatenate([xy, np.repeat(z[:, None, None], 3, 1)], 2)[rng.permutation(n_faces)]
    poses = np.tile([1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0.0], (n_views, 1))
    poses[:, 9] = 0.1 * np.arange(n_views)
    sc = Scene(pos.reshape(-1, 3).astype(np.float32), np.full((3 * n_faces, 3), 0.5, np.float32),
               np.full(3 * n_faces, 0.5, np.float32), None, np.array([[100.0, 100.0, 150.0, 100.0, 300, 200]] * n_views),
               poses.astype(np.float32))
    p, _ = params_pair(tile_w=8, tile_h=8)
    rast = gpu_run(sc, p, backward=False, pair_capacity=2_000_000)["rast"]
    rect = rast.debug("rect").cpu().numpy().view(np.int16).reshape(n_views, n_faces, 4)
    zb = rast.debug("zbits").cpu().numpy().view(np.uint32).reshape(n_views, n_faces)
    ids, ranges = rast.debug("ids").cpu().numpy().view(np.uint32), rast.debug("ranges").cpu().numpy()
    ranges = ranges.view(np.uint32).reshape(n_views, 25, 38, 2)
    for v in range(n_views):
        r = rect[v].astype(np.int64)
        for ty in range(25):
            for tx in range(38):
                on = np.flatnonzero((r[:, 0] >= 0) & (r[:, 0] <= tx) & (tx <= r[:, 2]) & (r[:, 1] <= ty) & (ty <= r[:, 3]))
                want = on[np.lexsort((on, zb[v][on]))]
                assert np.array_equal(ids[ranges[v, ty, tx, 0]:ranges[v, ty, tx, 1]], want), (v, ty, tx)


@pytest.mark.parametrize("n_faces", [1, 7, 33, 200])
@pytest.mark.parametrize("n_views", [1, 2, 3, 7, 8, 33])
def test_chain_rule_views_and_faces(oracle, n_views, n_faces):
    """The chain rule with map gradients at every number of faces a warp takes, ragged ones included,
    and the form without map gradients, whose pose gradient sums in another order."""
    sc = random_triangles_scene(seed=n_faces, n_faces=n_faces, W=40, H=30, f=40.0, z_lo=1.0, z_hi=2.0, side_lo=0.2,
                                side_hi=0.5)
    poses = np.repeat(sc.poses[:1], n_views, axis=0).copy()
    poses[:, 9] = np.linspace(-0.6, 0.6, n_views)  # some faces leave some views
    sc = Scene(sc.pos, sc.col, sc.opa, None, np.repeat(sc.cams[:1], n_views, axis=0), poses)
    sc.tgt_color, sc.tgt_depth = noise_targets(3, sc.cams)
    sc.pair_capacity = 64 * n_views * n_faces
    p, po = params_pair(sigma=1.0)
    r = oracle_run(oracle, sc, po)
    g = gpu_run(sc, p, dC=r["dC_used"], dD=r["dD_used"])
    for k in ("dpos", "dcol", "dopa"):
        assert_grad(g[k], r[k], k)
    assert_pose_grad(g["dtau"], r["dtau"], r["dtau_abs"])
    # the same backward without map gradients
    import torch
    import paper_2605_31419_gb300 as ts
    rast = g["rast"]
    rast.forward(ts.Map.from_numpy(sc.pos, sc.col, sc.opa), ts.poses_tensor(sc.poses))
    dev = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float32, device="cuda")  # noqa: E731
    rast.backward(dev(r["dC_used"]), dev(r["dD_used"]))
    assert_pose_grad(rast.pose_grad().cpu().numpy().astype(np.float64), r["dtau"], r["dtau_abs"])


@pytest.mark.parametrize("size", [(1, 1), (7, 3), (8, 4), (17, 9), (33, 18)])
@pytest.mark.parametrize("n_faces", [1, 31, 32, 33, 65, 129])
def test_forward_pixel_lists(oracle, n_faces, size):
    """The per-pixel face lists of the forward at ragged images and around 32 and 64 staged faces, with faces
    far larger than the image (vertices close to the camera) among them."""
    W, H = size
    sc = random_triangles_scene(seed=n_faces + W, n_faces=n_faces, W=W, H=H, f=20.0, z_lo=0.2, z_hi=2.0, side_lo=0.05,
                                side_hi=0.8, opa_lo=0.05, opa_hi=0.6, target_seed=None)
    p, po = params_pair()
    g = gpu_run(sc, p, backward=False, pair_capacity=4096)
    r = oracle_run(oracle, sc, po, backward=False)
    for k in ("color", "depth", "alpha", "T_final"):
        assert_images(g[k], r[k], k)
    assert np.array_equal(g["n_last"], r["n_last"])


def test_pho_loss_strip_edges(oracle):
    """The photometric loss around its strips: widths and heights on both sides of 64 columns and of 22 rows
    (the strip height of a small batch), and images smaller than the window."""
    from test_gpu_pho import _cams, _check, _gpu, _scene_arrays
    from ts_synth.scenes import loss_images
    cams = _cams([(63, 21), (64, 22), (65, 23), (128, 44), (129, 45), (5, 3), (3, 30), (70, 1)])
    C, D, tC, tD = loss_images(21, cams)
    _check(cams, _gpu(cams, C, D, tC, tD, 0.2, 0.05), oracle.pho_loss(_scene_arrays(cams), C, D, tC, tD, 0.2, 0.05))
