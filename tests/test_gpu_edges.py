"""Hand-overs between the threads of a CTA, totals beyond 32 bits and values at the ends of FP32's range
(needs a GB300)."""
import numpy as np
import pytest

from harness import pack_targets, params_pair
from ts_synth.scenes import Scene, random_triangles_scene

pytestmark = pytest.mark.gpu


def _two_views(sc):
    poses = np.repeat(sc.poses[:1], 2, axis=0).copy()
    poses[1, 9] = 0.15
    return Scene(sc.pos, sc.col, sc.opa, None, np.repeat(sc.cams[:1], 2, axis=0), poses)


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("fused", [False, True])
def test_coverage_of_lists_of_many_stages(fused, persistent):
    """The faces' coverage counts do not depend on the stage size: lists of 129 to 256 faces (two stages of
    128, so that no stage's records are replaced) give the counts that eight stages of 32 give, whose buffers
    are copied over while the counts of the stage before the last one copied are still written out."""
    import torch
    import paper_2605_31419_gb300 as ts
    sc = _two_views(random_triangles_scene(seed=12, n_faces=256, W=80, H=48, f=160.0, side_lo=1.5, side_hi=3.0,
                                           z_lo=2.0, z_hi=3.0, opa_lo=0.02, opa_hi=0.05, target_seed=None))
    m, poses = ts.Map.from_numpy(sc.pos, sc.col, sc.opa), ts.poses_tensor(sc.poses)
    got = {}
    for S in (128, 32, 64):
        p, _ = params_pair(flags=ts.TS_FLAG_STATS | (ts.TS_FLAG_PERSISTENT if persistent else 0), tris_per_stage=S)
        r = ts.Rasterizer(sc.cams, sc.n_faces, p, pair_capacity=200_000)
        zeros = torch.zeros_like(r.color), torch.zeros_like(r.depth)
        for _ in range(3):
            if fused:
                r.project(m, poses)
                r.bin()
                r.step_l1(*zeros, 0.05, None)
            else:
                r.forward(m, poses)
            st = r.face_stats()
            assert r.counters()["error_bits"] == 0
            cov = st["coverage"].cpu().numpy().copy()
            assert int(cov.sum()) == r.counters()["fwd_contrib"]
            assert np.array_equal(cov, got.setdefault("cov", cov)), S
        longest = r.debug("ranges").cpu().numpy().view(np.uint32).reshape(-1, 2)
        assert 128 < int((longest[:, 1] - longest[:, 0]).max()) <= 256


@pytest.mark.parametrize("persistent", [False, True])
def test_fused_step_of_short_lists(persistent):
    """Lists of one stage stay staged from the forward to the backward of the fused step, whose first batch
    then reads other lanes' pixel state with no barrier of the staging between: the gradients are those of
    the separate calls, run after run."""
    import torch
    import paper_2605_31419_gb300 as ts
    sc = random_triangles_scene(seed=15, n_faces=400, W=96, H=64, f=70.0, side_lo=0.1, side_hi=0.6)
    p, _ = params_pair(flags=ts.TS_FLAG_PERSISTENT if persistent else 0)
    m, poses = ts.Map.from_numpy(sc.pos, sc.col, sc.opa), ts.poses_tensor(sc.poses)
    tc, td = (torch.as_tensor(np.asarray(x), dtype=torch.float32, device="cuda") for x in pack_targets(sc))
    r = ts.Rasterizer(sc.cams, sc.n_faces, p, pair_capacity=100_000)
    r.forward(m, poses)
    _, dC, dD = r.l1_loss(tc, td)
    want = m.zeros_like()
    r.backward(dC, dD, None, want)
    lists = r.debug("ranges").cpu().numpy().view(np.uint32).reshape(-1, 2)
    assert 32 < int((lists[:, 1] - lists[:, 0]).max()) <= 64
    for _ in range(10):
        r.project(m, poses)
        r.bin()
        g = m.zeros_like()
        r.step_l1(tc, td, 0.05, g)
        for k in ("pos", "col", "opa"):
            a, b = getattr(g, k), getattr(want, k)
            # the faces' sums are the same terms in another order (atomics): some 300 roundings of 2^-24
            assert float((a - b).abs().max()) <= 2e-5 * float(b.abs().max()), k


def _random_soup(rng, n_faces, n_views, W, H, f):
    """n_faces small triangles on all sides of n_views cameras near the origin, a quarter of them in view."""
    centre = rng.normal(size=(n_faces, 3))
    centre *= rng.uniform(0.5, 4.0, (n_faces, 1)) / np.linalg.norm(centre, axis=1, keepdims=True)
    pos = centre[:, None] + rng.uniform(-0.06, 0.06, (n_faces, 3, 3))
    poses = np.tile(np.array([1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0.0]), (n_views, 1))
    poses[:, 9:] = rng.uniform(-0.3, 0.3, (n_views, 3))
    return Scene(pos.reshape(-1, 3).astype(np.float32), rng.random((3 * n_faces, 3), dtype=np.float32),
                 rng.uniform(0.5, 1.0, 3 * n_faces).astype(np.float32), None,
                 np.array([[f, f, W / 2, H / 2, W, H]] * n_views), poses.astype(np.float32))


@pytest.mark.parametrize("n_views,n_faces", [(9, 70_001), (2, 1_900_033), (1, 2_300_017)])
def test_projection_queue_of_large_maps(oracle, n_views, n_faces):
    """Faces that can be seen are queued over views and, on maps of millions of faces, over several groups of
    32 faces of a warp: every (view, face)'s tile box, tile count and depth key bit for bit, ragged ends
    included, and records that hold the projected vertices."""
    import paper_2605_31419_gb300 as ts
    from oracle.oracle import SceneArrays
    sc = _random_soup(np.random.default_rng(n_views), n_faces, n_views, 64, 48, 30.0)
    p, po = params_pair()
    r = ts.Rasterizer(sc.cams, n_faces, p)
    r.project(ts.Map.from_numpy(sc.pos, sc.col, sc.opa), ts.poses_tensor(sc.poses))
    want = oracle.project(SceneArrays.of(sc), po)
    count = r.debug("count").cpu().numpy().view(np.uint32)
    assert np.array_equal(count, want["count"])
    seen = np.flatnonzero(want["count"])
    assert len(seen) > 0.05 * n_views * n_faces
    assert np.array_equal(r.debug("rect").cpu().numpy().view(np.int16).reshape(-1, 4)[seen], want["rect"][seen])
    assert np.array_equal(r.debug("zbits").cpu().numpy().view(np.uint32)[seen], want["zbits"][seen])
    rec = r.debug("records").cpu().numpy().reshape(-1, 32)
    uvz = want["uvz"].reshape(-1, 9)[seen]
    assert np.array_equal(rec[seen][:, [0, 1, 2, 3, 4, 5, 26, 27, 28]], uvz.astype(np.float32))
    assert r.counters()["n_visible"] == len(seen)


@pytest.mark.parametrize("n_faces,size,tri", [
    # 2^27 faces over the 32 tiles of one group of the count matrix
    (1 << 27, (256, 8), [[-10.0, -10.0], [600.0, -10.0], [-10.0, 40.0]]),
    # 2^20 faces over the first 4096 tiles of a view that takes the global counts
    (1 << 20, (4096, 2560), [[0.2, 0.2], [4095.8, 0.2], [0.2, 63.8]]),
])
def test_pair_total_beyond_32_bits(n_faces, size, tri):
    """2^32 pairs in one group of tiles: the count is exact and latches the capacity error, also when the
    binning runs again, and the ranges stay inside the pair list."""
    import torch
    import paper_2605_31419_gb300 as ts
    W, H = size
    pos = np.array([[(u - W / 2) / 100.0, (v - H / 2) / 100.0, 1.0] for u, v in tri], np.float32).T
    m = ts.Map(torch.as_tensor(pos, device="cuda").contiguous(), torch.full((3, 3), 0.5, device="cuda"),
               torch.full((3,), 0.5, device="cuda"),
               torch.arange(3, dtype=torch.int32, device="cuda").repeat(n_faces, 1).contiguous())
    p, _ = params_pair(tile_w=8, tile_h=8, flags=ts.TS_FLAG_FORWARD_ONLY)
    r = ts.Rasterizer(np.array([[100.0, 100.0, W / 2, H / 2, W, H]]), n_faces, p, pair_capacity=1024)
    r.project(m, ts.poses_tensor(np.array([[1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0]], np.float32)))
    for _ in range(2):
        r.bin()
        c = r.counters(raise_on_error=False)
        assert c["n_pairs"] == 1 << 32 and c["error_bits"] == 1
        lists = r.debug("ranges").cpu().numpy().view(np.uint32).reshape(-1, 2).astype(np.int64)
        assert (lists[:, 0] <= lists[:, 1]).all() and (lists[:, 1] <= 1024).all()


def test_pho_loss_where_ssim_products_reach_the_range():
    """SSIM divides by a product of two sums of squares.  Where that product overflows (values of 2e10) the
    terms vanish and L1 is left; where its reciprocal is below the normal range (4e9) equal images still have
    SSIM = 1.  Both finite."""
    import torch
    import paper_2605_31419_gb300 as ts
    W, H, lam = 96, 80, 0.2
    r = ts.Rasterizer(np.array([[50.0, 50.0, W / 2, H / 2, W, H]]), 0)
    rng = np.random.default_rng(4)
    x = torch.as_tensor(rng.uniform(-2e10, 2e10, 3 * W * H), dtype=torch.float32, device="cuda")
    td = torch.zeros_like(r.depth)
    r.color.copy_(x)
    r.depth.zero_()
    loss, dC, _ = r.pho_loss(torch.zeros_like(x), td, lam)
    want = (1 - lam) * float(x.double().abs().mean()) + lam
    assert abs(float(loss[0]) - want) <= 1e-5 * want
    # SSIM's own gradient is below 1e-9 of the L1 one's
    assert torch.allclose(dC, (1 - lam) / (3 * W * H) * torch.sign(x), rtol=1e-6, atol=0)
    x = torch.as_tensor(4.16e9 * rng.uniform(0.5, 1.5, 3 * W * H), dtype=torch.float32, device="cuda")
    r.color.copy_(x)
    loss, dC, _ = r.pho_loss(x, td, lam)
    assert abs(float(loss[0])) < 1e-3 and bool(torch.isfinite(dC).all())


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8), (16, 32), (32, 16)], ids=lambda t: f"{t[0]}x{t[1]}")
def test_side_array_at_every_tile_shape(tile, persistent):
    """Images with normals and the gradients of all of them at every tile shape (each compiled for its own
    register budget) against those at 16 x 8: images bit for bit, gradients to the order of the faces' sums."""
    import torch
    import paper_2605_31419_gb300 as ts
    sc = _two_views(random_triangles_scene(seed=23, n_faces=600, W=101, H=67, f=60.0, side_lo=0.2, side_hi=0.8))
    m, poses = ts.Map.from_numpy(sc.pos, sc.col, sc.opa), ts.poses_tensor(sc.poses)
    out = []
    for tw, th in ((16, 8), tile):
        flags = ts.TS_FLAG_NORMALS | (ts.TS_FLAG_PERSISTENT if persistent else 0)
        r = ts.Rasterizer(sc.cams, sc.n_faces, ts.ts_default_params(tile_w=tw, tile_h=th, flags=flags), pair_capacity=400_000)
        images = [t.clone() for t in r.forward(m, poses)] + [r.normal.clone()]
        gen = torch.Generator(device="cuda").manual_seed(5)
        dC, dN = (torch.rand(3 * r.n_pix, generator=gen, device="cuda") - 0.5 for _ in range(2))
        dD, dA = (torch.rand(r.n_pix, generator=gen, device="cuda") - 0.5 for _ in range(2))
        g = m.zeros_like()
        r.backward(dC, dD, dA, g, dN=dN)
        assert r.counters()["error_bits"] == 0
        out.append((images, [g.pos, g.col, g.opa]))
    for a, b in zip(*(o[0] for o in out)):
        assert torch.equal(a, b)
    for a, b in zip(*(o[1] for o in out)):
        # some 300 roundings of 2^-24 in another order
        assert float((a - b).abs().max()) <= 2e-5 * float(a.abs().max())


def _padded(sc, n_faces, indexed):
    """The scene's map with faces behind every camera between its first and its second half: n_faces in all,
    and the places of the scene's own."""
    M = sc.n_faces
    keep = np.concatenate([np.arange(M // 2), np.arange(n_faces - (M - M // 2), n_faces)])
    if indexed:
        N = len(sc.pos)
        behind = np.array([[0, 0, -5], [0.1, 0, -5], [0, 0.1, -5]], np.float32)
        faces = np.tile(np.arange(N, N + 3, dtype=np.int32), (n_faces, 1))
        faces[keep] = sc.faces
        sigma = np.full(n_faces, 0.7, np.float32)
        sigma[keep] = sc.sigma
        out = Scene(np.concatenate([sc.pos, behind]), np.concatenate([sc.col, sc.col[:3]]),
                    np.concatenate([sc.opa, sc.opa[:3]]), faces, sc.cams, sc.poses)
        out.sigma = sigma
        return out, keep, np.arange(N)
    rows = (3 * keep[:, None] + np.arange(3)).reshape(-1)
    pos = np.tile(np.array([[0, 0, -5], [0.1, 0, -5], [0, 0.1, -5]], np.float32), (n_faces, 1))
    col, opa = np.full((3 * n_faces, 3), 0.5, np.float32), np.full(3 * n_faces, 0.5, np.float32)
    pos[rows], col[rows], opa[rows] = sc.pos, sc.col, sc.opa
    return Scene(pos, col, opa, None, sc.cams, sc.poses), keep, rows


@pytest.mark.parametrize("n_faces,n_views,indexed", [
    (5_001, 3, True), (4_865, 110, False), (5_001, 256, True),      # 4 faces a warp of the chain rule up to 110 views, 2
    (12_002, 2, False), (12_002, 110, True), (9_729, 111, False),   # 8 up to 110 views
    (19_457, 2, False), (19_500, 68, True), (19_457, 69, False),    # 16 up to 68
    (38_913, 1, True), (38_950, 23, False), (38_913, 24, True),     # 32 up to 23
    (49_152, 2, False),                                             # 256 faces a warp, pose only
    (65_601, 1, False), (65_600, 3, True), (140_003, 2, False),     # 65 and more face blocks; 512 faces a warp, pose only
])
def test_padded_maps(n_faces, n_views, indexed):
    """A map of 1000 faces, and the same faces at the two ends of a large map whose other faces nobody sees: the
    same images and tile lists, and the same gradients with and without map gradients, whatever number of faces
    a block bins and a warp of the chain rule takes."""
    import torch
    import paper_2605_31419_gb300 as ts
    sc = random_triangles_scene(seed=n_views, n_faces=1000, W=64, H=48, f=50.0, side_lo=0.1, side_hi=0.4, z_lo=1.0, z_hi=3.0)
    poses = np.repeat(sc.poses[:1], n_views, axis=0).copy()
    poses[:, 9] = np.linspace(-0.8, 0.8, n_views) if n_views > 1 else 0.0
    faces = None
    if indexed:  # every vertex shared by about three faces
        faces = np.random.default_rng(7).permutation(3000).astype(np.int32).reshape(-1, 3)
        faces[1:, 0] = faces[:-1, 2]
        pos = sc.pos.copy()
        pos[faces[:, 1]] = pos[faces[:, 0]] + np.float32([0.2, 0.03, 0.02])
        pos[faces[:, 2]] = pos[faces[:, 0]] + np.float32([0.05, 0.25, -0.03])
        sc.pos[:] = pos
    sc = Scene(sc.pos, sc.col, sc.opa, faces, np.repeat(sc.cams[:1], n_views, axis=0), poses)
    sc.sigma = np.random.default_rng(8).uniform(0.5, 1.2, 1000).astype(np.float32) if indexed else None
    big, keep, rows = _padded(sc, n_faces, indexed)
    flags = ts.TS_FLAG_MIN_OPACITY | ts.TS_FLAG_FACE_SIGMA if indexed else 0
    p, _ = params_pair(flags=flags)
    out = []
    for s in (sc, big):
        r = ts.Rasterizer(s.cams, s.n_faces, p, pair_capacity=200 * 1000 * n_views)
        m = ts.Map.from_numpy(s.pos, s.col, s.opa, s.faces, sigma=getattr(s, "sigma", None))
        d = {"images": [t.clone() for t in r.forward(m, ts.poses_tensor(s.poses))]}
        n = r.counters()["n_pairs"]
        d["ids"], d["ranges"] = r.debug("ids")[:n].cpu().numpy().copy(), r.debug("ranges").cpu().numpy().copy()
        gen = torch.Generator(device="cuda").manual_seed(5)
        dC, dD = torch.rand(3 * r.n_pix, generator=gen, device="cuda") - 0.5, torch.rand(r.n_pix, generator=gen, device="cuda") - 0.5
        g = m.zeros_like()
        r.backward(dC, dD, None, g)
        d["dtau"] = r.pose_grad().cpu().numpy().copy()
        d["grad"] = [t.cpu().numpy() for t in (g.pos, g.col, g.opa)] + ([g.sigma.cpu().numpy()] if indexed else [])
        r.forward(m, ts.poses_tensor(s.poses))
        r.backward(dC, dD)
        d["pose"] = r.pose_grad().cpu().numpy().copy()
        assert r.counters()["error_bits"] == 0 and n > 0
        out.append(d)
    a, b = out
    assert all(torch.equal(x, y) for x, y in zip(a["images"], b["images"]))
    assert np.array_equal(keep[a["ids"]], b["ids"]) and np.array_equal(a["ranges"], b["ranges"])
    for i, (x, y) in enumerate(zip(a["grad"], b["grad"])):
        at = y[keep] if i == 3 else y[..., rows]
        assert np.abs(x).max() > 0 and np.abs(x - at).max() <= 2e-5 * np.abs(x).max(), i  # the faces' sums in another order
        rest = np.ones(y.shape[-1], bool)
        rest[keep if i == 3 else rows] = False
        assert not y[..., rest].any(), i
    # sums over some 3000 vertices of such terms, which cancel in part
    for x, y in ((a["dtau"], b["dtau"]), (a["pose"], b["pose"]), (a["dtau"], a["pose"])):
        assert np.abs(x - y).max() <= 1e-4 * np.abs(x).max()


@pytest.mark.parametrize("n_views,n_faces,size", [
    (1, 700, (1021, 1030)),    # 16,512 tiles, one row of the count matrix: groups of 256 tiles, a tile per warp of the sort
    (3, 1500, (1021, 1019)),   # 49,152 tiles, two rows: two tiles per warp
    (5, 8200, (809, 803)),     # 51,510 tiles, nine rows: groups of 32
    (3, 900, (1090, 1011)),    # 52,197 tiles: one left for the last warp, a last group that is not full
])
def test_tile_lists_of_many_tiles(n_views, n_faces, size):
    """Every tile's list of views of many tiles, most of them empty and some with more than 512 faces: the whole
    pair list and the ranges against the faces' rectangles."""
    import paper_2605_31419_gb300 as ts
    W, H = size
    rng = np.random.default_rng(n_faces)
    z = rng.uniform(1.0, 2.0, n_faces)
    z[::3] = np.float32(1.5)  # ties go by the face
    centre = rng.uniform([0.0, 0.0], [W, H], (n_faces, 2))
    centre[:600] = rng.normal([0.7 * W, 0.3 * H], 5.0, (600, 2))  # a heap
    side = rng.uniform(2.0, 40.0, n_faces)
    tri = np.array([[-0.5, -0.5], [0.5, -0.5], [0.0, 0.5]])
    xy = (centre - [W / 2, H / 2])[:, None] + tri[None] * side[:, None, None]
    pos = np.concatenate([xy * (z / 500.0)[:, None, None], np.repeat(z[:, None, None], 3, 1)], 2)
    poses = np.tile([1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0.0], (n_views, 1))
    poses[:, 9] = 0.3 * np.arange(n_views)
    m = ts.Map.from_numpy(pos.reshape(-1, 3).astype(np.float32), np.full((3 * n_faces, 3), 0.5, np.float32),
                          np.full(3 * n_faces, 0.5, np.float32))
    r = ts.Rasterizer(np.array([[500.0, 500.0, W / 2, H / 2, W, H]] * n_views), n_faces,
                      ts.ts_default_params(tile_w=8, tile_h=8), pair_capacity=2_000_000)
    r.project(m, ts.poses_tensor(poses.astype(np.float32)))
    r.bin()
    TX, TY = (W + 7) // 8, (H + 7) // 8
    rect = r.debug("rect").cpu().numpy().view(np.int16).reshape(n_views * n_faces, 4).astype(np.int64)
    on = np.flatnonzero(rect[:, 0] >= 0)
    wid, hei = rect[on, 2] - rect[on, 0] + 1, rect[on, 3] - rect[on, 1] + 1
    n = wid * hei
    of = np.repeat(on, n)
    k = np.arange(n.sum()) - np.repeat(np.cumsum(n) - n, n)
    w = np.repeat(wid, n)
    tile = of // n_faces * (TX * TY) + (rect[of, 1] + k // w) * TX + rect[of, 0] + k % w
    zb = r.debug("zbits").cpu().numpy().view(np.uint32)[of].astype(np.uint64)
    order = np.lexsort((of % n_faces, zb, tile))
    total = len(order)
    assert r.counters()["n_pairs"] == total and r.counters()["error_bits"] == 0
    assert np.array_equal(r.debug("ids").cpu().numpy().view(np.uint32)[:total], (of % n_faces)[order])
    assert np.array_equal(r.debug("keys").cpu().numpy().view(np.uint64)[:total],
                          (tile[order].astype(np.uint64) << np.uint64(32)) | zb[order])
    ends = np.searchsorted(tile[order], np.arange(n_views * TX * TY), side="right")
    starts = np.searchsorted(tile[order], np.arange(n_views * TX * TY), side="left")
    assert np.array_equal(r.debug("ranges").cpu().numpy().view(np.uint32).reshape(-1, 2), np.stack([starts, ends], 1))
    assert (ends - starts).max() > 512


def test_losses_do_not_depend_on_the_batch():
    """The L1 and the normal loss of a view, and their gradients, bit for bit alone and among others (values of
    many magnitudes, so that another order of the sums shows)."""
    import torch
    import paper_2605_31419_gb300 as ts
    sizes = [(640, 480)] * 4 + [(317, 239)] + [(640, 480)] * 4

    def run(views, tensors):
        r = ts.Rasterizer(np.array([[100.0, 100.0, W / 2, H / 2, W, H] for W, H in views]), 0,
                          ts.ts_default_params(flags=ts.TS_FLAG_NORMALS))
        C, D, N, tC, tD, tN = (torch.cat([t[i] for t in tensors]) for i in range(6))
        r.color.copy_(C), r.depth.copy_(D), r.normal.copy_(N)
        loss, dC, dD = (t.clone() for t in r.l1_loss(tC, tD))
        nloss, dN = r.normal_loss(tN)[:2]
        return [t.cpu() for t in (loss, dC, dD, nloss, dN)]

    gen = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda n: torch.exp(3 * torch.randn(n, generator=gen, device="cuda"))  # noqa: E731
    data = [[rnd(k * W * H) for k in (3, 1, 3, 3, 1, 3)] for W, H in sizes]
    whole = run(sizes, data)
    off = np.cumsum([0] + [W * H for W, H in sizes])
    for v in range(len(sizes)):
        alone = run([sizes[v]], [data[v]])
        a, b = off[v], off[v + 1]
        parts = (whole[0][v:v + 1], whole[1][3 * a:3 * b], whole[2][a:b], whole[3][v:v + 1], whole[4][3 * a:3 * b])
        assert all(torch.equal(x, y) for x, y in zip(alone, parts)), v


def test_pose_gradient_after_another_plans_step():
    """The pose partials are the plan's own: a small plan's step on the same workspace, which ends before the large
    plan's partials, leaves the large plan's pose gradient as it is."""
    import torch
    import paper_2605_31419_gb300 as ts
    plans = []
    for n, V in ((3000, 2), (40, 1)):
        sc = random_triangles_scene(seed=n, n_faces=n, W=64, H=48, f=60.0)
        poses = np.repeat(sc.poses[:1], V, axis=0).copy()
        poses[:, 9] = 0.1 * np.arange(V)
        r = ts.Rasterizer(np.repeat(sc.cams[:1], V, axis=0), n, pair_capacity=200 * n)
        plans.append((r, ts.Map.from_numpy(sc.pos, sc.col, sc.opa), ts.poses_tensor(poses)))
    large, small = plans
    assert small[0].ws_bytes < 3000 * 2 * 128  # inside the large plan's records
    small[0].ws = large[0].ws

    def step(r, m, poses):
        r.forward(m, poses)
        r.backward(torch.ones_like(r.color), torch.ones_like(r.depth), None, m.zeros_like())

    step(*large)
    want = large[0].pose_grad().clone()
    step(*small)
    small[0].pose_grad()
    assert float(want.abs().max()) > 0 and torch.equal(large[0].pose_grad(), want)


@pytest.mark.parametrize("normals", [False, True])
def test_large_faces_are_summed_in_few_additions(oracle, normals):
    """Eight faces that cover 2048 sub-blocks of 32 pixels in full: each sub-block adds a face's 32 terms to its
    slot once.  n FP32 additions of like terms in any order leave a sum off by about sqrt(n / 3) roundings (each
    2^-23 0.72 / sqrt(12) of it on average), 6.5e-7 for 2048 and 1.3e-6 for four times as many; the error over the
    72 colour sums has to lie below what twice as many would leave."""
    import torch
    import paper_2605_31419_gb300 as ts
    from oracle.oracle import SceneArrays
    rng = np.random.default_rng(2)
    W = H = 256
    f, M = 200.0, 8
    z = np.linspace(1.0, 2.0, M)
    tri = np.array([[-300.0, -300.0], [1000.0, -300.0], [-300.0, 1000.0]]) + rng.uniform(-40, 40, (M, 3, 2))
    pos = np.concatenate([(tri - [W / 2, H / 2]) * (z / f)[:, None, None], np.repeat(z[:, None, None], 3, 1)], 2)
    sc = Scene(pos.reshape(-1, 3).astype(np.float32), rng.uniform(0.2, 0.8, (3 * M, 3)).astype(np.float32),
               rng.uniform(0.1, 0.3, 3 * M).astype(np.float32), None, np.array([[f, f, W / 2, H / 2, W, H]]),
               np.array([[1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0]], np.float32))
    p, po = params_pair(flags=ts.TS_FLAG_NORMALS if normals else 0)
    r = ts.Rasterizer(sc.cams, M, p, pair_capacity=100_000)
    m = ts.Map.from_numpy(sc.pos, sc.col, sc.opa)
    r.forward(m, ts.poses_tensor(sc.poses))
    assert r.counters()["fwd_contrib"] == M * W * H
    dC = rng.uniform(0.5, 1.0, 3 * W * H).astype(np.float32)
    want = oracle.backward(SceneArrays.of(sc), po, dC.astype(np.float64), np.zeros(W * H))["dcol"].T
    err = []
    for _ in range(4):
        g = m.zeros_like()
        r.forward(m, ts.poses_tensor(sc.poses))
        r.backward(torch.as_tensor(dC, device="cuda"), torch.zeros_like(r.depth), None, g)
        err.append(g.col.cpu().numpy().astype(np.float64) / want - 1)
    rms = float(np.sqrt(np.mean(np.square(err))))
    assert rms <= np.sqrt(2 * 2048 / 3) * 2.0 ** -23 * 0.72 / np.sqrt(12), rms


def test_photometric_loss_of_tall_strips():
    """A batch of 80 views of 310 x 300 walks strips of 246 rows (and 54 below them) where one view alone takes
    22: the images' gradients bit for bit, the losses to the rounding of their sums."""
    import torch
    import paper_2605_31419_gb300 as ts
    W, H, V = 310, 300, 80
    gen = torch.Generator(device="cuda").manual_seed(9)
    C, tC = (torch.rand(V, 3 * W * H, generator=gen, device="cuda") for _ in range(2))
    D, tD = (torch.rand(V, W * H, generator=gen, device="cuda") for _ in range(2))
    tD[tD < 0.1] = 0.0

    def run(views):
        r = ts.Rasterizer(np.array([[50.0, 50.0, W / 2, H / 2, W, H]] * len(views)), 0)
        r.color.copy_(C[views].reshape(-1)), r.depth.copy_(D[views].reshape(-1))
        loss, dC, dD = r.pho_loss(tC[views].reshape(-1), tD[views].reshape(-1), 0.2)
        return loss, dC.view(len(views), -1), dD.view(len(views), -1)

    loss, dC, dD = run(list(range(V)))
    for v in (0, 37, 79):
        a, b, c = run([v])
        assert torch.equal(b[0], dC[v]) and torch.equal(c[0], dD[v]), v
        # sums of 90,000 x 3 terms: partial sums of at most 64 x 246 of them in 32 bits
        assert abs(float(a[0]) - float(loss[v])) <= 2e-6 * abs(float(a[0]))
