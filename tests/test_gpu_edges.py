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
