"""Kernels at the sizes where their splits change: tile lists around the sort's register, warp and CTA
limits (needs a GB300)."""
import numpy as np
import pytest

from harness import gpu_run, params_pair
from ts_synth.scenes import Scene

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
