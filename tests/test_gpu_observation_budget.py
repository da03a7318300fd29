"""The device memory that an observation through the voxel hash needs at its peak: the
scene and either the hash's scratch or the two bitmaps of its cell box, not both."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_hash_build_peak():
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    H, W, f = 480, 640, 600.0
    rng = np.random.default_rng(2)
    depth = rng.integers(10000, 10100, (H, W)).astype(np.uint16)
    depth[::7, ::5] = 20000                       # some 1.2e8 cells of 3 mm: the hash, with bitmaps of 15 MB
    rgb = np.zeros((H, W, 3), np.uint8)
    params = P.perch_default_params(delta_m=0.003, color_check=0)

    def scene(ctx):
        return P.perch_set_observation(ctx.ctx, depth, rgb, None, f, f, W / 2.0, H / 2.0, params)

    def fits(budget):
        try:
            with P.Context(0, hbm_budget_bytes=budget) as ctx:
                scene(ctx)
            return True
        except P.PerchError as e:
            assert e.status == -3
            return False

    with P.Context(0) as ctx:
        base = ctx.hbm_used
        scene(ctx)
        kept = ctx.hbm_used - base                # the scene, and the colours' scratch
    cells = 1
    z = depth / 10000.0
    u, v = np.meshgrid(np.arange(W) - W / 2.0, np.arange(H) - H / 2.0)
    for x in (u * z / f, v * z / f, z):
        c = np.floor(x / (0.003 * (1 + 1 / 64)))
        cells *= int(c.max() - c.min()) + 3
    assert 1 << 24 < cells < 1 << 27
    bitmap = cells // 8
    cap = 1 << int(2 * H * W - 1).bit_length()    # slots of the hash build's table
    scratch = cap * (16 + 8 + 4 + 4 + 4) + 4 * H * W
    assert kept > 16 * H * W and scratch > bitmap
    # at the scratch's peak the scene's own bitmap is not there yet; 64 KB of slack for
    # alignment and small arrays
    assert fits(base + kept - bitmap + scratch + (64 << 10))
