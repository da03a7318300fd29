"""The rasteriser of images over 1023 pixels, which have no vertex cache: triangle
counts around a warp's 32, pixel boxes from a fraction of a sample to thousands, 32- and
64-bit keys, tiles smaller than the render, wide and tall.  Key buffers are bit-exact
against the oracle."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes
from test_gpu_raster import _meshes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(1200, 388), (97, 1500)])
@pytest.mark.parametrize("zbuf_words", [7064, 1024])
@pytest.mark.parametrize("name", ["tris1", "tris31", "tris33", "tris65", "coarse", "wedges", "slivers", "fine"])
def test_keys_without_the_vertex_cache(oracle, name, zbuf_words, size):
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    W, H = size
    f = 150.0
    depth = np.full((H, W), 6000, np.uint16)
    rgb = np.zeros((H, W, 3), np.uint8)
    mesh = _meshes()[name]
    rng = np.random.default_rng(17)
    om = oracle.OracleMesh.from_mesh(mesh)
    osc = oracle.OracleScene(depth, rgb, None, f, f, W / 2.0, H / 2.0)
    with P.Context(0) as ctx:
        ctx.set_launch_config(256, zbuf_words)
        sid = P.perch_set_observation(ctx.ctx, depth, rgb, None, f, f, W / 2.0, H / 2.0, P.perch_default_params())
        mid = ctx.load_mesh(mesh)
        for z in (0.12, 0.3, 0.8, 6.6):              # the last with 64-bit keys
            r = scenes.random_rotation(rng)
            pose = np.concatenate([r, (rng.normal(size=3) * 0.02 + [0, 0, z])[:, None]], 1).astype(np.float32).reshape(12)
            for roi in ((0, 0, W, H), (W // 2 - 21, H // 2 - 30, W // 2 + 40, H // 2 + 11)):
                got = ctx.render_keys(sid, mid, roi, pose, W, H)
                want, _ = oracle.render_keys(osc, om, pose, roi=roi)
                assert np.array_equal(got, want), (z, roi, int(np.sum(got != want)))
