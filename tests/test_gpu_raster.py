"""The rasteriser at the sizes where its queues can go wrong: triangle counts
around the warp's 32, pixel boxes from a fraction of a sample to hundreds (walked
in one lane, staged by samples, staged by rows for thin wedges, more larger ones
than are staged at a time), tiles smaller than the render.  Key buffers are
bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2008_00326_gb300 import build, perch
    build.build()
    perch.load()
    return perch


def _meshes():
    out = {f"tris{n}": scenes.box_mesh(0.1, 0.08, 0.12, 4, 4, 4) for n in (1, 31, 32, 33, 65)}
    for name, m in out.items():
        m.tris = np.ascontiguousarray(m.tris[:int(name[4:])])
    out["coarse"] = scenes.ellipsoid_mesh(0.05, 0.04, 0.06, 9, 8)
    out["wedges"] = scenes.cylinder_mesh(0.05, 0.02, 250, 1)
    out["slivers"] = scenes.cylinder_mesh(0.04, 0.15, 200, 1)
    out["fine"] = scenes.ellipsoid_mesh(0.05, 0.04, 0.06, 61, 60)
    return out


@pytest.mark.parametrize("zbuf_words", [7064, 1024])
@pytest.mark.parametrize("name", ["tris1", "tris31", "tris32", "tris33", "tris65", "coarse", "wedges", "slivers", "fine"])
def test_keys_at_queue_sizes(P, oracle, name, zbuf_words):
    sc = scenes.tabletop_small()
    mesh = _meshes()[name]
    rng = np.random.default_rng(17)
    om, osc = oracle.OracleMesh.from_mesh(mesh), oracle.OracleScene.from_scene(sc)
    with P.Context(0) as ctx:
        ctx.set_launch_config(256, zbuf_words)
        sid, mid = ctx.set_observation(sc), ctx.load_mesh(mesh)
        for z in (0.12, 0.3, 0.8, 2.5):
            r = scenes.random_rotation(rng)
            pose = np.concatenate([r, (rng.normal(size=3) * 0.02 + [0, 0, z])[:, None]], 1).astype(np.float32).reshape(12)
            for roi in ((0, 0, sc.W, sc.H), (37, 21, 118, 90)):
                got = ctx.render_keys(sid, mid, roi, pose, sc.W, sc.H)
                want, _ = oracle.render_keys(osc, om, pose, roi=roi)
                assert np.array_equal(got, want), (name, z, roi, int(np.sum(got != want)))
