"""Renders on both sides of the line between the two rasterisers (one sample a triangle,
for meshes whose triangles fill their boxes): key buffers bit-exact against the oracle,
in one tile and in several, and costs by every kind of call that renders."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,zbuf_words", [(256, 7064), (128, 1024), (512, 14336)])
@pytest.mark.parametrize("n", [3, 6, 12, 24, 48])
def test_keys_around_one_sample_a_triangle(oracle, n, threads, zbuf_words):
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    sc = scenes.tabletop_small()
    rng = np.random.default_rng(n)
    with P.Context(0) as ctx:
        ctx.set_launch_config(threads, zbuf_words)
        for jo_mode in (0, 1):
            sid = ctx.set_observation(sc, jo_mode=jo_mode, color_check=0)
            osc = oracle.OracleScene.from_scene(sc, jo_mode=jo_mode, color_check=0)
            for mesh in (scenes.ellipsoid_mesh(0.04, 0.05, 0.06, n, n), scenes.box_mesh(0.06, 0.08, 0.1, n, n, n)):
                mid, om = ctx.load_mesh(mesh), oracle.OracleMesh.from_mesh(mesh)
                poses = []
                for z in (0.1, 0.25, 0.5, 0.9, 1.6, 3.0, 7.0):
                    r = scenes.random_rotation(rng)
                    poses.append(np.concatenate([r, (rng.normal(size=3) * 0.03 + [0, 0, z])[:, None]], 1).reshape(12))
                poses = np.asarray(poses, np.float32)
                got = ctx.score(sid, mid, -1, None, poses)
                assert np.array_equal(got, oracle.score(osc, om, poses)[0]), (mesh.name, jo_mode)
                if jo_mode:
                    continue
                for pose in poses:
                    got = ctx.render_keys(sid, mid, None, pose, sc.W, sc.H)
                    want, _ = oracle.render_keys(osc, om, pose)
                    assert np.array_equal(got, want), (mesh.name, pose[11], int(np.sum(got != want)))
                got = ctx.refine(sid, mid, -1, None, poses[1:5])
                want = oracle.gicp(osc, om, poses[1:5])
                assert np.array_equal(got[0].view(np.uint32), want[0].view(np.uint32))
