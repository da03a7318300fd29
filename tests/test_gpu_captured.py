"""A call captured into a graph leaves no error behind for the calls that follow."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu


def test_a_context_that_was_captured_from_closes_clean():
    import torch
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    mesh = scenes.box_mesh(0.06, 0.08, 0.12, 3, 3, 3)
    pose = np.array([[1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0.5]], np.float32)
    moved = pose + np.float32(0.25) * (np.arange(12) == 7)
    dev = [torch.from_numpy(x).cuda() for x in (pose, moved)]
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with P.Context(0) as ctx:
        mid = ctx.load_mesh(mesh)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            P.perch_add_s(ctx.ctx, mid, *dev, False, out=out, stream=stream)
        graph.replay()
        torch.cuda.synchronize()
        assert abs(float(out) - 0.25) < 1e-7
        del graph
    with P.Context(0) as ctx:               # its first launch reports no earlier call's error
        mid = ctx.load_mesh(mesh)
        assert abs(float(P.perch_add_s(ctx.ctx, mid, pose, moved, False)[0]) - 0.25) < 1e-7
