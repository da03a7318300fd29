"""Regions of interest are clipped to the image on every side, also those that lie
wholly past it: the box is empty, with its bounds inside the image, which is what the
kernels' 16-bit pixels and binary32 divisions are made for.  Host code only: the
library's own clip_roi, called from a small C++ program."""
import subprocess

import numpy as np
import pytest

from host_program import build_program

PROGRAM = r"""
#include "perch_host.cuh"
#include <cstdio>
int main()
{
    int W, H, r[4], out[4];
    while (scanf("%d %d %d %d %d %d", &W, &H, &r[0], &r[1], &r[2], &r[3]) == 6) {
        perch_host::SceneRec s;
        s.ds.W = W;
        s.ds.H = H;
        perch_host::clip_roi(nullptr, s, r, out);
        printf("%d %d %d %d\n", out[0], out[1], out[2], out[3]);
    }
}
"""


@pytest.fixture(scope="module")
def clip(tmp_path_factory):
    exe = build_program(tmp_path_factory.mktemp("clip"), PROGRAM)

    def run(W, H, rois):
        text = "\n".join(" ".join(str(int(x)) for x in (W, H, *r)) for r in rois)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return np.array([[int(x) for x in line.split()] for line in out.splitlines()])

    return run


@pytest.mark.parametrize("W,H", [(160, 120), (1023, 455), (1, 466033)])
def test_boxes_end_inside_the_image(clip, W, H):
    big = 2 ** 31 - 1
    xs = [-big, -5, 0, 1, W - 1, W, W + 1, 2 * W, 64512, 67108867, big]
    ys = [-big, -5, 0, 1, H - 1, H, H + 1, 2 * H, 64512, 67108867, big]
    rng = np.random.default_rng(1)
    rois = [(x, y, x + w, y + h) for x in xs for y in ys for w, h in ((0, 0), (1, 7), (W, H), (-9, 3))
            if abs(x + w) <= big and abs(y + h) <= big]
    rois += [tuple(rng.integers(-2 * W, 2 * W, 4)) for _ in range(200)]
    got = clip(W, H, rois)
    assert (got[:, 0] >= 0).all() and (got[:, 1] >= 0).all()
    assert (got[:, 0] <= got[:, 2]).all() and (got[:, 1] <= got[:, 3]).all()
    assert (got[:, 2] <= W).all() and (got[:, 3] <= H).all()
    for r, g in zip(rois, got):         # and hold the region's pixels, no others
        u0, v0, u1, v1 = max(0, r[0]), max(0, r[1]), min(W, r[2]), min(H, r[3])
        if u0 < u1:
            assert (g[0], g[2]) == (u0, u1)
        else:
            assert g[0] == g[2]
        if v0 < v1:
            assert (g[1], g[3]) == (v0, v1)
        else:
            assert g[1] == g[3]
