"""Culling for cameras that see part of the grid, where the erosion leaves out the
bricks no march can reach: from inside the grid and an orthographic close-up, at
the grid sides where a warp takes 2, 8 and 32 bricks. The image is that of no
culling, bitwise, and few voxels need repair: the marks still keep what the view
shows."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, tiny_walks

pytestmark = pytest.mark.gpu


def _views(n):
    c = n / 2.0
    return [Camera(width=97, height=61, ortho=0, eye=(c, c, c), target=(c + 10.0, c + 3.0, c + 2.0),
                   up=(0, 0, 1), fovy_deg=45.0),
            Camera(width=97, height=61, ortho=1, eye=(c, -1.0, c), target=(c + 3.0, float(n), c),
                   up=(0, 0, 1), ortho_h=n / 4.0)]


@pytest.mark.parametrize("n", [16, 64, 256, 512])
@pytest.mark.parametrize("alpha", [1.0, 0.4])
def test_partial_views(n, alpha):
    ls = tiny_walks(n_lines=40 * min(n, 128), n_verts=60, n=n, seed=n, start_lo=n / 4.0,
                    start_hi=max(n / 4.0 + 1.0, min(n - 2.0, n / 4.0 + 64.0)))
    r = vrt.Renderer(ls.n, ls.radius)
    r.upload(ls.xyz, ls.offsets)
    for cam in _views(n):
        out = []
        for cull in (0, 1):
            img = r.frame(cam, alpha=alpha, cull_on=cull)
            vrt.sync(r.h)
            out.append([t.cpu().numpy().copy() for t in img])
        st = vrt.get_stats(r.h)
        for a, b in zip(*out):
            assert np.array_equal(a, b)
        assert st["visible_voxels"] <= st["occupied_voxels"]
        assert st["repaired_voxels"] <= 0.02 * st["occupied_voxels"]
    r.close()
