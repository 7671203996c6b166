"""Pixels of an opaque AO frame that the repair rounds leave unfinished (reported by
vrt_sync) keep what the caller's image held, whatever its bits: they are not taken
for hits to shade. Rays are stopped early by the test limit, so that the last
repair round still meets voxels without lists."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, tiny_walks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_unfinished_pixels_keep_the_image():
    ls = tiny_walks(n_lines=1500, n_verts=40, n=64, seed=31)
    n = ls.n
    cam = Camera(width=157, height=93, ortho=0, eye=(n * 1.6, n * 1.3, n * 0.9),
                 target=(n / 2, n / 2, n / 2), up=(0, 0, 1), fovy_deg=45.0)
    r = vrt.Renderer(n, ls.radius)
    r.upload(ls.xyz, ls.offsets)
    vrt.set_option(r.h, vrt.OPT_CULL_DEPTH, 1)  # nearly everything behind the first voxels
    before = torch.tensor([0.0, 0.25, 0.5, 1.0], device="cuda")  # x as bits: segment 0
    unfinished = 0
    for calls in range(2, 40):
        vrt.set_option(r.h, vrt.OPT_TEST_TRACE_CALLS, calls)
        rgba, ids, depth = r.buffers(cam.width, cam.height)
        rgba[:] = before
        ids.fill_(-77)
        try:
            r.frame(cam, alpha=1.0, ao_cones=6, cull_on=1)
            vrt.sync(r.h)
        except vrt.VrtError as e:
            assert e.status == vrt.ERR_TIMEOUT
        left = ids == -77
        unfinished += int(left.sum())
        assert bool((rgba[left] == before).all()), calls
    assert unfinished > 0
    r.close()
