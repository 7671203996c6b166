"""What the server reserves for a set before it is resident covers what the set then
holds: culled, shaded frames at 1080p on the smallest and larger grids, few vertices
(whose record buffers are larger than their lists) and many."""
import ctypes

import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, walk_set

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("segments,n,max_fragments", [(300, 16, 0), (2000, 64, 0), (20_000, 128, 0),
                                                      (20_000, 64, 3_000_000), (60_000, 128, 0),
                                                      (100_000, 512, 0)])
def test_the_estimate_covers_the_set(segments, n, max_fragments):
    ls = walk_set(segments, n, radius=0.4, seed=3)
    # the mean the server estimates from, over the same vertices
    d = np.linalg.norm(np.diff(ls.xyz.astype(np.float64), axis=0), axis=1)
    ends = np.zeros(ls.n_vertices, bool)
    ends[ls.offsets[1:] - 1] = True
    estimate = vrt.load()._ZN3vrt9set_bytesEifmld
    estimate.restype = ctypes.c_uint64
    estimate.argtypes = [ctypes.c_int, ctypes.c_float, ctypes.c_uint64, ctypes.c_int64, ctypes.c_double]
    reserved = estimate(n, ls.radius, max_fragments, ls.n_vertices, d[~ends[:-1]].mean())
    cam = Camera(width=1920, height=1080, ortho=0, eye=(n * 1.6, n * 1.3, n * 0.9),
                 target=(n / 2, n / 2, n / 2), up=(0, 0, 1), fovy_deg=45.0)
    r = vrt.Renderer(n, ls.radius, max_fragments=max_fragments)
    r.upload(ls.xyz, ls.offsets)
    r.frame(cam, alpha=0.5, ao_cones=6, cull_on=1, voxel_shading=1)
    vrt.sync(r.h)
    held = vrt.grid_device_bytes(r.h)
    r.close()
    assert held <= reserved
    assert reserved - held < 0.2 * held + (64 << 20)
