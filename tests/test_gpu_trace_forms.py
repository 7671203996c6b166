"""Forms of the trace that meet where no other test has them meet, on the lists of
one build: voxels with more hits than the warp's pool with the 16+16 key and with
AO at every hit, against the whole-warp path, which composites the same hits in the
same order; and the opaque trace's tile shapes, against the default one."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, LineSet, tiny_walks

pytestmark = pytest.mark.gpu


def _same(r, cam, option, values, **kw):
    images = []
    for v in values:
        vrt.set_option(r.h, option, v)
        out = r.trace_only(cam, **kw)
        vrt.sync(r.h)
        images.append([t.cpu().numpy().copy() for t in out])
    assert (images[0][1] >= 0).any()
    for other in images[1:]:
        for a, b in zip(images[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("tubes", [60, 200, 900])  # past the pool by many rays, by one, far
@pytest.mark.parametrize("key,ao", [(vrt.HIT_KEY_16_16, 0), (vrt.HIT_KEY_DEPTH_ID, 6),
                                    (vrt.HIT_KEY_16_16, 6)])
def test_full_pool(tubes, key, ao):
    rng = np.random.default_rng(tubes)
    off = 16.5 + rng.uniform(-0.45, 0.45, (tubes, 1, 2))
    xyz = np.concatenate([np.tile([[[2.0], [30.0]]], (tubes, 1, 1)), np.tile(off, (1, 2, 1))], 2)
    ls = LineSet(xyz=xyz.reshape(-1, 3).astype(np.float32), offsets=np.arange(0, 2 * tubes + 1, 2), n=32,
                 radius=0.4)
    r = vrt.Renderer(ls.n, ls.radius)
    r.upload(ls.xyz, ls.offsets)
    vrt.set_option(r.h, vrt.OPT_HIT_KEY, key)
    for w, h in ((24, 20), (480, 270)):  # tiles of 4 and of 32 rays
        cam = Camera(width=w, height=h, ortho=1, eye=(16.0, 16.5, -5.0), target=(16.0, 16.5, 40.0),
                     up=(0.0, 1.0, 0.0), ortho_h=2.0)
        r.frame(cam, alpha=0.05, ao_cones=ao)
        _same(r, cam, vrt.OPT_TRACE_SHORT_LIST, (1024, 0), alpha=0.05, ao_cones=ao)
    r.close()


@pytest.mark.parametrize("w,h", [(1, 1), (15, 33), (157, 93)])
@pytest.mark.parametrize("ao,cull", [(0, 0), (6, 1)])
def test_opaque_tile_shapes(w, h, ao, cull):
    ls = tiny_walks(n_lines=1500, n_verts=40, n=64, seed=31)
    n = ls.n
    cam = Camera(width=w, height=h, ortho=0, eye=(n * 1.6, n * 1.3, n * 0.9),
                 target=(n / 2, n / 2, n / 2), up=(0, 0, 1), fovy_deg=45.0)
    r = vrt.Renderer(n, ls.radius)
    r.upload(ls.xyz, ls.offsets)
    r.frame(cam, alpha=1.0, ao_cones=ao, cull_on=cull)
    _same(r, cam, vrt.OPT_TRACE_TILE, (4, 2, 8, 16), alpha=1.0, ao_cones=ao)
    r.close()
