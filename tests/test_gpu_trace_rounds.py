"""The trace's rounds at the sizes where they change form: images so small that a
tile holds 4, 8 or 16 rays, images that end inside a tile, and voxel lists of
thousands of entries whose hits overflow the warp's pool, so that rays take a
voxel in parts of its interval. Against the oracle within tests/parity.py's
tolerances, and bitwise equal to the whole-warp path, which composites the same
hits in the same order."""
import numpy as np
import pytest

import oracle
import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, LineSet, tiny_walks
from parity import compare_image

pytestmark = pytest.mark.gpu


def _frame(r, cam, alpha):
    out = r.frame(cam, alpha=alpha)
    vrt.sync(r.h)
    return [t.cpu().numpy().copy() for t in out]


def _check(ls, cam, alpha):
    ref = oracle.Oracle.from_lineset(ls).render(cam, alpha=alpha)
    r = vrt.Renderer(ls.n, ls.radius)
    r.upload(ls.xyz, ls.offsets)
    default = _frame(r, cam, alpha)
    vrt.set_option(r.h, vrt.OPT_TRACE_SHORT_LIST, 0)  # every list on the whole-warp path
    whole_warp = _frame(r, cam, alpha)
    r.close()
    res = compare_image(*default, ref)
    assert res["hits"] > 0 and res["col_bad"] == 0 and res["id_bad"] == 0, res
    assert res["max_t_rel"] < 2e-4, res
    for a, b in zip(default, whole_warp):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("w,h", [(1, 1), (7, 3), (121, 93), (173, 141), (251, 197), (331, 301)])
def test_small_images(w, h):
    ls = tiny_walks(n_lines=600, n_verts=40, seed=123)
    n = ls.n
    cam = Camera(width=w, height=h, ortho=0, eye=(n * 1.6, n * 1.3, n * 0.9),
                 target=(n / 2, n / 2, n / 2), up=(0, 0, 1), fovy_deg=45.0)
    _check(ls, cam, 0.3)


@pytest.mark.parametrize("n_lines", [190, 1500, 3000])
@pytest.mark.parametrize("alpha", [0.3, 0.02])
def test_lists_past_the_pool(n_lines, alpha):
    # straight tubes along x through one column of voxels, all of one colour: a
    # ray down z through the middle hits every one of them, most in one voxel
    rng = np.random.default_rng(n_lines)
    y = 16.5 + rng.uniform(-0.05, 0.05, n_lines)
    z = 16.5 + rng.uniform(-0.45, 0.45, n_lines)
    xyz = np.stack([np.stack([np.full(n_lines, 2.0), y, z], 1),
                    np.stack([np.full(n_lines, 30.0), y, z], 1)], 1).reshape(-1, 3)
    ls = LineSet(xyz=xyz.astype(np.float32), offsets=np.arange(0, 2 * n_lines + 1, 2), n=32,
                 radius=0.4)
    cam = Camera(width=24, height=20, ortho=1, eye=(16.0, 16.5, -5.0), target=(16.0, 16.5, 40.0),
                 up=(0.0, 1.0, 0.0), ortho_h=2.0)
    _check(ls, cam, alpha)
