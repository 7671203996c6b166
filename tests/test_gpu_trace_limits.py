"""The limits of the trace's loops: a trace whose rays use up their walk calls ends and says so,
and the next one is whole again; hits that share one depth, as many as the warp's pool holds, more, and lists past
the shared path's longest."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, LineSet, tiny_walks

pytestmark = pytest.mark.gpu


def _frame(r, cam, **kw):
    out = r.frame(cam, **kw)
    vrt.sync(r.h)
    return [t.cpu().numpy().copy() for t in out]


@pytest.mark.parametrize("alpha,ao,cull", [(1.0, 0, 0), (1.0, 6, 1), (0.3, 0, 1), (0.3, 6, 0)])
@pytest.mark.parametrize("w,h", [(33, 5), (640, 480)])
def test_rays_that_are_given_up_are_reported(alpha, ao, cull, w, h):
    ls = tiny_walks(n_lines=600, n_verts=40, seed=7)
    n = ls.n
    cam = Camera(width=w, height=h, ortho=0, eye=(n * 1.6, n * 1.3, n * 0.9),
                 target=(n / 2, n / 2, n / 2), up=(0, 0, 1), fovy_deg=45.0)
    kw = dict(alpha=alpha, ao_cones=ao, cull_on=cull)
    r = vrt.Renderer(n, ls.radius)
    r.upload(ls.xyz, ls.offsets)
    want = _frame(r, cam, **kw)
    vrt.set_option(r.h, vrt.OPT_TEST_TRACE_CALLS, 2)
    with pytest.raises(vrt.VrtError) as e:
        _frame(r, cam, **kw)
    assert e.value.status == vrt.ERR_TIMEOUT
    vrt.set_option(r.h, vrt.OPT_TEST_TRACE_CALLS, 0)
    got = _frame(r, cam, **kw)
    r.close()
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("copies", [30, 190, 200, 1000, 1030, 2000, 20000])
@pytest.mark.parametrize("alpha", [0.3, 0.02])
def test_hits_at_one_depth(copies, alpha):
    # one tube along x, `copies` times: a ray down z hits all of them at one depth
    one = np.array([[10.0, 16.5, 16.5], [22.0, 16.5, 16.5]], np.float32)
    ls = LineSet(xyz=np.tile(one, (copies, 1)), offsets=np.arange(0, 2 * copies + 1, 2), n=32, radius=0.4)
    cam = Camera(width=24, height=20, ortho=1, eye=(16.0, 16.5, -5.0), target=(16.0, 16.5, 40.0),
                 up=(0.0, 1.0, 0.0), ortho_h=2.0)
    r = vrt.Renderer(ls.n, ls.radius, occ_scale=2)  # the voxels' 16-bit occupancy sums hold 20000
    r.upload(ls.xyz, ls.offsets)
    default = _frame(r, cam, alpha=alpha)
    vrt.set_option(r.h, vrt.OPT_TRACE_SHORT_LIST, 0)  # every list on the whole-warp path
    whole_warp = _frame(r, cam, alpha=alpha)
    r.close()
    assert (default[1] >= 0).any()
    for a, b in zip(default, whole_warp):
        assert np.array_equal(a, b)
