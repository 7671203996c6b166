"""The trace's testing limits (longest list and most hits on the shared path) can be
set and taken back to the default."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, LineSet

pytestmark = pytest.mark.gpu


# tubes along x through the same voxels: opaque, lists longer than the limit; transparent,
# more hits a ray than the limit, but fewer for the 4 rays of a tile than the pool holds
@pytest.mark.parametrize("option,limit,default_value,refused,tubes,alpha", [
    (vrt.OPT_TRACE_SHORT_LIST, 5, 1024, (-1, 1025), 40, 1.0),
    (vrt.OPT_TRACE_RAY_KEYS, 8, -1, (-2, 0, 33), 40, 0.02)])
def test_limits_return_to_the_default(option, limit, default_value, refused, tubes, alpha):
    rng = np.random.default_rng(3)
    off = 16.5 + rng.uniform(-0.3, 0.3, (tubes, 1, 2))
    xyz = np.concatenate([np.tile([[[4.0], [28.0]]], (tubes, 1, 1)), np.tile(off, (1, 2, 1))], 2)
    ls = LineSet(xyz=xyz.reshape(-1, 3).astype(np.float32), offsets=np.arange(0, 2 * tubes + 1, 2), n=32, radius=0.4)
    cam = Camera(width=24, height=20, ortho=1, eye=(16.0, 16.5, -5.0), target=(16.0, 16.5, 40.0),
                 up=(0.0, 1.0, 0.0), ortho_h=2.0)
    r = vrt.Renderer(ls.n, ls.radius, occ_scale=2)
    r.upload(ls.xyz, ls.offsets)
    vrt.set_option(r.h, vrt.OPT_TRACE_COUNTERS, 1)

    def lists_taken_by_whole_warps():
        r.frame(cam, alpha=alpha)
        vrt.sync(r.h)
        return vrt.get_stats(r.h)["trace_wholewarp_voxels"]

    default = lists_taken_by_whole_warps()
    vrt.set_option(r.h, option, limit)
    limited = lists_taken_by_whole_warps()
    vrt.set_option(r.h, option, default_value)
    again = lists_taken_by_whole_warps()
    for value in refused:
        with pytest.raises(vrt.VrtError) as e:
            vrt.set_option(r.h, option, value)
        assert e.value.status == vrt.ERR_INVALID_ARG
    r.close()
    assert limited > default == again == 0
