"""Cone AO of opaque traces, shaded per pixel after the trace and its repair
rounds, against the oracle: ragged and tiny images (tile edges), the smallest
grid (whose pyramid ends below the widest cone sample's upper level), hits found
on the whole-warp path and hits found by repair rounds."""
import numpy as np
import pytest

import oracle
import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, tiny_walks
from parity import compare_image

pytestmark = pytest.mark.gpu


def _frame(r, cam, cull):
    out = r.frame(cam, alpha=1.0, ao_cones=6, cull_on=cull)
    vrt.sync(r.h)
    return [t.cpu().numpy().copy() for t in out]


@pytest.mark.parametrize("n,lines,w,h", [(16, 60, 33, 5), (16, 60, 1, 1), (64, 1500, 16, 8),
                                         (64, 1500, 157, 93)])
def test_opaque_ao_matches_oracle_on_every_route(n, lines, w, h):
    ls = tiny_walks(n_lines=lines, n_verts=40, n=n, seed=31)
    cam = Camera(width=w, height=h, ortho=0, eye=(n * 1.6, n * 1.3, n * 0.9),
                 target=(n / 2, n / 2, n / 2), up=(0, 0, 1), fovy_deg=45.0)
    ref = oracle.Oracle.from_lineset(ls).render(cam, alpha=1.0, ao_cones=6)
    r = vrt.Renderer(ls.n, ls.radius)
    r.upload(ls.xyz, ls.offsets)
    plain = _frame(r, cam, 0)
    res = compare_image(*plain, ref)
    assert res["hits"] > 0 and res["col_bad"] == 0 and res["id_bad"] == 0, res
    vrt.set_option(r.h, vrt.OPT_TRACE_SHORT_LIST, 0)
    whole_warp = _frame(r, cam, 0)
    vrt.set_option(r.h, vrt.OPT_TRACE_SHORT_LIST, 1024)
    vrt.set_option(r.h, vrt.OPT_CULL_DEPTH, 500)  # culls voxels that rays reach
    repaired = _frame(r, cam, 1)
    st = vrt.get_stats(r.h)
    r.close()
    assert n == 16 or w < 100 or st["repaired_voxels"] > 0
    for other in (whole_warp, repaired):
        for a, b in zip(plain, other):
            assert np.array_equal(a, b)
