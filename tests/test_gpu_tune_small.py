"""The tile width of a small transparent image, whose tiles the trace shapes itself,
is not chosen by the noise of equal measurements."""
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, tiny_walks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,alpha,own", [(160, 120, 0.3, True), (320, 300, 0.3, True),
                                           (400, 300, 0.3, False), (160, 120, 1.0, False)])
def test_widths_are_compared_where_they_differ(w, h, alpha, own):
    ls = tiny_walks(n_lines=300, n_verts=30, seed=5)
    n = ls.n
    cam = Camera(width=w, height=h, ortho=0, eye=(n * 1.6, n * 1.3, n * 0.9),
                 target=(n / 2, n / 2, n / 2), up=(0, 0, 1), fovy_deg=45.0)
    (side, tile), ms = vrt.tune_shapes(ls.xyz, ls.offsets, n, ls.radius, cam, [32, 64], tiles=(8, 4, 16, 2),
                                       alpha=alpha, frames=2)
    assert ms[side, tile] == min(ms.values())
    if own:
        assert tile == 8 and all(len({ms[s, t] for t in (8, 4, 16, 2)}) == 1 for s in (32, 64))
    else:
        assert all(len({ms[s, t] for t in (8, 4, 16, 2)}) > 1 for s in (32, 64))
