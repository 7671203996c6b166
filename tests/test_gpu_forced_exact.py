"""A voxel's packed word does not depend on the stage that decided its segments: every
pair decided on the exact path gives the words of the filter, counts and occupancy
sums alike, on dense and clipped sets."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import random_polylines, tiny_walks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ls,occ_scale", [
    (tiny_walks(n_lines=2000, n_verts=50, n=64, seed=3), 32),
    (tiny_walks(n_lines=400, n_verts=50, n=64, radius=1.7, seed=4), 200),
    (random_polylines(200, (2, 30), 64, 0.7, seed=5), 1000)], ids=["walks", "thick", "polylines"])
def test_words_equal_the_filters(ls, occ_scale):
    words = []
    for forced in (0, 1):
        r = vrt.Renderer(ls.n, ls.radius, occ_scale=occ_scale)
        vrt.set_option(r.h, vrt.OPT_FORCE_EXACT, forced)
        r.upload(ls.xyz, ls.offsets)
        vrt.voxelize(r.h)
        vrt.sync(r.h)
        words.append(vrt.read_grid(r.h, ls.n))
        r.close()
    assert np.array_equal(words[0] & 0xFFFF, words[1] & 0xFFFF)
    assert np.array_equal(words[0], words[1]), int((words[0] != words[1]).sum())
