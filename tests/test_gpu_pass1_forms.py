"""Pass 1 at the sizes where its work changes form: sets small enough that a warp
takes 4, 8 or 16 segments, segments with more candidates than one owner table
holds, and long segments (no slab boxes) next to short ones in one warp. Voxel
words and lists against the oracle, bit-exact (occupancy within its near-tie
range)."""
import numpy as np
import pytest

import oracle
import paper_2510_09081_gb300 as vrt
from gen.linesets import LineSet, random_polylines, tiny_walks, tiny_walks_camera
from parity import check_lists, check_words

pytestmark = pytest.mark.gpu


def _check(ls):
    L = oracle.Oracle.from_lineset(ls).lists()
    r = vrt.Renderer(ls.n, ls.radius)
    r.upload(ls.xyz, ls.offsets)
    vrt.voxelize(r.h)
    vrt.cull(r.h, vrt.camera_c(tiny_walks_camera(ls.n, 16, 16)), vrt.params_c(cull=0))
    vrt.sync(r.h)
    words = vrt.read_grid(r.h, ls.n)
    lists = vrt.read_lists(r.h, ls.n)
    st = vrt.get_stats(r.h)
    r.close()
    check_words(words, L)
    check_lists(*lists, L)
    assert st["fragments"] == int(L["count"].sum())


@pytest.mark.parametrize("n_lines", [1, 40, 300, 600, 1200])
def test_segments_per_warp(n_lines):
    _check(tiny_walks(n_lines=n_lines, n_verts=50, n=64, seed=n_lines))


@pytest.mark.parametrize("radius", [0.05, 1.3, 3.9])
def test_candidates_past_one_table(radius):
    _check(random_polylines(60, (2, 30), 64, radius, seed=int(radius * 100)))


def test_long_segments_next_to_short_ones():
    short = random_polylines(200, (2, 6), 64, 0.4, seed=5)
    rng = np.random.default_rng(8)
    xyz, lens = [], []
    for p in range(200):
        xyz.append(short.xyz[short.offsets[p]:short.offsets[p + 1]])
        lens.append(xyz[-1].shape[0])
        if p % 3 == 0:  # a line across the grid and beyond it
            a, b = rng.uniform(-20.0, 84.0, (2, 3))
            xyz.append(np.array([a, b], np.float32))
            lens.append(2)
    ls = LineSet(xyz=np.concatenate(xyz), offsets=np.concatenate([[0], np.cumsum(lens)]).astype(np.int64),
                 n=64, radius=0.4)
    _check(ls)
