"""The occupancy pyramid's two finest levels, exactly: level 0 is each voxel's
occupancy code over the scale, stored in the texel format, level 1 the mean of the 8
stored children, summed z, y, x. At the smallest grid side, where a warp's bricks
span two rows, and above."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import tiny_walks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DTYPE = {vrt.MIPS_F32: torch.float32, vrt.MIPS_F16: torch.float16, vrt.MIPS_BF16: torch.bfloat16}


def _stored(a, fmt):
    return torch.from_numpy(a).to(DTYPE[fmt]).to(torch.float32).numpy()


@pytest.mark.parametrize("n", [16, 32, 128])
@pytest.mark.parametrize("fmt", [vrt.MIPS_F32, vrt.MIPS_F16, vrt.MIPS_BF16])
@pytest.mark.parametrize("occ_scale", [32, 21])
def test_two_finest_levels(n, fmt, occ_scale):
    ls = tiny_walks(n_lines=300, n_verts=40, n=n, seed=n, start_lo=2.0, start_hi=n - 2.0)
    r = vrt.Renderer(ls.n, ls.radius, occ_scale=occ_scale)
    r.upload(ls.xyz, ls.offsets)
    vrt.set_option(r.h, vrt.OPT_MIPS_FORMAT, fmt)
    vrt.voxelize(r.h)
    vrt.build_mips(r.h)
    codes = (vrt.read_grid(r.h, n) >> 16).reshape(n, n, n).astype(np.float32)
    got = vrt.read_mips(r.h, n)
    r.close()
    assert codes.max() > 0
    inv = np.float32(1.0) / np.float32(occ_scale)
    l0 = _stored(np.minimum(np.float32(1.0), codes * inv), fmt)
    s = np.zeros((n // 2,) * 3, np.float32)
    for dz in range(2):
        for dy in range(2):
            for dx in range(2):
                s = s + l0[dz::2, dy::2, dx::2]
    assert np.array_equal(got[0], l0)
    assert np.array_equal(got[1], _stored(s * np.float32(0.125), fmt))
