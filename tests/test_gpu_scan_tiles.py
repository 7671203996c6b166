"""The list-offset scan's tiles: every position in a tile, marks in every nibble,
full 16-bit counts beside non-zero upper halves, the sizes at and beside a full
cluster, and more tiles than one look-back window or one set of resident blocks."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_tiles", [1, 2, 3, 8, 9, 33, 1301])
@pytest.mark.parametrize("marked", ["all", "random", "one per tile", "none"])
def test_offsets_equal_the_prefix_sum(n_tiles, marked):
    n = 4096 * n_tiles
    rng = np.random.default_rng(n_tiles)
    top = 65536 if n_tiles < 16 else 400          # totals stay below 2^32
    words = (rng.integers(0, top, n) | (rng.integers(0, 65536, n) << 16)).astype(np.uint32)
    bits = {"all": np.ones(n, bool), "random": rng.random(n) < 0.5,
            "one per tile": np.arange(n) % 4096 == (np.arange(n) // 4096 * 1237) % 4096,
            "none": np.zeros(n, bool)}[marked]
    marks = np.packbits(bits.reshape(-1, 32), axis=1, bitorder="little").view("<u4").reshape(-1)
    marks = None if marked == "all" else torch.from_numpy(marks.astype(np.uint32).view(np.int32)).cuda()
    counts = np.where(bits, words & 0xFFFF, 0).astype(np.uint64)
    want = np.cumsum(counts) - counts
    offsets = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    total = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    vrt.scan_counts_noalloc(torch.from_numpy(words.view(np.int32)).cuda(), offsets, marks=marks,
                            total=total, status=status)
    torch.cuda.synchronize()
    assert int(status.cpu()[0]) == 0
    assert np.array_equal(offsets.cpu().numpy().view(np.uint32), want.astype(np.uint32))
    assert int(total.cpu().numpy().view(np.uint32)[0]) == int(counts.sum())
