"""Scans whose words are the offsets of the scan before, call after call on one
stream without a wait: every call reads what the one before it wrote, for sizes
of one to eight tiles (one cluster) and beyond, with the words changing between
rounds."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_tiles", [1, 2, 3, 5, 8, 9, 40])
def test_each_scan_reads_the_offsets_of_the_one_before(n_tiles):
    n, rounds, calls = 4096 * n_tiles, 40, 5
    rng = np.random.default_rng(n_tiles)
    words = rng.integers(0, 65536, (rounds, n)).astype(np.uint32)
    marks = rng.integers(0, 2 ** 32, n // 32, dtype=np.uint64).astype(np.uint32)
    bits = np.unpackbits(marks.view(np.uint8), bitorder="little").astype(bool)
    dev = torch.from_numpy(words.view(np.int32)).cuda()
    dev_marks = torch.from_numpy(marks.view(np.int32)).cuda()
    bufs = torch.zeros((rounds, calls, n), dtype=torch.int32, device="cuda")
    src, steps = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty((calls, n), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for r in range(rounds):  # the same buffers each round: stale words are the last round's
        src.copy_(dev[r])
        for c in range(calls):
            vrt.scan_counts_noalloc(src if c == 0 else steps[c - 1], steps[c], marks=dev_marks if c % 2 else None)
        bufs[r].copy_(steps)
    got = bufs.cpu().numpy().view(np.uint32)
    for r in range(rounds):
        w = words[r]
        for c in range(calls):
            count = (w & 0xFFFF).astype(np.uint64) * (bits if c % 2 else 1)
            w = (np.cumsum(count) - count).astype(np.uint32)
            assert np.array_equal(got[r, c], w), (r, c)
