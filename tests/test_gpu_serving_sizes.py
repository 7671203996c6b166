"""Frames of 256^3 and 512^3 sets overlapping on the server's streams, culling on
and off, from the first frame of each set (which sizes its buffers) on: bitwise
equal to the same frames one at a time on grids that saw the same updates."""
import numpy as np
import pytest

import paper_2510_09081_gb300 as vrt
from gen.linesets import Camera, walk_set

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _requests(sets, n_req):
    rng = np.random.default_rng(11)
    reqs = []
    for i in range(n_req):
        k = i % len(sets)
        n, th = sets[k].n, rng.uniform(0, 2 * np.pi)
        w, h = [(1280, 720), (641, 363), (1920, 1080)][int(rng.integers(3))]
        cam = Camera(width=w, height=h, ortho=0,
                     eye=(n / 2 + 1.7 * n * np.cos(th), n / 2 + 1.7 * n * np.sin(th), n),
                     target=(n / 2, n / 2, n / 2), up=(0.0, 0.0, 1.0), fovy_deg=45.0)
        cnt = sets[k].n_vertices // 50
        first = int(rng.integers(0, sets[k].n_vertices - cnt))
        upd = np.clip(sets[k].xyz[first:first + cnt] + rng.normal(0, 0.05, (cnt, 3)), 1.0,
                      n - 1.0).astype(np.float32)
        reqs.append((k, cam, float(rng.choice([0.2, 0.6, 1.0])), 1 + i // len(sets) % 2, first, upd))
    return reqs


def _images(cam):
    shape = (cam.height, cam.width)
    return [torch.zeros((*shape, 4), device="cuda"), torch.zeros(shape, dtype=torch.int32, device="cuda"),
            torch.zeros(shape, device="cuda")]


def test_overlapped_frames_equal_frames_alone():
    sets = [walk_set(S, n, seed=50 + i) for i, (S, n) in enumerate(
        [(300_000, 256), (1_600_000, 512), (900_000, 256), (400_000, 512), (60_000, 128)])]
    reqs = _requests(sets, 30)
    served = [_images(q[1]) for q in reqs]
    srv = vrt.Server(max_inflight=4)
    ids = [srv.add_set(ls.xyz, ls.offsets, ls.n, ls.radius) for ls in sets]
    for (k, cam, alpha, cull, first, upd), out in zip(reqs, served):
        srv.submit(ids[k], cam, out[0], alpha=alpha, cull_on=cull, first_id=out[1], first_t=out[2],
                   first_vertex=first, update=upd)
    res = srv.poll(wait=True)
    srv.close()
    assert len(res) == len(reqs) and all(r["status"] == 0 for r in res)
    grids = []
    for ls in sets:
        grids.append(vrt.Renderer(ls.n, ls.radius))
        grids[-1].upload(ls.xyz, ls.offsets)
    for (k, cam, alpha, cull, first, upd), out in zip(reqs, served):
        grids[k].update(first, upd)
        alone = grids[k].frame(cam, alpha=alpha, cull_on=cull)
        vrt.sync(grids[k].h)
        for a, b in zip(out, alone):
            assert torch.equal(a, b)
    for r in grids:
        r.close()
