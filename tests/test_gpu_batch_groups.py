"""A batch at the edges of what its kernels count: a job's first sample comes from sums over its
own tiles of 32 rays, groups of 32 tiles and groups of 1024; the job of a tile from a search 32
entries wide.  Jobs are stretches of one ray array, so the single call over all rays gives every
job's samples exactly."""
import numpy as np
import pytest
import torch

from paper_2404_10272_gb300 import scenes
from _helpers import to_np

pytestmark = pytest.mark.gpu

SIZES = {
    "one": [7],
    "groups": [1, 31, 0, 32, 33, 1023, 1024, 1025, 0, 0, 32767, 32768, 32769, 5, 66000, 2],
    "32 jobs": [40] * 31 + [1100],
    "33 jobs": [0] + [33, 64] * 16,
    "1025 jobs": [1 + (i * 7) % 70 for i in range(1025)],
    "2100 jobs": [(i % 3) * 20 for i in range(2100)],
}


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


@pytest.mark.parametrize("name", list(SIZES))
def test_job_sizes(H, name):
    sizes = np.array(SIZES[name])
    rng = np.random.default_rng(sizes.size)
    n = int(sizes.sum())
    occ = (rng.random((1, 32, 32, 32)) < 0.3).astype(np.uint8)
    grid = H.build_vdb(torch.from_numpy(occ).cuda(), np.array([[-1, -1, -1, 1, 1, 1]], np.float32))
    prm = H.make_params(0.05, 6.0, 0.03, 0.0, 1e10, 1000)
    o = torch.from_numpy(rng.uniform(-2.0, 2.0, (n, 3)).astype(np.float32)).cuda()
    d = rng.normal(size=(n, 3)) - 0.5 * to_np(o)
    d = torch.from_numpy((d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)).cuda()
    off, ray, t0, t1 = (to_np(x) for x in H.traverse_hdda(o, d, grid, prm).trimmed())
    assert off[-1] > n // 2
    beg = np.concatenate([[0], np.cumsum(sizes)])
    jobs = []
    for a, b in zip(beg[:-1], beg[1:]):
        jobs.append(dict(rays_o=o[a:b], rays_d=d[a:b], grid=grid, params=prm,
                         out=H.alloc_samples(int(b - a), max(1, int(off[b] - off[a])))))
    batch = H.Batch(jobs)
    for _ in range(2):
        for j in jobs:
            j["out"].offsets.fill_(-1)
        batch.launch()
        totals, status = batch.results()
        assert status == [0] * len(jobs)
        for i, (a, b, j) in enumerate(zip(beg[:-1], beg[1:], jobs)):
            x, y = off[a], off[b]
            assert totals[i] == y - x
            got = [to_np(v) for v in j["out"].trimmed()]
            for u, v in zip(got, (off[a:b + 1] - x, ray[x:y] - a, t0[x:y], t1[x:y])):
                assert np.array_equal(u, v), i
    batch.free()
