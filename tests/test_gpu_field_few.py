"""Fields of few blobs: up to 32 of them the compositor's lane groups set up their own rays, sixteen
blobs per step.  Blob counts around the steps and the limit, rays that end together and rays that
do not, some of them without a blob in reach; pixels against the binary64 oracle within the
compositor's 1e-5."""
import numpy as np
import pytest
import torch

import oracle
from _helpers import to_np

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


@pytest.mark.parametrize("G", [0, 1, 8, 9, 15, 16, 17, 31, 32, 33])
@pytest.mark.parametrize("lengths", ["two", "mixed"])
def test_few_blobs(H, G, lengths):
    rng = np.random.default_rng(100 * G + len(lengths))
    n = 333
    counts = np.full(n, 2) if lengths == "two" else rng.choice([0, 1, 5, 33, 64, 190], n)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    S = int(off[-1])
    o = rng.uniform(-1.0, 1.0, (n, 3)).astype(np.float32)
    o[:, 2] -= 2.0
    d = rng.normal(0.0, 0.3, (n, 3))
    d[:, 2] = 1.0
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    t0 = np.concatenate([np.sort(rng.uniform(0.5, 4.0, c)) for c in counts]).astype(np.float32)
    t1 = (t0 + rng.uniform(0.002, 0.03, S).astype(np.float32)).astype(np.float32)
    field = np.zeros((G, 8), np.float32)
    field[:, :3] = rng.uniform(-1.5, 1.5, (G, 3))
    field[:, 3] = rng.uniform(0.03, 0.15, G)
    field[:, 4] = rng.uniform(0.5, 50.0, G)
    field[:, 5:] = rng.uniform(0.0, 1.0, (G, 3))
    s = H.Samples(torch.from_numpy(off).cuda(), torch.zeros(S, dtype=torch.int32, device="cuda"),
                  torch.from_numpy(t0).cuda(), torch.from_numpy(t1).cuda(), S)
    rgba = to_np(H.composite(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), s,
                             torch.from_numpy(field).cuda())).astype(np.float64)
    ref = oracle.composite(o, d, off, t0, t1, field)
    assert np.abs(rgba - ref).max() <= TOL, np.abs(rgba - ref).max()


@pytest.mark.parametrize("G", [0, 5, 16, 17])
def test_large_calls(H, G):
    # from 65,536 rays on: tasks of 16 rays over up to 16 blobs, of 8 over more; the last one is cut
    rng = np.random.default_rng(G)
    n = 65541
    counts = rng.choice([0, 1, 2, 3, 40], n)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    S = int(off[-1])
    o = rng.uniform(-1.0, 1.0, (n, 3)).astype(np.float32)
    o[:, 2] -= 2.0
    d = np.tile(np.array([[0.0, 0.6, 0.8]], np.float32), (n, 1))
    first = rng.uniform(0.5, 3.0, n).astype(np.float32)
    k = np.arange(S) - np.repeat(off[:-1], counts)
    t0 = (np.repeat(first, counts) + 0.02 * k).astype(np.float32)
    t1 = (t0 + np.float32(0.02)).astype(np.float32)
    field = np.zeros((G, 8), np.float32)
    field[:, :3] = rng.uniform(-1.5, 1.5, (G, 3))
    field[:, 3] = rng.uniform(0.1, 0.3, G)
    field[:, 4] = rng.uniform(0.5, 50.0, G)
    field[:, 5:] = rng.uniform(0.0, 1.0, (G, 3))
    s = H.Samples(torch.from_numpy(off).cuda(), torch.zeros(S, dtype=torch.int32, device="cuda"),
                  torch.from_numpy(t0).cuda(), torch.from_numpy(t1).cuda(), S)
    rgba = to_np(H.composite(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), s,
                             torch.from_numpy(field).cuda())).astype(np.float64)
    ref = oracle.composite(o, d, off, t0, t1, field)
    assert np.abs(rgba - ref).max() <= TOL, np.abs(rgba - ref).max()
