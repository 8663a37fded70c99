"""The compositor's work split at its edges: a warp's four lane groups take rays in turn, 32
samples per step read from positions rounded down to a multiple of four, with a record per blob
near the ray (up to 64 blobs) or passes over them (more).  Rays whose lengths straddle the
steps, sample arrays at every alignment (and ending on the last element), ray counts around the
task sizes; pixels against the binary64 oracle within the compositor's 1e-5."""
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


def _field(rng, G):
    f = np.zeros((G, 8), np.float32)
    f[:, :3] = rng.uniform(-1.5, 1.5, (G, 3))
    f[:, 3] = rng.uniform(0.03, 0.3, G)
    f[:, 4] = rng.uniform(0.5, 20.0, G)
    f[:, 5:] = rng.uniform(0.0, 1.0, (G, 3))
    return f


@pytest.mark.parametrize("G", [33, 64, 65, 130])
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_chunk_edges_and_alignment(H, G, shift):
    rng = np.random.default_rng(9000 + 10 * G + shift)
    counts = np.array([0, 1, 31, 32, 33, 0, 0, 5, 63, 64, 65, 2, 29, 35, 0, 97, 3, 128, 30, 1, 34])
    n = counts.size
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    S = int(off[-1])
    o = rng.uniform(-0.5, 0.5, (n, 3)).astype(np.float32)
    o[:, 2] -= 2.0
    d = rng.normal(0.0, 0.2, (n, 3))
    d[:, 2] = 1.0
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    t0 = np.concatenate([np.sort(rng.uniform(0.5, 4.0, c)) for c in counts]).astype(np.float32)
    t1 = (t0 + rng.uniform(0.002, 0.03, S).astype(np.float32)).astype(np.float32)
    field = _field(rng, G)
    # the arrays start `shift` elements into their allocation and end with it
    buf = [torch.full((S + shift,), float("nan"), dtype=torch.float32, device="cuda") for _ in range(2)]
    for b, v in zip(buf, (t0, t1)):
        b[shift:].copy_(torch.from_numpy(v))
    s = H.Samples(torch.from_numpy(off).cuda(), torch.zeros(S, dtype=torch.int32, device="cuda"),
                  buf[0][shift:], buf[1][shift:], S)
    rgba = to_np(H.composite(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), s,
                             torch.from_numpy(field).cuda())).astype(np.float64)
    ref = oracle.composite(o, d, off, t0, t1, field)
    assert np.abs(rgba - ref).max() <= TOL, np.abs(rgba - ref).max()
    assert ref[:, 3].max() > 0.5


@pytest.mark.parametrize("n", [1, 3, 4, 5, 33, 65535, 65536, 65541])
def test_ray_counts(H, n):
    # three samples on every seventh ray, none on the others
    rng = np.random.default_rng(n)
    counts = np.where(np.arange(n) % 7 == n % 7, 3, 0)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    S = int(off[-1])
    o = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
    d = torch.tensor([[0.6, 0.0, 0.8]] * n, dtype=torch.float32, device="cuda")
    s = H.alloc_samples(n, max(1, S))
    s.offsets.copy_(torch.from_numpy(off))
    t0 = np.array([0.5, 0.6, 0.9], np.float32)
    t1 = np.array([0.6, 0.7, 1.0], np.float32)
    s.t0[:S].copy_(torch.from_numpy(np.tile(t0, S // 3)))
    s.t1[:S].copy_(torch.from_numpy(np.tile(t1, S // 3)))
    field = _field(rng, 40)
    rgba = to_np(H.composite(o, d, s, torch.from_numpy(field).cuda())).astype(np.float64)
    want = oracle.composite(np.zeros((1, 3), np.float32), np.array([[0.6, 0.0, 0.8]], np.float32),
                            np.array([0, 3]), t0, t1, field)
    assert np.abs(rgba - np.where(counts[:, None] > 0, want, 0.0)).max() <= TOL
