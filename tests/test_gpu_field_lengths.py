"""Ray directions of any length: parameters are in units of |d|, so a direction 2^x times as long
with parameters 2^-x times as large (and amplitudes 2^x times, which keeps the optical depths)
gives the same pixel.  Lengths whose square leaves the normal binary32 range among them; pixels
against the binary64 oracle within the compositor's 1e-5."""
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


@pytest.mark.parametrize("x", [-80, -60, -49, -20, 0, 20, 49, 60, 80])
@pytest.mark.parametrize("G", [20, 60, 100])
def test_direction_lengths(H, x, G):
    rng = np.random.default_rng(50 + G)
    counts = rng.choice([0, 1, 7, 40, 120], 60)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    S = int(off[-1])
    o = rng.uniform(-1.0, 1.0, (60, 3)).astype(np.float32)
    o[:, 2] -= 2.0
    d = rng.normal(0.0, 0.3, (60, 3))
    d[:, 2] = 1.0
    f = np.float32(2.0 ** x)
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32) * f
    t0 = np.concatenate([np.sort(rng.uniform(0.5, 4.0, c)) for c in counts]).astype(np.float32)
    t1 = (t0 + rng.uniform(0.002, 0.03, S).astype(np.float32)).astype(np.float32)
    t0, t1 = t0 / f, t1 / f
    field = np.zeros((G, 8), np.float32)
    field[:, :3] = rng.uniform(-1.5, 1.5, (G, 3))
    field[:, 3] = rng.uniform(0.05, 0.3, G)
    field[:, 4] = rng.uniform(0.5, 20.0, G).astype(np.float32) * f
    field[:, 5:] = rng.uniform(0.0, 1.0, (G, 3))
    s = H.Samples(torch.from_numpy(off).cuda(), torch.zeros(S, dtype=torch.int32, device="cuda"),
                  torch.from_numpy(t0).cuda(), torch.from_numpy(t1).cuda(), S)
    rgba = to_np(H.composite(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), s,
                             torch.from_numpy(field).cuda())).astype(np.float64)
    ref = oracle.composite(o, d, off, t0, t1, field)
    assert ref[:, 3].max() > 0.5
    assert np.abs(rgba - ref).max() <= TOL, np.abs(rgba - ref).max()
