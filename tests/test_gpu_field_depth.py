"""Long rays of equal samples: the roundings of a transmittance taken as a product of (1 - alpha)
all go one way there (here 0.45 of a unit of 2^-24 per sample, 2e-5 of opacity in all), those of a
sum of optical depths do not.  n samples of a constant density, optical depth 1 in all; against
the binary64 oracle.  Tolerance: the sum is rounded once per 32 samples and within a step, each
time by at most 2^-24 of it; the density, opacity and exponentials add a few units more."""
import numpy as np
import pytest
import torch

import oracle
from _helpers import to_np

pytestmark = pytest.mark.gpu
N = 2048
TOL = 2.0 ** -24 * (N / 32 + 16)


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


@pytest.mark.parametrize("path", ["composite", "render"])
@pytest.mark.parametrize("blobs", [1, 65])
def test_equal_samples(H, path, blobs):
    h = 2.0 ** -10
    f = 1.0 - (8192 + 0.45) * 2.0 ** -24  # 1 - alpha, 0.45 units from a binary32 value
    field = np.zeros((blobs, 8), np.float32)
    field[:, 3] = 0.1
    field[0] = [0, 0, 0, 1e6, -np.log(f) / h, 0.2, 0.5, 0.9]
    o = np.tile(np.array([[0.0, 0.25, -0.25]], np.float32), (5, 1))
    d = np.tile(np.array([[1.0, 0.0, 0.0]], np.float32), (5, 1))
    t = np.arange(N + 1, dtype=np.float32) * np.float32(h)
    off = np.arange(6, dtype=np.int64) * N
    t0, t1 = np.tile(t[:-1], 5), np.tile(t[1:], 5)
    ot, dt, ft = (torch.from_numpy(v).cuda() for v in (o, d, field))
    if path == "composite":
        s = H.Samples(torch.from_numpy(off).cuda(), torch.zeros(5 * N, dtype=torch.int32, device="cuda"),
                      torch.from_numpy(t0).cuda(), torch.from_numpy(t1).cuda(), 5 * N)
        rgba = H.composite(ot, dt, s, ft)
    else:
        occ = torch.ones((1, 8, 8, 8), dtype=torch.uint8, device="cuda")
        g = H.build_vdb(occ, np.array([[-4, -4, -4, 4, 4, 4]], np.float32))
        rgba = H.render(ot, dt, g, H.make_params(0.0, N * h, h), ft)
    ref = oracle.composite(o, d, off, t0, t1, field)
    assert abs(ref[0, 3] - (1.0 - np.exp(-1.0))) < 0.01
    assert np.abs(to_np(rgba).astype(np.float64) - ref).max() <= TOL
