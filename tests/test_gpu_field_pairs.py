"""The compositor looks at two blobs per lane, 64 per step: fields whose last step is empty in
one half, ends within either, or fills both, up to the largest field.  Every blob counts (each has
its own place and colour along the rays); pixels against the binary64 oracle within the
compositor's 1e-5."""
import numpy as np
import pytest
import torch

import oracle
from _helpers import to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


@pytest.mark.parametrize("G", [1, 31, 32, 34, 63, 96, 97, 127, 128, 129, 160, 192, 225, 255, 256])
def test_field_sizes(H, G):
    rng = np.random.default_rng(8000 + G)
    n, c = 37, 70
    o = rng.uniform(-0.3, 0.3, (n, 3)).astype(np.float32)
    o[:, 2] -= 3.0
    d = rng.normal(0.0, 0.1, (n, 3))
    d[:, 2] = 1.0
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    off = (np.arange(n + 1) * c).astype(np.int64)
    t0 = np.tile((1.5 + 3.0 * np.arange(c) / c).astype(np.float32), n)
    t1 = (t0 + np.float32(0.04)).astype(np.float32)
    # narrow blobs one behind the other, in an order that mixes the steps' halves
    field = np.zeros((G, 8), np.float32)
    field[:, 2] = (-1.5 + 3.0 * (np.arange(G) + 0.5) / G)[rng.permutation(G)]
    field[:, :2] = rng.uniform(-0.2, 0.2, (G, 2))
    field[:, 3] = rng.uniform(0.05, 0.2, G)
    field[:, 4] = 40.0 / G
    field[:, 5:] = rng.uniform(0.0, 1.0, (G, 3))
    s = H.Samples(torch.from_numpy(off).cuda(), torch.zeros(n * c, dtype=torch.int32, device="cuda"),
                  torch.from_numpy(t0).cuda(), torch.from_numpy(t1).cuda(), n * c)
    rgba = to_np(H.composite(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), s,
                             torch.from_numpy(field).cuda())).astype(np.float64)
    ref = oracle.composite(o, d, off, t0, t1, field)
    assert ref[:, 3].max() > 0.1
    assert np.abs(rgba - ref).max() <= 1e-5
