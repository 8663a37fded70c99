"""Nearly transparent rays, whose opacity the compositor takes from a product in a fixed order:
segments of 64 places counted from the first of four rays, steps of 32 samples from positions
rounded down to a multiple of four.  Lengths around both, ray opacities on both sides of the
limit (0.02), arrays that do and do not allow 16-byte loads; opacities against the binary64
oracle.  Tolerance: n factors and as many products, each rounded by 2^-25 near 1, and 1e-5 of the
opacity for the samples' own."""
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


@pytest.mark.parametrize("first", [0, 1, 2, 3, 27, 61])
@pytest.mark.parametrize("shift", [0, 1])
def test_faint_rays(H, first, shift):
    rng = np.random.default_rng(7000 + 10 * first + shift)
    counts = np.array([first, 1, 2, 3, 60, 61, 62, 63, 64, 65, 66, 31, 32, 33, 0, 127, 128, 129, 130,
                       0, 300, 5, 95, 96, 97, 257] + [int(c) for c in rng.integers(1, 200, 20)])
    n = counts.size
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    S = int(off[-1])
    o = np.tile(np.array([[0.0, 0.0, -2.0]], np.float32), (n, 1))
    d = np.tile(np.array([[0.0, 0.0, 1.0]], np.float32), (n, 1))
    t0 = np.concatenate([np.sort(rng.uniform(1.0, 3.0, c)) for c in counts]).astype(np.float32)
    t1 = (t0 + 0.005).astype(np.float32)
    # wide blobs of a density that gives the rays an opacity around 0.02
    field = np.zeros((40, 8), np.float32)
    field[:, :3] = rng.uniform(-0.5, 0.5, (40, 3))
    field[:, 3] = rng.uniform(0.5, 1.0, 40)
    field[:, 4] = 0.002
    field[:, 5:] = rng.uniform(0.0, 1.0, (40, 3))
    buf = [torch.full((S + shift,), float("nan"), dtype=torch.float32, device="cuda") for _ in range(2)]
    for b, v in zip(buf, (t0, t1)):
        b[shift:].copy_(torch.from_numpy(v))
    s = H.Samples(torch.from_numpy(off).cuda(), torch.zeros(S, dtype=torch.int32, device="cuda"),
                  buf[0][shift:], buf[1][shift:], S)
    rgba = to_np(H.composite(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), s,
                             torch.from_numpy(field).cuda())).astype(np.float64)
    ref = oracle.composite(o, d, off, t0, t1, field)
    a = ref[:, 3]
    assert a.min() == 0.0 and 0.001 < np.quantile(a, 0.3) < 0.02 < np.quantile(a, 0.9) < 0.1
    assert (np.abs(rgba[:, 3] - a) <= counts * 2.0 ** -24 + 1e-5 * a).all()
    assert np.abs(rgba[:, :3] - ref[:, :3]).max() <= 1e-5
