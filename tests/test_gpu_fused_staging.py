"""The fused sampler form at the edges of what its CTAs hold in shared memory: the record lists
leave 101,120 bytes for the walk's tables, where the separate form stages up to 131,072.  A small
grid with a lattice of K steps needs 4 K + 8200 + 1920 bytes (plain tree: 1540 more, rounded up to
16).  Both forms give the same samples on either side of both limits, in every kind of walk."""
import numpy as np
import pytest
import torch

from _helpers import assert_same, oracle_samples, sampler_form, to_np
from paper_2404_10272_gb300 import scenes

pytestmark = pytest.mark.gpu

LAST_FUSED, LAST_SEPARATE = (101120 - 10120) // 4, (131072 - 10120) // 4


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


@pytest.mark.parametrize("K", [LAST_FUSED - 400, LAST_FUSED, LAST_FUSED + 1, 25000, LAST_SEPARATE,
                               LAST_SEPARATE + 1])
@pytest.mark.parametrize("kind", ["dense", "refined", "plain"])
def test_both_forms_agree(H, K, kind):
    rng = np.random.default_rng(K)
    occ = (rng.random((1, 16, 16, 16)) < 0.02).astype(np.uint8)
    boxes = np.array([[-1, -1, -1, 1, 1, 1]], np.float32)
    n = 100
    o = rng.uniform(-1.0, 1.0, (n, 3)).astype(np.float32)
    d = rng.normal(size=(n, 3))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    p = scenes.SamplerParams(near=0.0, far=K * 2.0 ** -13, step=2.0 ** -13)
    prm = H.make_params(p.near, p.far, p.step, p.cone, p.max_step, p.max_steps)
    dense = torch.from_numpy(occ).cuda()
    grid = H.pack_dense(dense, boxes) if kind == "dense" else H.build_vdb(dense, boxes)
    if kind == "plain":
        grid.set_refine(False)
    fn = H.traverse_dense if kind == "dense" else H.traverse_hdda
    ot, dt = torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda()
    want = tuple(to_np(x) for x in fn(ot, dt, grid, prm).trimmed())
    with sampler_form(H, H.SAMPLER_FUSED):
        got = tuple(to_np(x) for x in fn(ot, dt, grid, prm).trimmed())
    assert want[0][-1] > 100
    assert_same(got, want, f"fused {kind}, {K} steps")
    if kind == "refined" and K == 25000:
        assert_same(got, oracle_samples(o, d, occ, boxes, p), "oracle")
