"""Render-only rays of 0 to 64 runs side by side, so that a warp's lane groups need a different
number of rounds of 16 runs each: a group that walks on has the others walk ahead too.  In tasks
of four and of eight rays; the fused call's samples equal the sampler's bit for bit, its frame the
render-only one, and pixels the binary64 oracle's within the compositor's 1e-5."""
import numpy as np
import pytest
import torch

import oracle
from _helpers import slab_scene, to_np

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


@pytest.mark.parametrize("n", [703, 65603])
@pytest.mark.parametrize("kind", ["refined", "plain", "dense"])
@pytest.mark.parametrize("blobs", [8, 70])
def test_mixed_rounds(H, n, kind, blobs):
    occ, aabbs, o, d, field, p = slab_scene(128, 2, n, 31 + n)
    rng = np.random.default_rng(n + blobs)
    last = rng.permutation([0, 0, 8, 20, 40, 60, 90, 128] * 2).repeat(8)  # where slabs end, by y
    occ[0] *= (np.arange(128)[:, None] < last[None, :]).astype(np.uint8)[:, :, None]
    field = np.concatenate([field, np.repeat(field[:1], blobs - 8, 0)])
    field[8:, 4] = 0.01
    ot, dt, ft = (torch.from_numpy(v).cuda() for v in (o, d, field))
    prm = H.make_params(p.near, p.far, p.step, p.cone, p.max_step, p.max_steps)
    dense = torch.from_numpy(occ).cuda()
    g = H.pack_dense(dense, aabbs) if kind == "dense" else H.build_vdb(dense, aabbs)
    if kind == "plain":
        g.set_refine(False)
    s = (H.traverse_dense if kind == "dense" else H.traverse_hdda)(ot, dt, g, prm)
    off, _, t0, t1 = (to_np(x) for x in s.trimmed())
    sel = np.arange(0, n, max(1, n // 600))
    runs = [int((t0[a + 1:b] != t1[a:b - 1]).sum()) + 1 if b > a else 0
            for a, b in zip(off[sel], off[sel + 1])]
    assert min(runs) == 0 and max(runs) > 48 and 0.2 < np.mean(np.array(runs) > 16) < 0.8
    frame = H.render(ot, dt, g, prm, ft)
    out = H.alloc_samples(n, s.total)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    both = H.traverse_composite(ot, dt, g, prm, out, ft, st)
    assert int(st.item()) == 0 and torch.equal(both, frame)
    for x, y in ((out.offsets, s.offsets), (out.ray_idx, s.ray_idx), (out.t0, s.t0), (out.t1, s.t1)):
        assert torch.equal(x, y)
    sub = np.concatenate([[0], np.cumsum(off[sel + 1] - off[sel])])
    idx = np.concatenate([np.arange(off[r], off[r + 1]) for r in sel])
    want = oracle.composite(o[sel], d[sel], sub, t0[idx], t1[idx], field)
    assert np.abs(to_np(frame)[sel].astype(np.float64) - want).max() <= TOL
