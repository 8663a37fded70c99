"""The walk's per-level stretches and mirrored coordinates against the oracle, bit for bit: level
boxes that overlap in part, lie apart or share faces (at zero among them), so that a ray enters
and leaves levels in every order; directions of every sign, parallel to faces, and rays on
voxel and box faces; parameters that start behind the origin; closed-form and bucketed lattices;
odd resolutions, all walks and both sampler forms."""
import itertools

import numpy as np
import pytest
import torch

from paper_2404_10272_gb300 import scenes
from _helpers import assert_same, gpu_samples, oracle_samples, sampler_form

pytestmark = pytest.mark.gpu

BOXES = {
    "nested": [[-1, -1, -1, 1, 1, 1], [-2, -2, -2, 2, 2, 2], [-4, -4, -4, 4, 4, 4]],
    "shared faces at zero": [[0, 0, 0, 1, 1, 1], [-1, -1, -1, 0, 0, 0], [-1, -1, -1, 1, 1, 1]],
    "apart": [[-3, -1, -1, -2, 1, 1], [2, -1, -1, 3, 1, 1], [-0.3, -0.3, -5, 0.4, 0.4, 5]],
    "crossing": [[-2, -0.5, -0.5, 2, 0.5, 0.5], [-0.5, -2, -0.5, 0.5, 2, 0.5],
                 [-0.7, -0.7, -2.1, 0.7, 0.7, 1.9]],
    "one": [[-1.5, -1.5, -1.5, 1.5, 1.25, 1.0]],
}
LATTICES = {
    "constant": dict(near=0.0, far=9.0, step=0.013, cone=0.0, max_step=1e10),
    "growing": dict(near=0.02, far=60.0, step=0.004, cone=0.01, max_step=1e10),
    "capped, from behind": dict(near=-2.0, far=9.0, step=0.01, cone=0.02, max_step=0.05),
}


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


def _rays(rng, R):
    o, d = [], []
    for s in itertools.product([-1, 0, 1], repeat=3):  # axis-parallel, diagonal, zero
        for at in (0.0, 0.5, -0.25, 1.0, -2.0 / R):
            o.append([at - 3.0 * v for v in s])
            d.append(s)
    r = rng.normal(size=(600, 3))
    r /= np.linalg.norm(r, axis=1, keepdims=True)
    o += list(rng.uniform(-3.5, 3.5, (600, 3)))
    d += list(r * rng.uniform(0.3, 2.0, (600, 1)))
    return np.array(o, np.float32), np.array(d, np.float32)


@pytest.mark.parametrize("lattice", list(LATTICES))
@pytest.mark.parametrize("boxes", list(BOXES))
@pytest.mark.parametrize("R", [7, 16])
def test_walks_match_the_oracle(H, boxes, lattice, R):
    rng = np.random.default_rng(len(boxes) * 100 + len(lattice) + R)
    aabbs = np.array(BOXES[boxes], np.float32)
    occ = scenes.random_grid(rng, len(aabbs), R, 0.3)
    occ[:, R // 2:, : R // 2] = 0      # empty and full blocks beside the noise
    occ[:, : R // 2, R // 2:] = 1
    o, d = _rays(rng, R)
    p = scenes.SamplerParams(**LATTICES[lattice])
    ref = oracle_samples(o, d, occ, aabbs, p)
    assert ref[0][-1] > 0
    dense = torch.from_numpy(occ).cuda()
    ot, dt = torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda()
    prm = H.make_params(p.near, p.far, p.step, p.cone, p.max_step, p.max_steps)
    gd, gv = H.pack_dense(dense, aabbs), H.build_vdb(dense, aabbs)
    for form in (H.SAMPLER_SEPARATE, H.SAMPLER_FUSED):
        with sampler_form(H, form):
            assert_same(gpu_samples(H, "dense", ot, dt, gd, prm), ref, "dense")
            assert_same(gpu_samples(H, "hdda", ot, dt, gv, prm), ref, "hdda")
            gv.set_refine(False)
            assert_same(gpu_samples(H, "hdda", ot, dt, gv, prm), ref, "plain")
            gv.set_refine(True)
    gv.set_walk(H.WALK_SKIP)
    assert_same(gpu_samples(H, "hdda", ot, dt, gv, prm), ref, "skip")
    gv.set_walk(H.WALK_BRANCH)
    out = H.alloc_samples(o.shape[0], int(ref[0][-1]))
    H.traverse_hdda_noalloc(ot, dt, gv, prm, out)
    assert_same(tuple(t.cpu().numpy() for t in out.trimmed()), ref, "noalloc")
    job = H.alloc_samples(o.shape[0], int(ref[0][-1]))
    b = H.Batch([dict(rays_o=ot, rays_d=dt, grid=gv, params=prm, out=job)])
    b.launch()
    b.results()
    assert_same(tuple(t.cpu().numpy() for t in job.trimmed()), ref, "batch")
