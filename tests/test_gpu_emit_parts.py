"""The emit writes a tile of 32 rays with one warp, or with two, four or eight in calls of few
tiles, and a ray with more than 16 runs from its 16th run on by walking on from there.  Rays
across slabs, of 0 to 60 runs with 15 to 18 and 31 to 33 among them, in calls of every split and
in every form of the sampler, with room for all samples and with too little; the samples are the
oracle's."""
import numpy as np
import pytest
import torch

from paper_2404_10272_gb300 import scenes
from _helpers import gpu_samples, oracle_samples, sampler_form, to_np

pytestmark = pytest.mark.gpu
R = 128


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


@pytest.fixture(scope="module")
def slabs(H):
    rng = np.random.default_rng(31)
    occ = np.zeros((1, R, R, R), np.uint8)
    occ[:, ::2] = 1
    aabbs = np.array([[-1, -1, -1, 1, 1, 1]], np.float32)
    m = np.concatenate([[0, 1, 14, 15, 16, 17, 18, 31, 32, 33, 60], rng.integers(0, 61, 86)])
    n = m.size
    o = rng.uniform(-0.5, 0.5, (n, 3)).astype(np.float32)
    o[:, 0] = 1.0 - (m * 2 + 0.5) * (2.0 / R) - 0.05   # m slabs ahead of the nearest sample
    d = np.zeros((n, 3))
    d[:, 0] = 1.0
    d[:, 1:] = rng.uniform(-0.01, 0.01, (n, 2))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    p = scenes.SamplerParams(near=0.05, far=4.0, step=0.006, cone=0.0, max_step=1e10, max_steps=2000)
    ref = oracle_samples(o, d, occ, aabbs, p)
    off, ray, t0, t1 = ref
    new = np.ones(t0.size, bool)
    new[1:] = (ray[1:] != ray[:-1]) | (t0[1:] != t1[:-1])
    runs = np.bincount(ray[new], minlength=n)
    assert {15, 16, 17, 18, 31, 32, 33} <= set(runs.tolist()) and runs.min() == 0
    return occ, aabbs, o, d, p, ref


def _repeat(ref, idx):
    """The samples of rays `idx` of ref, in that order."""
    off, ray, t0, t1 = ref
    cnt = np.diff(off)[idx]
    noff = np.concatenate([[0], np.cumsum(cnt)])
    at = np.arange(noff[-1]) - np.repeat(noff[:-1] - off[:-1][idx], cnt)
    return noff, np.repeat(np.arange(idx.size), cnt), t0[at], t1[at]


@pytest.mark.parametrize("n", [1, 31, 97, 2081, 17000, 34100, 68200, 140001])
def test_splits(H, slabs, n):
    occ, aabbs, o, d, p, ref = slabs
    idx = np.random.default_rng(n).integers(0, o.shape[0], n)
    if n == 97:
        idx = np.arange(97)
    want = _repeat(ref, idx)
    ot, dt = torch.from_numpy(o[idx]).cuda(), torch.from_numpy(d[idx]).cuda()
    prm = H.make_params(p.near, p.far, p.step, p.cone, p.max_step, p.max_steps)
    g = H.build_vdb(torch.from_numpy(occ).cuda(), aabbs)
    gd = H.pack_dense(torch.from_numpy(occ).cuda(), aabbs)

    def same(got, total, what):
        assert np.array_equal(got[0], np.minimum(want[0], total)), what
        for u, v in zip(got[1:], want[1:]):
            k = min(total, len(v))   # a buffer has room for one sample at least
            assert np.array_equal(u[:k], v[:k]), what

    total = int(want[0][-1])
    for form in (H.SAMPLER_SEPARATE, H.SAMPLER_FUSED):
        with sampler_form(H, form):
            same(gpu_samples(H, "hdda", ot, dt, g, prm), total, "hdda")
            same(gpu_samples(H, "dense", ot, dt, gd, prm), total, "dense")
            for cap in (total, max(1, total - 3), max(1, total // 2)):
                out = H.alloc_samples(n, max(1, total))
                for t in (out.t0, out.t1):
                    t.fill_(-1.0)
                cut = H.Samples(out.offsets, out.ray_idx[:cap], out.t0[:cap], out.t1[:cap], 0)
                st = torch.zeros(1, dtype=torch.int32, device="cuda")
                H.traverse_async(ot, dt, g, prm, cut, st)
                torch.cuda.synchronize()
                assert (int(st.item()) != 0) == (cap < total)
                same([to_np(t) for t in (out.offsets, out.ray_idx, out.t0, out.t1)], cap, cap)
                assert (to_np(out.t0)[cap:total] == -1.0).all()
    job = H.alloc_samples(n, max(1, total))
    b = H.Batch([dict(rays_o=ot, rays_d=dt, grid=g, params=prm, out=job)])
    b.launch()
    b.results()
    same([to_np(t) for t in (job.offsets, job.ray_idx, job.t0, job.t1)], total, "batch")
    out = H.alloc_samples(n, max(1, total))
    H.traverse_hdda_noalloc(ot, dt, g, prm, out)
    same([to_np(t) for t in (out.offsets, out.ray_idx, out.t0, out.t1)], total, "noalloc")
