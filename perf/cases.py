"""What users of this package have it do, as measurable cases: sample, composite and render
frames, build and update occupancy grids between training batches, and sample many cameras in
one batch.  Every input is made on the GPU from a seed: occupancy with the shapes of the three
workload families (coarse shells, object-centric, unbounded cascade), pinhole cameras, random
training rays and Gaussian-blob fields.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2404_10272_gb300 import hdda

# Scene families.  `samples`: kept samples per image ray, `blobs`: blobs (of 64) within 7
# standard deviations of a sample; both are averages over many seeds, for work().  `room`: the
# samples per ray that a program keeps room for.
FAMILIES = {
    "shells": dict(half=1.5, near=2.0, far=6.0, step=5e-3, cone=0.0, fov=0.69, samples=45.0, blobs=7.6, room=96),
    "object": dict(half=1.5, near=2.0, far=6.0, step=math.sqrt(3.0) * 3.0 / 1024.0, cone=0.0,
                   fov=0.69, samples=53.0, blobs=9.4, room=128),
    "unbounded": dict(half=1.0, near=0.02, far=1e3, step=1.73e-3, cone=0.004, fov=1.0,
                      samples=190.0, blobs=8.1, room=448),
}
MAX_STEP = 1e10


def _case(name, kind, scene, res, levels, width, height, **more):
    c = dict(name=name, kind=kind, scene=scene, res=res, levels=levels, width=width,
             height=height, blobs=64)
    c.update(more)
    return c


def listed():
    return [
        # a preview-sized frame, sampled and composited in stream order: launches and latency
        _case("tiny_frame", "frame", "shells", 64, 1, 96, 96, rebuild=False),
        # the sampler alone on the object-centric test frame; the consumer is the user's own model
        _case("object_sample", "sample", "object", 128, 1, 800, 800, grid="vdb"),
        # the sampler alone on an unbounded capture: a four-level cascade, growing steps
        _case("unbounded_sample", "sample", "unbounded", 128, 4, 1245, 825, grid="vdb"),
        # the dense-grid DDA that the hierarchical one is compared with, on the same frame
        _case("object_dense_sample", "sample", "object", 128, 1, 800, 800, grid="dense"),
        # compositing of stored samples: an object frame of short rays, many of them empty ...
        _case("object_composite", "composite", "object", 128, 1, 800, 800),
        # ... and an unbounded frame, whose rays are long
        _case("unbounded_composite", "composite", "unbounded", 128, 4, 1245, 825),
        # a server's largest request, without sample buffers
        _case("hd_render", "render", "object", 128, 1, 1920, 1080),
        # a server's small request of an odd size, from a two-level cascade
        _case("small_render", "render", "shells", 64, 2, 253, 187),
        # the whole unbounded frame: the occupancy changed, so rebuild, then sample and composite
        _case("unbounded_frame", "frame", "unbounded", 128, 4, 1245, 825, rebuild=True),
        # two training steps on a 128^3 grid: 1 % of the blocks change, then an odd number of
        # random rays is sampled, the total read by the host
        _case("train_update", "train", "object", 128, 1, 16381, 1, rebuild=False),
        # two training steps on a large cascade, each with a full rebuild
        _case("train_rebuild", "train", "object", 512, 2, 65536, 1, rebuild=True),
        # 64 cameras over small and object scenes of 1 to 4 levels in one batch
        _case("batch", "batch", "object", 128, 4, 800, 800, jobs=64),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["frame", "sample", "sample", "composite", "render", "train", "batch"])
    scene = rng.choice(["shells", "object", "unbounded"])
    levels = rng.randint(2, 4) if scene == "unbounded" else rng.randint(1, 3)
    res = 4 * rng.randint(16, 40)
    if levels == 1:
        res += rng.randint(-3, 3)
    most = (1245, 825) if scene == "unbounded" else (1920, 1080)
    c = dict(kind=kind, scene=scene, res=res, levels=levels, width=log_int(64, most[0]),
             height=log_int(64, most[1]), blobs=rng.randint(32, 64))
    if kind == "frame":
        c["rebuild"] = rng.random() < 0.5
    elif kind == "sample":
        c["grid"] = rng.choice(["vdb", "vdb", "dense"])
    elif kind == "train":
        c.update(scene=rng.choice(["shells", "object"]), width=log_int(1024, 65536), height=1,
                 rebuild=rng.random() < 0.5, levels=rng.randint(1, 2), res=4 * rng.randint(16, 128))
    elif kind == "batch":
        c.update(scene=rng.choice(["shells", "object"]), jobs=rng.randint(2, 48), res=4 * rng.randint(16, 32),
                 width=log_int(96, 800), height=log_int(96, 800))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _boxes(levels, half):
    out = np.zeros((levels, 6), np.float32)
    for l in range(levels):
        h = half * 2.0 ** l
        out[l] = [-h, -h, -h, h, h, h]
    return out


def _axis(res, half):
    return (torch.arange(res, device="cuda", dtype=torch.float32) + 0.5) * (2.0 * half / res) - half


def _add_ellipsoids(occ, half, rng, n, centre, axes, thickness):
    """Marks voxels near the surface of n random ellipsoids, or inside them (thickness None)."""
    x = _axis(occ.shape[0], half)
    for _ in range(n):
        c, a = rng.uniform(-centre, centre, 3), rng.uniform(axes[0], axes[1], 3)
        q, r = np.linalg.qr(rng.normal(size=(3, 3)))
        m = (q * np.sign(np.diag(r))) / a
        rho = None
        for j in range(3):
            px, py, pz = ((x - float(c[k])) * float(m[k, j]) for k in range(3))
            p = px[:, None, None] + py[None, :, None] + pz[None, None, :]
            rho = p.mul_(p) if rho is None else rho.add_(p.mul_(p))
        rho.sqrt_()
        occ |= rho <= 1.0 if thickness is None else (rho - 1.0).abs_() <= thickness / float(a.min())


def _dilate(occ):
    o = occ[None, None].to(torch.float16)
    for axis in range(3):
        k = [1, 1, 1]
        k[axis] = 3
        o = torch.nn.functional.max_pool3d(o, k, stride=1, padding=[(v - 1) // 2 for v in k])
    return o[0, 0] > 0


def _add_boxes(occ, half, rng, n, lo, hi):
    """Marks n random boxes centred outside the next finer level's box."""
    x = _axis(occ.shape[0], half).cpu().numpy()
    while n:
        c = rng.uniform(-half, half, 3)
        if np.all(np.abs(c) < 0.5 * half):
            continue
        e = rng.uniform(lo, hi, 3) * half
        b = np.searchsorted(x, np.stack([c - e, c + e]))
        occ[b[0, 0]:b[1, 0], b[0, 1]:b[1, 1], b[0, 2]:b[1, 2]] = True
        n -= 1


def _occupancy(scene, res, levels, rng):
    """uint8 [levels, res, res, res] on the GPU."""
    half = FAMILIES[scene]["half"]
    occ = torch.zeros((levels, res, res, res), dtype=torch.bool, device="cuda")
    if scene == "shells":
        _add_ellipsoids(occ[0], half, rng, 3, 0.8, (0.3, 0.9), 0.05)
    elif scene == "object":
        _add_ellipsoids(occ[0], half, rng, 8, 0.6, (0.25, 0.8), 0.006)
        _add_ellipsoids(occ[0], half, rng, 2, 0.5, (0.1, 0.25), None)
        occ[0] = _dilate(occ[0])
    else:
        _add_ellipsoids(occ[0], half, rng, 6, 0.4, (0.2, 0.6), 0.008)
        occ[0] = _dilate(occ[0])
    for l in range(1, levels):
        if scene == "unbounded":
            _add_boxes(occ[l], half * 2.0 ** l, rng, int(rng.integers(20, 201)), 0.02, 0.12)
        else:  # the finer level, pooled, in the middle, and some clutter around it
            q = res // 4
            p = occ[l - 1].reshape(res // 2, 2, res // 2, 2, res // 2, 2).amax((1, 3, 5))
            occ[l, q:q + res // 2, q:q + res // 2, q:q + res // 2] = p
            _add_boxes(occ[l], half * 2.0 ** l, rng, 12, 0.03, 0.1)
    return occ.to(torch.uint8)


def _camera(scene, rng):
    """Eye and unit axes (forward, right, up) of a pinhole camera, float64."""
    if scene == "unbounded":
        eye, f = rng.uniform(-0.5, 0.5, 3), rng.normal(size=3)
    else:
        az, el = rng.uniform(0.0, 2.0 * math.pi), rng.uniform(0.1, 1.2)
        eye = 4.0 * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
        f = -eye
    f = f / np.linalg.norm(f)
    up = np.array([0.0, 0.0, 1.0]) if abs(f[2]) < 0.999 else np.array([0.0, 1.0, 0.0])
    r = np.cross(f, up)
    r /= np.linalg.norm(r)
    return np.stack([eye, f, r, np.cross(r, f)])


def _rays(cam, u, v):
    """float32 origins and unit directions through image-plane points (u, v), float64 tensors."""
    eye, f, r, up = (torch.as_tensor(cam[..., k, :], device="cuda") for k in range(4))
    d = f + u[:, None] * r + v[:, None] * up
    d = (d / d.norm(dim=-1, keepdim=True)).float()
    return eye.expand(d.shape).float().contiguous(), d.contiguous()


def _image_rays(scene, width, height, rng):
    th = math.tan(0.5 * FAMILIES[scene]["fov"])
    x = torch.arange(width, device="cuda", dtype=torch.float64)
    y = torch.arange(height, device="cuda", dtype=torch.float64)
    u = ((x + 0.5) / width * 2.0 - 1.0) * th
    v = (1.0 - (y + 0.5) / height * 2.0) * (th * height / width)
    v, u = torch.meshgrid(v, u, indexing="ij")
    return _rays(_camera(scene, rng), u.reshape(-1), v.reshape(-1))


def _random_rays(scene, n, rng):
    """Random pixels of 20 square images, in random order."""
    cams = np.stack([_camera(scene, rng) for _ in range(20)])[rng.integers(0, 20, n)]
    th = math.tan(0.5 * FAMILIES[scene]["fov"])
    uv = torch.as_tensor(rng.uniform(-th, th, (2, n)), device="cuda")
    return _rays(cams, uv[0], uv[1])


def _field(n, rng):
    d = rng.normal(size=(n, 3))
    d *= (0.9 + rng.uniform(-0.35, 0.35, (n, 1))) / np.linalg.norm(d, axis=-1, keepdims=True)
    f = np.concatenate([d, rng.uniform(0.03, 0.15, (n, 1)), rng.uniform(5.0, 50.0, (n, 1)),
                        rng.uniform(0.0, 1.0, (n, 3))], axis=1)
    return torch.as_tensor(f.astype(np.float32), device="cuda")


def _changed(dense, rng):
    """The grid after an occupancy update: one voxel flipped in 1 % of its 8^3 blocks, and the
    indices of those blocks."""
    L, R = dense.shape[0], dense.shape[1]
    B = (R + 7) // 8
    blk = rng.choice(L * B ** 3, max(1, L * B ** 3 // 100), replace=False)
    l, b = blk // B ** 3, blk % B ** 3
    x, y, z = (np.minimum(8 * q + rng.integers(0, 8, blk.size), R - 1)
               for q in (b // (B * B), (b // B) % B, b % B))
    new = dense.clone()
    at = tuple(torch.as_tensor(q, device="cuda") for q in (l, x, y, z))
    new[at] = 1 - new[at]
    return new, torch.as_tensor(blk.astype(np.int64), device="cuda")


def _job_sizes(case):
    """The image sizes of a batch: part of the case, not of the seed."""
    rng = np.random.default_rng([case["jobs"], case["width"], case["height"]])
    return [(int(rng.integers(64, case["width"] + 1)), int(rng.integers(64, case["height"] + 1)),
             int(rng.integers(0, 2 * case["levels"]))) for _ in range(case["jobs"])]


def _room(case, scene, n_rays):
    """Sample buffer size for n_rays rays; training batches keep room for the worst."""
    return 4 * n_rays * (80 if case["kind"] == "train" else FAMILIES[scene]["room"] // 4)


def _inputs(case, seed):
    """Everything a case is made of, in plain tensors (shared by prepare and exact)."""
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, case["res"], case["width"]])
    scene, res, levels = case["scene"], case["res"], case["levels"]
    fam = FAMILIES[scene]
    s = {"boxes": _boxes(levels, fam["half"]), "field": _field(case["blobs"], rng)}
    if case["kind"] == "batch":  # jobs over one scene per (family, number of levels)
        names = ["shells", "object"]
        s["scenes"] = [(f, _occupancy(f, 64 if f == "shells" else res, l, rng), _boxes(l, 1.5))
                       for f in names for l in range(1, levels + 1)]
        s["jobs"] = [(k, *_image_rays(s["scenes"][k][0], w, h, rng)) for w, h, k in _job_sizes(case)]
        return s
    s["dense"] = _occupancy(scene, res, levels, rng)
    if case["kind"] == "train":
        s["dense2"], s["blocks"] = _changed(s["dense"], rng)
        s["rays"] = [_random_rays(scene, case["width"], rng) for _ in range(2)]
    else:
        s["rays"] = [_image_rays(scene, case["width"], case["height"], rng)]
    return s


def _params(scene, width):
    f = FAMILIES[scene]
    return hdda.make_params(f["near"], f["far"], f["step"], f["cone"], MAX_STEP, image_width=width)


def _zero_samples(n_rays, room):
    out = hdda.alloc_samples(n_rays, room)
    for t in (out.ray_idx, out.t0, out.t1):
        t.zero_()
    return out


def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"], s["rebuild"] = case["kind"], case.get("rebuild", False)
    s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    if s["kind"] == "batch":
        grids = [(hdda.build_vdb(dense, boxes), _params(f, 0)) for f, dense, boxes in s["scenes"]]
        # one allocation per output array; every job's part starts 16-byte aligned
        n_off = [(o.shape[0] + 2) // 2 * 2 for _, o, _ in s["jobs"]]
        n_smp = [_room(case, s["scenes"][k][0], o.shape[0]) for k, o, _ in s["jobs"]]
        whole = [torch.zeros(sum(n), dtype=t, device="cuda") for n, t in
                 ((n_off, torch.int64), (n_smp, torch.int32), (n_smp, torch.float32), (n_smp, torch.float32))]
        parts = [w.split(n) for w, n in zip(whole, (n_off, n_smp, n_smp, n_smp))]
        jobs = []
        for j, (k, o, d) in enumerate(s["jobs"]):
            out = hdda.Samples(parts[0][j][:o.shape[0] + 1], *(p[j] for p in parts[1:]), 0)
            jobs.append(dict(rays_o=o, rays_d=d, grid=grids[k][0], params=grids[k][1], out=out))
        s.update(whole=whole, batch=hdda.Batch(jobs))
        return s
    width = 0 if s["kind"] == "train" else case["width"]
    s["params"] = _params(case["scene"], width)
    build = hdda.pack_dense if case.get("grid") == "dense" else hdda.build_vdb
    s["grid"] = build(s["dense"], s["boxes"])
    o, d = s["rays"][0]
    if s["kind"] in ("frame", "sample", "train"):
        s["out"] = [_zero_samples(o.shape[0], _room(case, case["scene"], o.shape[0])) for o, _ in s["rays"]]
    elif s["kind"] == "composite":
        s["out"] = [hdda.traverse_hdda(o, d, s["grid"], s["params"])]
    return s


def run(state):
    s = state
    if s["kind"] == "batch":
        s["batch"].launch()
        return s["whole"]
    grid, prm = s["grid"], s["params"]
    if s["kind"] == "train":  # two steps; the second brings the first occupancy back
        got = []
        for dense, (o, d), out in zip((s["dense2"], s["dense"]), s["rays"], s["out"]):
            if s["rebuild"]:
                grid.rebuild(dense)
            else:
                grid.update(dense, s["blocks"], status=s["status"])
            out = hdda.traverse_hdda(o, d, grid, prm, out)
            got.append([out.offsets, out.ray_idx, out.t0, out.t1, out.total])
        return got
    o, d = s["rays"][0]
    if s["kind"] == "render":
        return [hdda.render(o, d, grid, prm, s["field"], status=s["status"])]
    if s["kind"] == "composite":
        return [hdda.composite(o, d, s["out"][0], s["field"])]
    if s["rebuild"]:
        grid.rebuild(s["dense"])
    out = hdda.traverse_async(o, d, grid, prm, s["out"][0], s["status"])
    got = [out.offsets, out.ray_idx, out.t0, out.t1]
    if s["kind"] == "frame":
        got.append(hdda.composite(o, d, out, s["field"]))
    return got


def work(case):
    """Rays, occupancy and field read once, every output written once; per sample, the blobs in
    reach at 12 operations each (the exponent along the ray 4, the exponential, four sums 7)."""
    fam = FAMILIES[case["scene"]]
    kind, voxels = case["kind"], case["levels"] * case["res"] ** 3
    grid = voxels / 8  # the bit array; the tree is of the same order
    if kind == "batch":
        n = sum(w * h for w, h, _ in _job_sizes(case))
        s = n * 0.5 * (FAMILIES["shells"]["samples"] + FAMILIES["object"]["samples"])
        return {"bytes": 32 * n + 12 * s + 2 * grid, "flops": 0}
    n = case["width"] * case["height"]
    s = n * fam["samples"]
    field = 12 * s * fam["blobs"] * case["blobs"] / 64
    if kind == "train":
        changed = voxels if case["rebuild"] else voxels / 100
        return {"bytes": 2 * (changed + grid + 32 * n + 12 * s), "flops": 0}
    if kind == "render":
        return {"bytes": 40 * n + grid, "flops": field}
    if kind == "composite":
        return {"bytes": 48 * n + 8 * s, "flops": field}
    sample = 32 * n + 12 * s + (voxels if case.get("rebuild") else 0) + grid
    if kind == "sample":
        return {"bytes": sample, "flops": 0}
    return {"bytes": sample + 16 * n, "flops": field}


# ---------------------------------------------------------------------------
# plain restatement
# ---------------------------------------------------------------------------

def _lattice(scene):
    """The shared lattice t_0, t_1, ...: a binary32 recurrence by definition."""
    f = FAMILIES[scene]
    near, far, step, cone, cap = (np.float32(v) for v in (f["near"], f["far"], f["step"], f["cone"], MAX_STEP))
    t = [near]
    while True:
        nxt = t[-1] + min(max(t[-1] * cone, step), cap)
        if nxt > far:
            return torch.as_tensor(np.array(t, np.float32), device="cuda")
        t.append(nxt)


def _kept(o, d, dense, boxes, t):
    """Every lattice interval of every ray whose midpoint (binary32, by definition) falls in an
    occupied voxel of the finest level holding it: bool [rays, intervals]."""
    L, R = dense.shape[0], dense.shape[1]
    tm = (t[:-1] + t[1:]) * 0.5
    x = [tm[None, :] * d[:, c, None] for c in range(3)]
    for c in range(3):
        x[c] += o[:, c, None]
    keep = torch.zeros(x[0].shape, dtype=torch.bool, device="cuda")
    free = torch.ones_like(keep)
    for l in range(L):
        lo, hi = boxes[l, :3], boxes[l, 3:]
        inside = free.clone()
        lin = torch.zeros(keep.shape, dtype=torch.int32, device="cuda")
        for c in range(3):
            inside &= (x[c] >= float(lo[c])) & (x[c] < float(hi[c]))
            scale = float(np.float32(R) / np.float32(hi[c] - lo[c]))
            i = (x[c] - float(lo[c])).mul_(scale).floor_().clamp_(0, R - 1)
            lin = lin.mul_(R).add_(i.to(torch.int32))
        at = inside.nonzero(as_tuple=True)
        keep[at] = dense[l].reshape(-1)[lin[at].long()] != 0
        free &= ~inside
    return keep


def _samples(o, d, dense, boxes, scene, room=None):
    """[offsets, ray_idx, t0, t1] of all rays: cut off at `room` samples and zero behind the
    last one, or, without it, just as many as there are."""
    t = _lattice(scene)
    counts, idx, ks = [], [], []
    step = max(1, (1 << 26) // max(1, t.numel()))
    for a in range(0, o.shape[0], step):
        keep = _kept(o[a:a + step], d[a:a + step], dense, boxes, t)
        counts.append(keep.sum(1))
        r, k = keep.nonzero(as_tuple=True)
        idx.append((r + a).to(torch.int32))
        ks.append(k.to(torch.int32))
    off = torch.zeros(o.shape[0] + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.cat(counts), 0, out=off[1:])
    k = torch.cat(ks)
    out = [torch.cat(idx), t[k], t[k + 1]]
    if room is not None:
        off.clamp_(max=room)
        out = [torch.nn.functional.pad(v[:room], (0, max(0, room - v.numel()))) for v in out]
    return [off, *out]


def _composite64(o, d, smp, field):
    """Front-to-back accumulation in binary64."""
    off, idx, t0, t1 = smp
    f = field.double()
    mu, a, rgb = f[:, :3], f[:, 4], f[:, 5:8]
    coef = -0.5 / f[:, 3] ** 2
    n = o.shape[0]
    rgba = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    ends = off.cpu().numpy()
    r0 = 0
    while r0 < n:  # as many whole rays at once as hold about four million samples
        r1 = max(r0 + 1, int(np.searchsorted(ends, ends[r0] + (1 << 22), "right")) - 1)
        b, e = int(ends[r0]), int(ends[r1])
        if e > b:
            i = idx[b:e].long()
            ta, tb = t0[b:e].double(), t1[b:e].double()
            x = o[i].double() + (0.5 * (ta + tb))[:, None] * d[i].double()
            w = torch.zeros((e - b, f.shape[0]), dtype=torch.float64, device="cuda")
            for c in range(3):
                w += (x[:, c, None] - mu[None, :, c]) ** 2
            w = w.mul_(coef).exp_().mul_(a)
            sigma = w.sum(1)
            tau = sigma * (tb - ta)
            before = tau.cumsum(0) - tau
            before = before - before[(off[i] - b)]
            weight = torch.exp(-before) * -torch.expm1(-tau)
            col = (w @ rgb) * (weight / sigma.clamp_min(1e-300))[:, None]
            rgba[:, :3].index_add_(0, i, col)
            rgba[:, 3].index_add_(0, i, weight)
        r0 = r1
    return rgba


def exact(case, seed):
    s = _inputs(case, seed)
    kind, scene = case["kind"], case["scene"]
    if kind == "batch":
        parts = []
        for k, o, d in s["jobs"]:
            f, dense, boxes = s["scenes"][k]
            got = _samples(o, d, dense, boxes, f, _room(case, f, o.shape[0]))
            got[0] = torch.nn.functional.pad(got[0], (0, (o.shape[0] + 2) // 2 * 2 - got[0].numel()))
            parts.append(got)
        return [torch.cat(p) for p in zip(*parts)]
    if kind == "train":
        out = []
        for dense, (o, d) in zip((s["dense2"], s["dense"]), s["rays"]):
            got = _samples(o, d, dense, s["boxes"], scene, _room(case, scene, o.shape[0]))
            out.append(got + [int(got[0][-1])])
        return out
    o, d = s["rays"][0]
    if kind in ("composite", "render"):
        return [_composite64(o, d, _samples(o, d, s["dense"], s["boxes"], scene), s["field"])]
    smp = _samples(o, d, s["dense"], s["boxes"], scene, _room(case, scene, o.shape[0]))
    return smp if kind == "sample" else smp + [_composite64(o, d, smp, s["field"])]
