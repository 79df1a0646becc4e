"""The work this framework is measured on, through its public entry points.

Each case is one call sequence of a user's program: open a handle, load a
problem, iterate or solve, read the poses; a batch of uneven jobs; the planes,
gradient and cost at given poses; raw scans to voxels; points to clusters.
Sizes are those of the repository's workloads (scenegen: tiny, mid, city;
bench.py: batched jobs of 20-2000 scans, the preprocessing of 1,000 scans) and
of its tests, from the smallest to the largest, odd sizes among them.

The scenes are drawn on the GPU from the seed alone: planar patches seen by
random scans (all of them, or those near the patch), points uniform on the
patch with Gaussian noise along its normal, initial poses off by a fraction of
a degree and centimetres.
"""
import math

import torch

import paper_2608_14266_gb300 as mm

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # a small local map solved to convergence in plain FP64 from host
        # arrays: a robot's sliding window, where call latency is everything
        dict(name="solve_tiny_host", kind="solve", precision="fp64", scans=20, voxels=200, obs_min=5, obs_max=20,
             pts=50, box=50.0, height=50.0, side_min=1.0, side_max=1.0, strips=0.0, radius=0.0, rot_deg=1.0,
             trans=0.05, noise=0.01, iters=0, where="host", form="centred", gauss_newton=False),
        # one served job: a few hundred scans, clusters already on the device
        dict(name="solve_job_mixed", kind="solve", precision="mixed", scans=500, voxels=25003, obs_min=5, obs_max=30,
             pts=32, box=50.0, height=50.0, side_min=1.0, side_max=1.0, strips=0.0, radius=0.0, rot_deg=0.5,
             trans=0.10, noise=0.02, iters=20, where="device", form="centred", gauss_newton=False),
        # a drive's worth of scans in the reference precision, with the
        # Gauss-Newton Hessian and clusters given as raw sums
        dict(name="solve_mid_fp64", kind="solve", precision="fp64", scans=1000, voxels=50000, obs_min=8, obs_max=40,
             pts=100, box=50.0, height=50.0, side_min=1.0, side_max=1.0, strips=0.0, radius=0.0, rot_deg=0.5,
             trans=0.10, noise=0.02, iters=10, where="device", form="raw", gauss_newton=True),
        # the headline problem: a city, 10,000 scans and 15M clusters
        dict(name="solve_city_mixed", kind="solve", precision="mixed", scans=10000, voxels=500000, obs_min=10,
             obs_max=50, pts=32, box=2000.0, height=50.0, side_min=0.5, side_max=4.0, strips=0.05, radius=200.0,
             rot_deg=0.5, trans=0.10, noise=0.02, iters=30, where="device", form="centred", gauss_newton=False),
        # the same end to end from pinned host memory, a quarter of the city
        dict(name="solve_district_host", kind="solve", precision="mixed", scans=2500, voxels=125001, obs_min=10,
             obs_max=50, pts=32, box=1000.0, height=50.0, side_min=0.5, side_max=4.0, strips=0.05, radius=200.0,
             rot_deg=0.5, trans=0.10, noise=0.02, iters=30, where="pinned", form="centred", gauss_newton=False),
        # many uneven maps at once (a mapping service's queue), loaded and
        # stepped together
        dict(name="batch_jobs_mixed", kind="batch", precision="mixed", jobs=24, scans_min=20, scans_max=2000,
             obs_min=5, obs_max=30, pts=32, iters=20),
        # planes, gradient, Hessian and cost at poses from elsewhere: a resume,
        # or the evaluation of another optimiser's step
        dict(name="evaluate_fp64", kind="evaluate", precision="fp64", scans=1200, voxels=60001, obs_min=8,
             obs_max=40, pts=32, box=120.0, height=30.0, side_min=0.5, side_max=2.0, strips=0.05, radius=0.0,
             rot_deg=0.3, trans=0.05, noise=0.02, form="centred", gauss_newton=False),
        # the cost alone, from the caller's own buffers: the call an on-vehicle
        # loop makes between steps
        dict(name="cost_noalloc", kind="cost", scans=777, voxels=40003, obs_min=2, obs_max=40, pts=32, box=120.0,
             height=30.0, side_min=0.5, side_max=2.0, strips=0.05, radius=0.0, rot_deg=0.3, trans=0.05, noise=0.02),
        # preprocessing of a handful of scans as they come off the sensor (a
        # plane is asked of voxels that at least three scans have seen)
        dict(name="voxelize_few_scans", kind="voxelize", scans=8, pts_per_scan=8192, ragged=True, box=40.0,
             breadth=40.0, height=20.0, road=False, patches=200, voxel=0.5, levels=2, tau=0.1, min_obs=3, run=64,
             where="device", room=20000),
        # preprocessing of a whole drive: 1,000 scans, 120M points, three levels
        dict(name="voxelize_drive", kind="voxelize", scans=1000, pts_per_scan=120000, ragged=False, box=50.0,
             breadth=50.0, height=50.0, road=False, patches=50000, voxel=0.5, levels=3, tau=0.1, min_obs=3, run=100,
             where="device", room=2000000),
        # raw scans streamed from pinned host memory, 20 km of a winding road
        # (keys of more than 32 bits), every voxel kept
        dict(name="voxelize_host_road", kind="voxelize", scans=60, pts_per_scan=131071, ragged=True, box=20000.0,
             breadth=2000.0, height=50.0, road=True, patches=60000, voxel=0.5, levels=1, tau=0.0, min_obs=1, run=100,
             where="pinned", room=2000000),
        # point clusters per observation, a served job's points just generated
        dict(name="clusters_ragged", kind="clusters", obs=600001, pts_min=1, pts_max=64, reach=80.0, side=1.0,
             noise=0.02),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "evaluate", "cost", "voxelize", "voxelize", "clusters"])
    scene = dict(pts=rng.randint(20, 100), strips=rng.choice([0.0, 0.05]), rot_deg=rng.uniform(0.2, 1.0),
                 trans=rng.uniform(0.03, 0.10), noise=rng.uniform(0.01, 0.02))
    small = dict(box=rng.uniform(40.0, 150.0), height=rng.uniform(20.0, 50.0), side_min=rng.uniform(0.5, 1.0),
                 side_max=rng.uniform(1.0, 2.0), radius=0.0)
    if kind == "solve":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        if precision == "mixed" and rng.random() < 0.4:  # a town: scans see what is near them
            scans = _log(rng, 1500, 9000)
            area = dict(box=20.0 * math.sqrt(scans), height=rng.uniform(20.0, 50.0), side_min=0.5, side_max=4.0,
                        radius=200.0)
            obs_min, obs_max = 10, 50
        else:
            scans, area = _log(rng, 20, 1500 if precision == "mixed" else 1000), small
            obs_min = rng.randint(4, 8)
            obs_max = min(scans, rng.randint(16, 40))
        return dict(kind="solve", precision=precision, scans=scans, voxels=_log(rng, 20, 50) * scans + rng.randint(0, 31),
                    obs_min=obs_min, obs_max=obs_max, iters=rng.choice([10, 20]),
                    where=rng.choice(["device", "device", "pinned"]), form=rng.choice(["centred", "raw"]),
                    gauss_newton=rng.random() < 0.25, **scene, **area)
    if kind == "batch":
        lo = _log(rng, 20, 100)
        return dict(kind="batch", precision="mixed", jobs=rng.randint(2, 40), scans_min=lo,
                    scans_max=_log(rng, 2 * lo, 1500), obs_min=rng.randint(4, 8), obs_max=rng.randint(16, 20),
                    pts=rng.randint(20, 64), iters=rng.choice([10, 20]))
    if kind == "evaluate":
        scans = _log(rng, 30, 1500)
        return dict(kind="evaluate", precision="fp64", scans=scans, voxels=_log(rng, 10, 50) * scans + rng.randint(0, 31),
                    obs_min=rng.randint(2, 8), obs_max=rng.randint(16, 29), form=rng.choice(["centred", "raw"]),
                    gauss_newton=rng.random() < 0.5, **scene, **small)
    if kind == "cost":
        scans = _log(rng, 30, 1500)
        return dict(kind="cost", scans=scans, voxels=_log(rng, 10, 60) * scans + rng.randint(0, 31),
                    obs_min=rng.randint(1, 8), obs_max=rng.randint(16, 29), **scene, **small)
    if kind == "voxelize":
        scans = _log(rng, 3, 300)
        per = _log(rng, 2000, 120000)
        road, run = rng.random() < 0.3, rng.randint(32, 128)
        # planarity is asked of voxels that three scans and more have seen (two
        # points are a plane in every direction)
        tau = 0.0 if road or scans < 12 else rng.choice([0.0, 0.1, 0.1])
        box = rng.uniform(2000.0, 20000.0) if road else rng.uniform(30.0, 80.0)
        return dict(kind="voxelize", scans=scans, pts_per_scan=per, ragged=rng.random() < 0.7,
                    box=box, breadth=0.1 * box if road else box, height=rng.uniform(15.0, 50.0), road=road,
                    patches=max(32, int(scans * per / run / rng.uniform(8.0, 30.0))),
                    voxel=rng.choice([0.3, 0.5, 0.5, 1.0]), levels=rng.randint(1, 3), tau=tau,
                    min_obs=3 if tau else rng.randint(1, 2), run=run, where=rng.choice(["device", "device", "pinned"]),
                    room=2 * scans * per)
    lo = rng.randint(1, 24)
    return dict(kind="clusters", obs=_log(rng, 2000, 900000), pts_min=lo, pts_max=lo + rng.randint(8, 64),
                reach=rng.uniform(20.0, 150.0), side=rng.uniform(0.5, 2.0), noise=rng.uniform(0.01, 0.03))


# ---- scenes ------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _uniform(g, *shape, dtype=F64):
    return torch.rand(shape, generator=g, device=DEV, dtype=dtype)


def _normal(g, *shape, dtype=F64):
    return torch.randn(shape, generator=g, device=DEV, dtype=dtype)


def _mul(a, b):
    """Products of 3x3 matrices, batch by batch."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _vec(a, x):
    return (a * x.unsqueeze(-2)).sum(-1)


def _rotations(g, n):
    """Uniformly distributed rotations, from normal quaternions."""
    q = _normal(g, n, 4)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(n, 3, 3)


def _cross_matrix(v):
    x, y, z = v.unbind(-1)
    o = torch.zeros_like(x)
    return torch.stack([o, -z, y, z, o, -x, -y, x, o], -1).view(*v.shape[:-1], 3, 3)


def _exp(phi):
    """Rotations of the rotation vectors phi (Rodrigues)."""
    t2 = (phi * phi).sum(-1)
    t = t2.sqrt()
    a = torch.where(t > 1e-6, torch.sin(t) / t.clamp_min(1e-300), torch.ones_like(t))
    b = torch.where(t > 1e-6, 2 * torch.sin(t / 2) ** 2 / t2.clamp_min(1e-300), torch.full_like(t, 0.5))
    k = _cross_matrix(phi)
    return torch.eye(3, dtype=F64, device=DEV) + a[..., None, None] * k + b[..., None, None] * _mul(k, k)


def _poses(g, n, box, breadth, height, rot_deg, trans):
    """Ground truth (R, t) and the perturbed initial poses, n x 12; scan 0 unperturbed."""
    r = _rotations(g, n)
    t = _uniform(g, n, 3) * torch.tensor([box, breadth, height], dtype=F64, device=DEV)
    phi, dt = _normal(g, n, 3) * math.radians(rot_deg), _normal(g, n, 3) * trans
    phi[0], dt[0] = 0.0, 0.0
    return r, t, torch.cat([_mul(_exp(phi), r).reshape(n, 9), t + dt], 1).contiguous()


def _observers(g, c, centre, t):
    """Observing scans of every voxel: (voxel_off, obs_scan), a voxel's scans ascending and distinct."""
    nv, ns = centre.shape[0], t.shape[0]
    lo, hi = c["obs_min"], min(c["obs_max"], ns)
    count = torch.randint(min(lo, hi), hi + 1, (nv,), generator=g, device=DEV)
    if c["radius"] > 0.0:  # the scans within the radius of the voxel's 50 m cell
        side = max(1, int(math.ceil(c["box"] / 50.0)))
        at = (torch.arange(side * side, device=DEV).unsqueeze(1).expand(-1, 2).clone())
        mid = torch.stack([(at[:, 0] % side) * 50.0 + 25.0, (at[:, 1] // side) * 50.0 + 25.0], 1).to(F64)
        near = torch.cdist(mid, t[:, :2]) <= c["radius"]
        n_near = near.sum(1)
        width = int(n_near.max())
        cand = torch.sort(near.to(torch.int8), dim=1, descending=True, stable=True)[1][:, :width].to(torch.int32)
        cell = ((centre[:, 0] / 50.0).long().clamp(0, side - 1) + (centre[:, 1] / 50.0).long().clamp(0, side - 1) * side)
        cand[n_near == 0] = 0
        n_near = n_near.clamp_min(1)
    else:
        cand, width = torch.arange(ns, device=DEV, dtype=torch.int32).unsqueeze(0), ns
        n_near = torch.tensor([ns], device=DEV)
        cell = torch.zeros(nv, dtype=torch.long, device=DEV)
    count = torch.minimum(count, n_near[cell])
    lists, top = [], min(hi, width)
    step = max(1, (1 << 26) // width)
    slot = torch.arange(width, device=DEV)
    for a in range(0, nv, step):
        b = min(nv, a + step)
        key = _uniform(g, b - a, width, dtype=torch.float32)
        key.masked_fill_(slot >= n_near[cell[a:b]].unsqueeze(1), -1.0)
        pick = torch.topk(key, top, dim=1)[1]
        scan = torch.gather(cand[cell[a:b]], 1, pick)
        scan.masked_fill_(slot[:top] >= count[a:b].unsqueeze(1), 1 << 30)
        scan = torch.sort(scan, 1)[0]
        lists.append(scan[scan < 1 << 30])
    off = torch.zeros(nv + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(count, 0)
    return off, torch.cat(lists).to(torch.int32)


def _scene(c, seed):
    """Voxel-major observations of a planar scene: voxel_off, obs_scan, centred clusters, initial poses."""
    g = _gen(seed)
    ns, nv = c["scans"], c["voxels"]
    r, t, init = _poses(g, ns, c["box"], c["box"], c["height"], c["rot_deg"], c["trans"])
    centre = _uniform(g, nv, 3) * torch.tensor([c["box"], c["box"], c["height"]], dtype=F64, device=DEV)
    frame = _rotations(g, nv)
    side = c["side_min"] * (c["side_max"] / c["side_min"]) ** _uniform(g, nv)
    ratio = 2.0 + 8.0 * _uniform(g, nv)
    width = torch.where(_uniform(g, nv) < c["strips"], c["noise"] * torch.sqrt(12.0 * ratio), side)
    off, scan = _observers(g, c, centre, t)
    vox = torch.repeat_interleave(torch.arange(nv, device=DEV), off[1:] - off[:-1])
    agg = torch.empty(scan.shape[0], 10, dtype=F64, device=DEV)
    n = c["pts"]
    step = max(1, (1 << 26) // n)
    for a in range(0, scan.shape[0], step):
        v, j = vox[a:a + step], scan[a:a + step].long()
        m = v.shape[0]
        p = _uniform(g, m, n, 3, dtype=torch.float32) - 0.5
        p[..., 2] = _normal(g, m, n, dtype=torch.float32)
        scale = torch.stack([side[v], width[v], torch.full_like(side[v], c["noise"])], 1)
        p = p.to(F64) * scale.unsqueeze(1)  # patch coordinates
        mean = p.mean(1)
        p -= mean.unsqueeze(1)
        x, y, z = p.unbind(2)
        s = torch.stack([(x * x).sum(1), (x * y).sum(1), (x * z).sum(1), (x * y).sum(1), (y * y).sum(1),
                         (y * z).sum(1), (x * z).sum(1), (y * z).sum(1), (z * z).sum(1)], 1).view(m, 3, 3)
        rt = r[j].transpose(1, 2)
        to_scan = _mul(rt, frame[v])
        s = _mul(_mul(to_scan, s), to_scan.transpose(1, 2))
        out = agg[a:a + step]
        out[:, 0], out[:, 1], out[:, 2] = s[:, 0, 0], s[:, 0, 1], s[:, 0, 2]
        out[:, 3], out[:, 4], out[:, 5] = s[:, 1, 1], s[:, 1, 2], s[:, 2, 2]
        out[:, 6:9] = _vec(to_scan, mean) + _vec(rt, centre[v] - t[j])
        out[:, 9] = float(n)
    return dict(off=off, scan=scan, agg=agg, poses=init)


def _raw_sums(agg):
    """Clusters as raw sums: P = S + N m m^T, v = N m, N."""
    m, n = agg[:, 6:9], agg[:, 9:]
    out = agg.clone()
    k = 0
    for a in range(3):
        for b in range(a, 3):
            out[:, k] += n[:, 0] * m[:, a] * m[:, b]
            k += 1
    out[:, 6:9] = n * m
    return out


def _scan_points(c, seed):
    """Raw scans: runs of `run` consecutive points on one patch each, in scan coordinates at the ground truth."""
    g = _gen(seed)
    ns, run = c["scans"], c["run"]
    per = torch.full((ns,), c["pts_per_scan"], dtype=torch.int64, device=DEV)
    if c["ragged"]:  # scans of uneven length, the same total for every seed
        k = torch.arange(ns, device=DEV)
        per = (c["pts_per_scan"] * (0.4 + 1.2 * ((k * 37) % ns).to(F64) / max(1, ns - 1))).long()
    off = torch.zeros(ns + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(per, 0)
    n = int(off[-1])
    r, t, init = _poses(g, ns, c["box"], c["breadth"], c["height"], 0.5, 0.10)
    patches = c["patches"]
    centre = _uniform(g, patches, 3)
    centre[:, 0] = torch.sort(centre[:, 0])[0]
    centre *= torch.tensor([c["box"], c["breadth"], c["height"]], dtype=F64, device=DEV)
    if c["road"]:  # scans and patches within 50 m of a winding line along the box
        for x in (centre, t, init[:, 9:]):
            line = 0.5 * c["breadth"] * (1.0 + torch.sin(x[:, 0] * (6.0 * math.pi / c["box"])))
            x[:, 1] = line + 100.0 * (x[:, 1] / c["breadth"] - 0.5)
    frame = _rotations(g, patches)
    # each run's patch: one within 100 m along the box's long side
    runs = n // run + ns + 1
    who = torch.searchsorted(off // run + torch.arange(ns + 1, device=DEV),
                             torch.arange(runs, device=DEV), right=True).sub_(1).clamp_(0, ns - 1)
    reach = patches * min(1.0, 100.0 / c["box"])
    pick = t[who, 0] / c["box"] * patches + (2.0 * _uniform(g, runs) - 1.0) * reach
    pick = pick.long().abs_()  # reflected at both ends
    pick = torch.where(pick >= patches, 2 * patches - 1 - pick, pick).clamp_(0, patches - 1)
    scan = torch.repeat_interleave(torch.arange(ns, device=DEV), per)
    pts = torch.empty(n, 3, dtype=F64, device=DEV)
    step = 1 << 24
    for a in range(0, n, step):
        j = scan[a:a + step]
        i = torch.arange(a, a + j.shape[0], device=DEV)
        v = pick[(i - off[j]) // run + off[j] // run + j]
        p = _uniform(g, j.shape[0], 3, dtype=torch.float32) - 0.5
        p[:, 2] = 0.02 * _normal(g, j.shape[0], dtype=torch.float32)
        w = _vec(frame[v], p.to(F64)) + centre[v]
        pts[a:a + step] = _vec(r[j].transpose(1, 2), w - t[j])
    return dict(off=off, pts=pts, poses=init)


def _job_scans(c):
    """Scan counts of a batch's jobs, evenly spread over the logarithm of their range."""
    k = max(1, c["jobs"] - 1)
    return [int(round(c["scans_min"] * (c["scans_max"] / c["scans_min"]) ** (i / k))) for i in range(c["jobs"])]


def _job_case(c, scans):
    return dict(scans=scans, voxels=50 * scans, obs_min=min(c["obs_min"], scans), obs_max=c["obs_max"], pts=c["pts"],
                box=50.0, height=50.0, side_min=1.0, side_max=1.0, strips=0.0, radius=0.0, rot_deg=0.5, trans=0.10,
                noise=0.02)


def _place(x, where):
    if where == "device":
        return x
    x = x.cpu()
    return x.pin_memory().numpy() if where == "pinned" else x.numpy()


def _precision(c):
    return mm.BA_MIXED if c["precision"] == "mixed" else mm.BA_FP64


def _cluster_points(c, seed):
    g = _gen(seed)
    counts = torch.randint(c["pts_min"], c["pts_max"] + 1, (c["obs"],), generator=g, device=DEV)
    off = torch.zeros(c["obs"] + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(counts, 0)
    centre = (_uniform(g, c["obs"], 3) - 0.5) * 2.0 * c["reach"]
    frame = _rotations(g, c["obs"])
    of = torch.repeat_interleave(torch.arange(c["obs"], device=DEV), counts)
    p = (_uniform(g, int(off[-1]), 3) - 0.5) * c["side"]
    p[:, 2] = c["noise"] * _normal(g, int(off[-1]))
    return off, _vec(frame[of], p) + centre[of]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        s = _scene(case, seed)
        if case["form"] == "raw":
            s["agg"] = _raw_sums(s["agg"])
        s = {k: _place(v, case["where"]) for k, v in s.items()}
        return dict(case=case, **s)
    if kind == "batch":
        return dict(case=case, jobs=[_scene(_job_case(case, n), 1000 * seed + i)
                                     for i, n in enumerate(_job_scans(case))])
    if kind == "evaluate":
        s = _scene(case, seed)
        if case["form"] == "raw":
            s["agg"] = _raw_sums(s["agg"])
        ba = mm.BundleAdjuster(precision=_precision(case), hessian_mode=int(case["gauss_newton"]))
        ba.load_observations(case["scans"], s["off"], s["scan"], s["agg"], s["poses"], _form(case))
        return dict(case=case, ba=ba, poses=_moved(s["poses"], seed))
    if kind == "cost":
        s = _scene(case, seed)
        return dict(case=case, **s, cost=torch.zeros(1, dtype=F64, device=DEV),
                    lam=torch.zeros(case["voxels"], dtype=F64, device=DEV))
    if kind == "voxelize":
        s = _scan_points(case, seed)
        return dict(case=case, out=_buffers(case["room"]), **{k: _place(v, case["where"]) for k, v in s.items()})
    off, pts = _cluster_points(case, seed)
    return dict(case=case, off=off, pts=pts, out=torch.empty(case["obs"], 10, dtype=F64, device=DEV))


def _buffers(room):
    """Observation lists of fixed room, as a program that maps scan after scan keeps them."""
    zeros = lambda *shape, dtype=torch.int32: torch.zeros(shape, dtype=dtype, device=DEV)  # noqa: E731
    return dict(voxel_off=zeros(room + 1, dtype=torch.int64), obs_scan=zeros(room), agg=zeros(room, 10, dtype=F64),
                level=zeros(room), index=zeros(room, 3))


def _into(buffers, lists):
    """The lists at the front of their buffers, with their lengths."""
    for k, x in buffers.items():
        x[:lists[k].shape[0]].copy_(lists[k])
    return dict(buffers, voxels=lists["level"].shape[0], observations=lists["obs_scan"].shape[0])


def _form(c):
    return mm.BA_AGG_RAW_SUMS if c["form"] == "raw" else mm.BA_AGG_CENTRED


def _moved(poses, seed):
    """Poses a small step away, as a resume or another optimiser hands over."""
    g = _gen(seed + 50000)
    n = poses.shape[0]
    r = _mul(_exp(_normal(g, n, 3) * 2e-3), poses[:, :9].view(n, 3, 3))
    return torch.cat([r.reshape(n, 9), poses[:, 9:] + 0.01 * _normal(g, n, 3)], 1).contiguous()


# ---- the calls -----------------------------------------------------------------

def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "solve":
        with mm.BundleAdjuster(precision=_precision(c), hessian_mode=int(c["gauss_newton"])) as ba:
            ba.load_observations(c["scans"], state["off"], state["scan"], state["agg"], state["poses"], _form(c))
            st = ba.iterate(c["iters"]) if c["iters"] else ba.solve()
            out = torch.empty(c["scans"], 12, dtype=F64, device=DEV) if c["where"] == "device" else None
            return {"poses": ba.poses(out), "cost": st["cost"], "accepted": st["accepted"]}
    if kind == "batch":
        bas = []
        with mm.Batch() as b:
            for s in state["jobs"]:
                ba = mm.BundleAdjuster(precision=_precision(c))
                bas.append(ba)
                ba.load_observations(s["poses"].shape[0], s["off"], s["scan"], s["agg"], s["poses"])
                b.add(ba)
            b.iterate(c["iters"])
            poses = [ba.poses(torch.empty_like(s["poses"])) for ba, s in zip(bas, state["jobs"])]
        for ba in bas:
            ba.close()
        return poses
    if kind == "evaluate":
        ba = state["ba"]
        ba.set_state(state["poses"])
        g, h = ba.gradient()
        p = ba.planes()
        return {"cost": ba.cost(), "g": g, "H": h, "lambda": p[:, :3], "normal": p[:, 3:6], "centroid": p[:, 6:]}
    if kind == "cost":
        mm.ba_eval_cost_noalloc(c["scans"], state["off"], state["scan"], state["agg"], state["poses"], state["cost"],
                                state["lam"])
        return {"cost": state["cost"], "lambda": state["lam"]}
    if kind == "voxelize":
        v = mm.voxelize(state["off"], state["pts"], state["poses"], c["voxel"], levels=c["levels"], tau=c["tau"],
                        min_obs=c["min_obs"], out="device")
        return _into(state["out"], v)
    return mm.ba_aggregate_points(state["off"], state["pts"], state["out"])


# ---- what a pass cannot do without -----------------------------------------------

def _scene_obs(c):
    return c["voxels"] * 0.5 * (min(c["obs_min"], c["scans"]) + min(c["obs_max"], c["scans"]))


def _solve_work(c, iters):
    """The inputs read once, and per iteration the observations once for the
    trial cost and once for the derivatives (84 bytes each in FP64, 44 in the
    mixed path), with the poses and planes they meet."""
    no = _scene_obs(c)
    per_obs, word = (84, 8) if c["precision"] == "fp64" else (44, 4)
    load = no * 84 + c["voxels"] * 8 + c["scans"] * 96
    step = no * 2 * per_obs + c["voxels"] * 2 * 4 * word + c["scans"] * (2 * 96 + 2 * 27 * 8)
    return {"bytes": load + iters * step + c["scans"] * 96, "flops": (iters + 1) * no * 330}


def work(case):
    kind = case["kind"]
    if kind == "solve":
        return _solve_work(case, case["iters"] or 20)
    if kind == "batch":
        parts = [_solve_work(dict(_job_case(case, n), precision=case["precision"]), case["iters"])
                 for n in _job_scans(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "evaluate":
        no = _scene_obs(case)
        return {"bytes": no * 2 * 84 + case["voxels"] * 72 + case["scans"] * (96 + 42 * 8), "flops": no * 330}
    if kind == "cost":
        no = _scene_obs(case)
        return {"bytes": no * 84 + case["voxels"] * 16 + case["scans"] * 96, "flops": no * 103}
    if kind == "voxelize":
        n = case["scans"] * case["pts_per_scan"]
        return {"bytes": n * 24 + n / 30 * 84, "flops": n * 39}
    n = case["obs"] * 0.5 * (case["pts_min"] + case["pts_max"])
    return {"bytes": n * 24 + case["obs"] * 88, "flops": n * 18}


# ---- the same in plain 64-bit torch --------------------------------------------------

def _segsum(x, of, n):
    return torch.zeros((n,) + x.shape[1:], dtype=F64, device=DEV).index_add_(0, of, x)


def _full(s):
    return torch.stack([s[:, 0], s[:, 1], s[:, 2], s[:, 1], s[:, 3], s[:, 4], s[:, 2], s[:, 4], s[:, 5]],
                       1).view(-1, 3, 3)


def _eigen(a):
    """Eigenvalues (ascending) and eigenvectors (columns) of symmetric 3x3 matrices, by cyclic Jacobi."""
    a = a.clone()
    v = torch.eye(3, dtype=F64, device=DEV).expand_as(a).clone()
    for _ in range(8):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            off, d = a[:, p, q], a[:, q, q] - a[:, p, p]
            # tangent of the rotation angle: 2 off / (d + sign(d) sqrt(d^2 + 4 off^2))
            den = d + torch.where(d < 0, -1.0, 1.0) * torch.sqrt(d * d + 4 * off * off)
            t = torch.where(den != 0, 2 * off / torch.where(den != 0, den, torch.ones_like(den)),
                            torch.zeros_like(den))
            cs = 1 / torch.sqrt(1 + t * t)
            sn = t * cs
            for m, left in ((a, True), (a, False), (v, False)):
                x, y = (m[:, p].clone(), m[:, q].clone()) if left else (m[:, :, p].clone(), m[:, :, q].clone())
                nx, ny = cs[:, None] * x - sn[:, None] * y, sn[:, None] * x + cs[:, None] * y
                if left:
                    m[:, p], m[:, q] = nx, ny
                else:
                    m[:, :, p], m[:, :, q] = nx, ny
    lam, order = torch.sort(torch.diagonal(a, dim1=1, dim2=2), 1)
    return lam, torch.gather(v, 2, order.unsqueeze(1).expand(-1, 3, -1))


class _Exact:
    """The cost, planes, gradient and Hessian of a problem, and Levenberg-Marquardt iterations on it."""

    def __init__(self, s, raw=False, gauss_newton=False):
        as_dev = lambda x: torch.as_tensor(x).to(DEV)  # noqa: E731
        off, self.scan, agg, self.poses = (as_dev(s[k]) for k in ("off", "scan", "agg", "poses"))
        self.scan = self.scan.long()
        self.nv, self.ns = off.shape[0] - 1, self.poses.shape[0]
        self.vox = torch.repeat_interleave(torch.arange(self.nv, device=DEV), off[1:] - off[:-1])
        self.n = agg[:, 9]
        self.m = agg[:, 6:9] / self.n[:, None] if raw else agg[:, 6:9]
        self.s = _full(agg[:, :6])
        if raw:
            self.s = self.s - self.n[:, None, None] * self.m[:, :, None] * self.m[:, None, :]
        self.nvox = _segsum(self.n, self.vox, self.nv)
        self.gn = gauss_newton

    def planes(self, poses):
        r, t = poses[:, :9].view(-1, 3, 3)[self.scan], poses[self.scan, 9:]
        lever = _vec(r, self.m)
        q = lever + t
        a0 = torch.empty(self.nv, 3, dtype=F64, device=DEV)
        a0[self.vox] = q  # any one posed mean of the voxel
        d = q - a0[self.vox]
        mean = _segsum(self.n[:, None] * d, self.vox, self.nv) / self.nvox[:, None]
        d -= mean[self.vox]
        w = _mul(_mul(r, self.s), r.transpose(1, 2))
        cov = _segsum(w + self.n[:, None, None] * d[:, :, None] * d[:, None, :], self.vox, self.nv)
        lam, vec = _eigen(cov / self.nvox[:, None, None])
        return dict(lam=lam, u=vec[:, :, 0], c=a0 + mean, cost=float(lam[:, 0].sum()), w=w, lever=lever, d=d)

    def derivatives(self, e):
        u, k = e["u"][self.vox], (2.0 / self.nvox)[self.vox]
        n, lever = self.n, e["lever"]
        r = (u * e["d"]).sum(1)
        nr = n * r
        mv = _vec(e["w"], u) + nr[:, None] * lever
        g = torch.cat([torch.cross(mv, u, dim=1), nr[:, None] * u], 1) * k[:, None]
        ku = _cross_matrix(u)
        p = e["w"] + n[:, None, None] * lever[:, :, None] * lever[:, None, :]
        h = torch.empty(u.shape[0], 6, 6, dtype=F64, device=DEV)
        h[:, :3, :3] = _mul(_mul(ku, p), ku.transpose(1, 2))
        if not self.gn:
            um = u[:, :, None] * mv[:, None, :]
            h[:, :3, :3] += 0.5 * (um + um.transpose(1, 2))
            h[:, :3, :3] -= (u * mv).sum(1)[:, None, None] * torch.eye(3, dtype=F64, device=DEV)
        lu = n[:, None] * torch.cross(lever, u, dim=1)
        h[:, :3, 3:] = lu[:, :, None] * u[:, None, :]
        h[:, 3:, :3] = u[:, :, None] * lu[:, None, :]
        h[:, 3:, 3:] = n[:, None, None] * u[:, :, None] * u[:, None, :]
        h *= k[:, None, None]
        return _segsum(g, self.scan, self.ns), _segsum(h, self.scan, self.ns)

    def iterate(self, iters):
        """iters steps, or, with 0, until an accepted step gains no more than 1e-8 of the cost."""
        x, mu, nu, accepted, done = self.poses.clone(), 1e-4, 2.0, 0, 0
        e = self.planes(x)
        g, h = self.derivatives(e)
        seen = torch.zeros(self.ns, dtype=torch.bool, device=DEV)
        seen[self.scan] = True
        seen[0] = False  # the fixed scan
        eye = torch.eye(6, dtype=F64, device=DEV)
        rejected = 0
        while done < (iters or 200):
            a = torch.where(seen[:, None, None], h + mu * h * eye, eye)
            delta = torch.linalg.solve(a, -g) * seen[:, None]
            positive = bool((torch.linalg.cholesky_ex(a)[1] == 0).all())
            pred = -float((g * delta).sum() + 0.5 * (delta[:, None, :] @ h @ delta[:, :, None]).sum())
            y = torch.cat([_mul(_exp(delta[:, :3]), x[:, :9].view(-1, 3, 3)).reshape(-1, 9),
                           x[:, 9:] + delta[:, 3:]], 1)
            t = self.planes(y)
            done += 1
            if positive and pred > 0 and t["cost"] < e["cost"]:
                gain = e["cost"] - t["cost"]
                mu *= max(1.0 / 3.0, 1.0 - (2.0 * gain / pred - 1.0) ** 3)
                nu, accepted, rejected = 2.0, accepted + 1, 0
                stop = gain <= 1e-8 * e["cost"]
                x, e = y, t
                if not iters and stop:
                    break
                g, h = self.derivatives(e)
            else:
                mu, nu, rejected = mu * nu, nu * 2.0, rejected + 1
                if not iters and rejected >= 10:
                    break
        return x, e["cost"], accepted


def _voxelize_exact(c, s):
    off, pts, poses = (torch.as_tensor(s[k]).to(DEV) for k in ("off", "pts", "poses"))
    ns, n = c["scans"], pts.shape[0]
    scan = torch.repeat_interleave(torch.arange(ns, device=DEV), off[1:] - off[:-1])
    r, t = poses[:, :9].view(-1, 3, 3), poses[:, 9:]
    index = torch.empty(n, 3, dtype=torch.int64, device=DEV)
    for a in range(0, n, 1 << 24):
        j = scan[a:a + (1 << 24)]
        index[a:a + (1 << 24)] = torch.floor((_vec(r[j], pts[a:a + (1 << 24)]) + t[j]) / c["voxel"]).long()
    base = index.min(0)[0]

    def clusters(idx, sc, mean, scatter, count):
        """Merges items of the same (voxel, scan); voxels in index order, scans ascending inside."""
        span = idx.max(0)[0] - base_k + 1
        key = (((idx[:, 0] - base_k[0]) * span[1] + idx[:, 1] - base_k[1]) * span[2] + idx[:, 2] - base_k[2]) * ns + sc
        uniq, of = torch.unique(key, return_inverse=True)
        del key
        k = uniq.shape[0]
        cnt = _segsum(count, of, k)
        first = torch.empty(k, 3, dtype=F64, device=DEV)
        first[of] = mean
        mu = first + _segsum(count[:, None] * (mean - first[of]), of, k) / cnt[:, None]
        sc6 = torch.empty(k, 6, dtype=F64, device=DEV)
        i = 0
        d = mean - mu[of]
        for a in range(3):
            for b in range(a, 3):
                x = count * d[:, a] * d[:, b]
                sc6[:, i] = _segsum(x if scatter is None else x + scatter[:, i], of, k)
                i += 1
        vkey = uniq // ns
        out = torch.stack([vkey // (span[1] * span[2]) + base_k[0], vkey // span[2] % span[1] + base_k[1],
                           vkey % span[2] + base_k[2]], 1)
        return out, uniq % ns, mu, sc6, cnt, vkey

    parts = {k: [] for k in ("len", "scan", "agg", "level", "index")}
    base_k, items = base, (index, scan, pts, None, torch.ones(n, dtype=F64, device=DEV))
    for level in range(1, c["levels"] + 1):
        if level > 1:
            base_k = torch.div(base_k, 2, rounding_mode="floor")
            items = (torch.div(items[0], 2, rounding_mode="floor"),) + items[1:5]
        items = clusters(*items[:5])
        idx, sc, mu, s6, cnt, vkey = items
        voxels, of, per = torch.unique(vkey, return_inverse=True, return_counts=True)
        nv = voxels.shape[0]
        keep = per >= c["min_obs"]
        if c["tau"] > 0:
            w = _vec(r[sc], mu) + t[sc]
            tot = _segsum(cnt, of, nv)
            first = torch.empty(nv, 3, dtype=F64, device=DEV)
            first[of] = w
            d = w - first[of]
            d = d - (_segsum(cnt[:, None] * d, of, nv) / tot[:, None])[of]
            rot = _mul(_mul(r[sc], _full(s6)), r[sc].transpose(1, 2))
            lam = _eigen(_segsum(rot + cnt[:, None, None] * d[:, :, None] * d[:, None, :], of, nv))[0]
            keep &= lam[:, 0] < c["tau"] * lam[:, 1]
        rows = keep[of]
        parts["len"].append(per[keep])
        parts["scan"].append(sc[rows].to(torch.int32))
        parts["agg"].append(torch.cat([s6, mu, cnt[:, None]], 1)[rows])
        parts["level"].append(torch.full((int(keep.sum()),), level, dtype=torch.int32, device=DEV))
        first_row = torch.cumsum(per, 0) - per
        parts["index"].append(idx[first_row[keep]].to(torch.int32))
    length = torch.cat(parts["len"])
    voff = torch.zeros(length.shape[0] + 1, dtype=torch.int64, device=DEV)
    voff[1:] = torch.cumsum(length, 0)
    return dict(voxel_off=voff, obs_scan=torch.cat(parts["scan"]), agg=torch.cat(parts["agg"]),
                level=torch.cat(parts["level"]), index=torch.cat(parts["index"]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        s = prepare(case, seed)
        x, cost, accepted = _Exact(s, case["form"] == "raw", case["gauss_newton"]).iterate(case["iters"])
        return {"poses": x if case["where"] == "device" else x.cpu().numpy(), "cost": cost, "accepted": accepted}
    if kind == "batch":
        return [_Exact(s).iterate(case["iters"])[0] for s in prepare(case, seed)["jobs"]]
    if kind == "evaluate":
        s = _scene(case, seed)
        x = _Exact(s, False, case["gauss_newton"])  # the centred clusters: the raw sums round them
        e = x.planes(_moved(s["poses"], seed))
        g, h = x.derivatives(e)
        # a normal's sign is free
        return {"cost": e["cost"], "g": g.cpu().numpy(), "H": h.cpu().numpy(), "lambda": e["lam"].cpu().numpy(),
                "normal": None, "centroid": e["c"].cpu().numpy()}
    if kind == "cost":
        s = _scene(case, seed)
        e = _Exact(s).planes(s["poses"])
        return {"cost": e["lam"][:, 0].sum().reshape(1), "lambda": e["lam"][:, 0].contiguous()}
    if kind == "voxelize":
        return _into(_buffers(case["room"]), _voxelize_exact(case, _scan_points(case, seed)))
    off, pts = _cluster_points(case, seed)
    n = case["obs"]
    of = torch.repeat_interleave(torch.arange(n, device=DEV), off[1:] - off[:-1])
    count = (off[1:] - off[:-1]).to(F64)
    first = pts[off[:-1]]
    mean = first + _segsum(pts - first[of], of, n) / count[:, None]
    d = pts - mean[of]
    s6 = [_segsum(d[:, a] * d[:, b], of, n) for a in range(3) for b in range(a, 3)]
    return torch.cat([torch.stack(s6, 1), mean, count[:, None]], 1)
