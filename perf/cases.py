"""The workloads that the library's speed is measured on, through its public entry points.

Each case is one call (or the few calls that belong together) a program makes with its
inputs on the GPU: camera frames, batches of them, fused map clouds, a differentiable
decimation, an octree pyramid, a voxel map and the neighbour-count thinning loop.  Clouds
have the shapes of ``paper_2102_11084_gb300.synth`` (pinhole frames of planes and boxes;
40 x 40 x 10 m maps of planes, boxes and clutter, shuffled), generated on the device.

``listed()`` gives the cases, ``draw(rng)`` one more of the same ranges, ``prepare`` a
case's inputs and kept buffers, ``run`` one pass, ``work`` the bytes and operations a pass
cannot do without, ``exact`` its outputs in 64-bit arithmetic.
"""
import math

import numpy as np
import torch

from paper_2102_11084_gb300 import synth, vg

DEV = "cuda"
BAND = (0.05, 2.0)                # height band of posed frames, metres in the map frame
FIXED_ORIGIN = (-8.0, -8.0, 0.0)  # below every point of a camera frame
MAP_ORIGIN = (-10.0, -10.0, -5.0)  # below every point of a posed frame


def listed():
    return [
        # the smallest call: a crop of a frame on a fixed lattice, into kept buffers
        {"name": "crop_20k", "kind": "crop", "n": 20_011, "leaf": 0.05},
        # one VGA depth frame through the plain call, all defaults
        {"name": "frame_vga_default", "kind": "default", "width": 640, "height": 480,
         "leaf": 0.05},
        # one 720p depth frame through the single-frame method, into kept buffers
        {"name": "frame_hd_method", "kind": "frame", "width": 1280, "height": 720, "leaf": 0.02},
        # a cloud as a layer of a network: centroids, then the gradient of the points
        {"name": "autograd_hd", "kind": "autograd", "width": 1280, "height": 720, "leaf": 0.05},
        # four levels of detail of one 720p frame
        {"name": "pyramid_hd", "kind": "pyramid", "width": 1280, "height": 720, "leaf": 0.01,
         "levels": 4},
        # eight posed colour cameras of one robot: pose, height band, RGB means, two points
        # a voxel at least
        {"name": "posed_rgb_8", "kind": "posed_rgb", "frames": 8, "width": 640, "height": 480,
         "leaf": 0.02, "min_count": 2},
        # the paper's own thinning loop on one VGA frame, batches of 1000
        {"name": "thin_vga", "kind": "thin", "width": 640, "height": 480, "leaf": 0.05,
         "threshold": 20, "batch": 1000},
        # 64 frames of uneven size and leaf in one call of a kept plan (graph replay)
        {"name": "batch_64", "kind": "batch", "frames": 64, "n_min": 20_000, "n_max": 921_600},
        # 64 posed frames merged into an empty voxel map, then the map read out
        {"name": "voxel_map_64", "kind": "voxel_map", "frames": 64, "n_min": 20_000,
         "n_max": 921_600, "leaf": 0.05, "capacity": 4_000_000},
        # a site scan of 200 m at 1 cm: keys wider than 32 bits
        {"name": "scan_1m_wide", "kind": "scan", "n": 1_000_003, "leaf": 0.01, "extent": 200.0},
        # a map tile of odd size, unordered
        {"name": "map_2m5", "kind": "map", "n": 2_500_003, "leaf": 0.05},
        # the whole fused map, unordered
        {"name": "map_50m", "kind": "map", "n": 50_000_000, "leaf": 0.02},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice([c["kind"] for c in listed()])
    leaf = round(_log_uniform(rng, 0.01, 0.1), 4)
    w = int(_log_uniform(rng, 160, 1920))
    h = max(90, int(w * rng.choice([9 / 16, 3 / 4])))
    if kind == "crop":
        return {"kind": kind, "n": int(_log_uniform(rng, 1_000, 60_000)), "leaf": leaf}
    if kind in ("default", "frame", "autograd"):
        return {"kind": kind, "width": w, "height": min(h, 1080), "leaf": leaf}
    if kind == "pyramid":
        return {"kind": kind, "width": min(w, 1280), "height": min(h, 720), "leaf": leaf,
                "levels": rng.randint(2, 6)}
    if kind == "posed_rgb":
        return {"kind": kind, "frames": rng.randint(1, 16), "width": min(w, 640),
                "height": min(h, 480), "leaf": leaf, "min_count": rng.randint(1, 4)}
    if kind == "thin":
        return {"kind": kind, "width": min(w, 640), "height": min(h, 480),
                "leaf": round(rng.uniform(0.03, 0.06), 4), "threshold": rng.randint(10, 40),
                "batch": rng.randint(1000, 4000)}
    if kind == "batch":
        hi = int(_log_uniform(rng, 40_000, 921_600))
        return {"kind": kind, "frames": rng.randint(2, 64), "n_min": 20_000, "n_max": hi}
    if kind == "voxel_map":
        hi = int(_log_uniform(rng, 40_000, 921_600))
        return {"kind": kind, "frames": rng.randint(1, 64), "n_min": 20_000, "n_max": hi,
                "leaf": max(leaf, 0.03), "capacity": rng.choice([2_000_000, 4_000_000])}
    if kind == "scan":
        return {"kind": kind, "n": int(_log_uniform(rng, 100_000, 4_000_000)),
                "leaf": round(_log_uniform(rng, 0.005, 0.02), 4),
                "extent": round(rng.uniform(100.0, 300.0), 1)}
    n = int(_log_uniform(rng, 200_000, 50_000_000))
    return {"kind": kind, "n": n, "leaf": max(leaf, 0.02)}


# ---- inputs ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(0x9E3779B1 * (seed + 1) & 0x7FFFFFFF)
    return g


def _depth_frame(width, height, seed):
    """One back-projected depth frame [height*width, 3] (NaN where there is no depth): a
    fronto-parallel back plane, 5 tilted planes and 20 boxes, depth noise 0.002 z^2, 10 % of
    the pixels missing."""
    rng = np.random.default_rng(seed)
    g = _gen(seed)
    f = 525.0
    cx, cy = (width - 1) / 2.0, (height - 1) / 2.0
    u = torch.arange(width, device=DEV, dtype=torch.float64)
    v = torch.arange(height, device=DEV, dtype=torch.float64)
    dx = ((u - cx) / f)[None, :].expand(height, width)
    dy = ((v - cy) / f)[:, None].expand(height, width)
    inf = torch.full((), math.inf, device=DEV, dtype=torch.float64)
    best = torch.full((height, width), math.inf, device=DEV, dtype=torch.float64)

    def ray_point(z):
        return np.array([(rng.uniform(0, width) - cx) / f * z,
                         (rng.uniform(0, height) - cy) / f * z, z])

    for k in range(6):
        if k == 0:
            n, off = np.array([0.0, 0.0, 1.0]), rng.uniform(4.5, 5.0)
        else:
            n = rng.normal(size=3)
            n /= np.linalg.norm(n)
            off = float(n @ ray_point(rng.uniform(1.0, 5.0)))
        t = off / (float(n[0]) * dx + float(n[1]) * dy + float(n[2]))
        best = torch.minimum(best, torch.where((t >= 0.5) & (t <= 5.0), t, inf))
    for _ in range(20):
        c = ray_point(rng.uniform(1.0, 4.5))
        h = rng.uniform(0.05, 0.4, size=3)
        lo, hi = c - h, c + h
        x0, x1, y0, y1 = lo[0] / dx, hi[0] / dx, lo[1] / dy, hi[1] / dy
        near = torch.maximum(torch.minimum(x0, x1), torch.minimum(y0, y1)).clamp_min(lo[2])
        far = torch.minimum(torch.maximum(x0, x1), torch.maximum(y0, y1)).clamp_max(hi[2])
        best = torch.minimum(best, torch.where((near <= far) & (near >= 0.5) & (near <= 5.0),
                                               near, inf))
    noise = torch.randn((height, width), device=DEV, dtype=torch.float64, generator=g)
    z = torch.where(torch.isfinite(best), best + noise * 0.002 * best * best, math.nan)
    z = torch.where(torch.rand((height, width), device=DEV, generator=g) < 0.1, math.nan, z)
    return torch.stack([z * dx, z * dy, z], dim=-1).reshape(-1, 3).to(torch.float32).contiguous()


def _subset(cloud, n, seed):
    """n points of a cloud in their order."""
    keep = torch.randperm(cloud.shape[0], device=DEV, generator=_gen(seed))[:n].sort().values
    return cloud[keep].contiguous()


def _uneven_frames(case, seed):
    """Frames of uneven size (pixel-ordered subsets of 720p frames), concatenated."""
    rng = np.random.default_rng(seed + 77)
    sizes = rng.permutation(np.linspace(case["n_min"], case["n_max"], case["frames"]).astype(int))
    frames = [_subset(_depth_frame(1280, 720, 1000 * (seed + 1) + f), int(n), 31 * seed + f)
              for f, n in enumerate(sizes)]
    offsets = [0] + [int(v) for v in np.cumsum(sizes)]
    leaves = rng.choice(np.array([0.02, 0.05, 0.1], np.float32), size=case["frames"])
    return torch.cat(frames), offsets, torch.from_numpy(leaves).to(DEV)


def _map_cloud(n, seed):
    """An unordered fused map, 40 x 40 x 10 m: 70 % of the points on 8 planes and 400 boxes
    (noise 5 mm), the rest clutter, 2 % missing."""
    rng = np.random.default_rng(seed)
    g = _gen(seed)
    ext = np.array([40.0, 40.0, 10.0])
    n_surf = int(0.7 * n)
    out = torch.rand((n, 3), device=DEV, generator=g) * torch.tensor(ext, device=DEV,
                                                                     dtype=torch.float32)
    # planes: solve the axis of the largest normal component, folded back into the box
    n_plane = n_surf // 3
    per = n_plane // 8
    for k in range(8):
        nrm = rng.normal(size=3)
        nrm /= np.linalg.norm(nrm)
        pt = rng.uniform(size=3) * ext
        a = int(np.argmax(np.abs(nrm)))
        b, c = [i for i in range(3) if i != a]
        s = out[k * per:(k + 1) * per]
        s[:, a] = (float(pt[a]) - (float(nrm[b] / nrm[a]) * (s[:, b] - float(pt[b])) +
                                   float(nrm[c] / nrm[a]) * (s[:, c] - float(pt[c])))) \
            .remainder(float(ext[a]))
    # boxes: faces by area
    e = np.minimum(rng.uniform(0.2, 3.0, size=(400, 3)), ext)
    lo = rng.uniform(size=(400, 3)) * (ext - e)
    area = np.stack([e[:, 1] * e[:, 2], e[:, 0] * e[:, 2], e[:, 0] * e[:, 1]], axis=1)
    face = torch.tensor((area / area.sum()).reshape(-1), device=DEV)
    m = n_surf - n_plane
    cdf = face.cumsum(0)
    pick = torch.searchsorted(cdf, torch.rand(m, device=DEV, generator=g, dtype=torch.float64)) \
        .clamp_max(1199)
    box, axis = pick // 3, pick % 3
    q = torch.rand((m, 3), device=DEV, generator=g)
    side = torch.randint(0, 2, (m, 1), device=DEV, generator=g).to(torch.float32)
    q.scatter_(1, axis[:, None], side)
    lo_t = torch.tensor(lo, device=DEV, dtype=torch.float32)
    e_t = torch.tensor(e, device=DEV, dtype=torch.float32)
    out[n_plane:n_surf] = lo_t[box] + q * e_t[box]
    out[:n_surf] += 0.005 * torch.randn((n_surf, 3), device=DEV, generator=g)
    out[torch.randint(0, n, (int(0.02 * n),), device=DEV, generator=g)] = math.nan
    return out[torch.randperm(n, device=DEV, generator=g)].contiguous()


def _scan_cloud(n, extent, seed):
    """A terrestrial scan of a site of `extent` metres, in scan order: ground and facades
    seen from one station, range noise 5 mm, 3 % missing returns."""
    rng = np.random.default_rng(seed)
    g = _gen(seed)
    rows = 1 + n // 2048
    az = (torch.arange(2048 * rows, device=DEV) // rows).to(torch.float64)[:n] * (2 * math.pi / 2048)
    el = (torch.arange(2048 * rows, device=DEV) % rows).to(torch.float64)[:n] / rows * 0.9 - 0.5
    d = torch.stack([torch.cos(el) * torch.cos(az), torch.cos(el) * torch.sin(az),
                     torch.sin(el)], dim=-1)
    r = torch.full((n,), extent / 2, device=DEV, dtype=torch.float64)
    r = torch.minimum(r, torch.where(d[:, 2] < -1e-3, -2.0 / d[:, 2], math.inf))
    for _ in range(24):
        a = rng.uniform(0, 2 * math.pi)
        dist = rng.uniform(8.0, extent / 2)
        c = d[:, 0] * math.cos(a) + d[:, 1] * math.sin(a)
        t = torch.where(c > 0.5, dist / c, math.inf)
        r = torch.minimum(r, torch.where(c > math.cos(rng.uniform(0.05, 0.3)), t, math.inf))
    r = r + 0.005 * torch.randn(n, device=DEV, generator=g, dtype=torch.float64)
    p = (d * r[:, None] + extent / 2).to(torch.float32)
    p[torch.rand(n, device=DEV, generator=g) < 0.03] = math.nan
    return p.contiguous()


def _poses(frames, seed):
    poses, bands = synth.sensor_poses(frames, seed=seed, band=BAND)
    return torch.from_numpy(poses).to(DEV), torch.from_numpy(bands).to(DEV)


def _inputs(case, seed):
    """Everything `exact` needs too: the clouds of a case and what goes with them."""
    k = case["kind"]
    s = {"case": case}
    if k == "crop":
        s["xyz"] = _subset(_depth_frame(640, 480, seed), case["n"], seed)
    elif k in ("default", "frame", "autograd", "pyramid", "thin"):
        s["xyz"] = _depth_frame(case["width"], case["height"], seed)
        n = s["xyz"].shape[0]
        if k == "thin":
            s["priority"] = torch.randperm(n, device=DEV, generator=_gen(seed + 5)).to(torch.int32)
        if k == "autograd":
            s["grad"] = torch.randn((n, 3), device=DEV, generator=_gen(seed + 6))
    elif k == "posed_rgb":
        s["xyz"] = torch.cat([_depth_frame(case["width"], case["height"], 500 * (seed + 1) + f)
                              for f in range(case["frames"])])
        n = case["width"] * case["height"]
        s["offsets"] = [f * n for f in range(case["frames"] + 1)]
        s["leaves"] = torch.full((case["frames"],), case["leaf"], device=DEV)
        s["poses"], s["bands"] = _poses(case["frames"], seed)
        s["rgb"] = torch.randint(0, 256, (n * case["frames"], 3), device=DEV, dtype=torch.uint8,
                                 generator=_gen(seed + 7))
    elif k in ("batch", "voxel_map"):
        s["xyz"], s["offsets"], s["leaves"] = _uneven_frames(case, seed)
        if k == "voxel_map":
            s["poses"], s["bands"] = _poses(case["frames"], seed)
    elif k == "scan":
        s["xyz"] = _scan_cloud(case["n"], case["extent"], seed)
    else:
        s["xyz"] = _map_cloud(case["n"], seed)
    return s


def _rows_kept(s, n, channels=0):
    """Fixed buffers of the program that the rows of a call of its own size are copied to."""
    s["kept"] = [torch.zeros(n, dtype=torch.int64, device=DEV), torch.zeros((n, 3), device=DEV),
                 torch.zeros(n, dtype=torch.int32, device=DEV)]
    if channels:
        s["kept"].append(torch.zeros((n, channels), device=DEV))


def _keep(s, *rows):
    for dst, src in zip(s["kept"], rows):
        dst[:src.shape[0]].copy_(src)
    return tuple(s["kept"])


def _zeroed(buf):
    buf.keys.zero_()
    buf.centroids.zero_()
    buf.counts.zero_()
    return buf


def prepare(case, seed):
    s = _inputs(case, seed)
    k = case["kind"]
    n = s["xyz"].shape[0]
    if k in ("crop", "frame", "scan", "map"):
        method = "frame" if k == "frame" else "auto"
        origin = torch.tensor(FIXED_ORIGIN, device=DEV) if k == "crop" else None
        s["buf"] = _zeroed(vg.alloc_buffers(n, DEV, flags=vg.method_flag(method), origin=origin))
        s["method"] = method
    elif k == "batch":
        F = case["frames"]
        s["offsets_dev"] = torch.tensor(s["offsets"], dtype=torch.int64, device=DEV)
        s["origins"] = torch.zeros((F, 3), device=DEV)
        s["keys"] = torch.zeros(n, dtype=torch.int64, device=DEV)
        s["centroids"] = torch.zeros((n, 3), device=DEV)
        s["counts"] = torch.zeros(n, dtype=torch.int32, device=DEV)
        s["rows"] = torch.zeros(F + 1, dtype=torch.int64, device=DEV)
        s["error"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        s["plan"] = vg.Plan(F, n)
        s["stream"] = torch.cuda.Stream()  # a plan's graph needs a stream of its own
    elif k == "voxel_map":
        s["map"] = vg.VoxelMap(case["capacity"], MAP_ORIGIN, case["leaf"], device=DEV)
        _rows_kept(s, min(n, case["capacity"]))
    elif k == "pyramid":
        rows = n * case["levels"]
        s["workspace"] = torch.empty(
            vg.lib().vg_pyramid_workspace_bytes(n, case["levels"], vg.ORIGIN_FROM_MIN),
            dtype=torch.uint8, device=DEV)
        s["origin"] = torch.zeros(3, device=DEV)
        s["keys"] = torch.zeros(rows, dtype=torch.int64, device=DEV)
        s["centroids"] = torch.zeros((rows, 3), device=DEV)
        s["counts"] = torch.zeros(rows, dtype=torch.int32, device=DEV)
        s["offsets"] = torch.zeros(case["levels"] + 1, dtype=torch.int64, device=DEV)
        s["error"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    elif k in ("default", "autograd", "posed_rgb"):
        _rows_kept(s, n, 3 if k == "posed_rgb" else 0)
        s["xyz"].requires_grad_(k == "autograd")
    torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k in ("crop", "frame", "scan", "map"):
        b = s["buf"]
        vg.downsample_into(s["xyz"], case["leaf"], b, origin_from_min=k != "crop",
                           method=s["method"])
        return b.keys, b.centroids, b.counts, b.num_voxels, b.origin, b.error
    if k == "default":
        r = vg.downsample(s["xyz"], case["leaf"])
        return _keep(s, r.keys, r.centroids, r.counts) + (r.origin,)
    if k == "autograd":
        c, keys, counts = vg.VoxelDownsample.apply(s["xyz"], case["leaf"])
        (g,) = torch.autograd.grad(c, s["xyz"], s["grad"][:c.shape[0]])
        return _keep(s, keys, c.detach(), counts) + (g,)
    if k == "pyramid":  # the C interface, into kept buffers: level after level
        n, ws = s["xyz"].shape[0], s["workspace"]
        status = vg.lib().vg_pyramid(
            s["xyz"].data_ptr(), n, s["origin"].data_ptr(), case["leaf"], case["levels"],
            s["keys"].data_ptr(), s["centroids"].data_ptr(), s["counts"].data_ptr(),
            s["keys"].shape[0], s["offsets"].data_ptr(), None, s["error"].data_ptr(),
            ws.data_ptr(), ws.numel(), vg.ORIGIN_FROM_MIN,
            torch.cuda.current_stream().cuda_stream)
        if status != 0:
            raise vg.VGError(status, "vg_pyramid")
        return s["offsets"], s["error"], s["keys"], s["centroids"], s["counts"]
    if k == "thin":
        r = vg.thin(s["xyz"], case["leaf"], case["threshold"], s["priority"], batch=case["batch"])
        return r.keep, r.num_kept, r.passes, r.origin
    if k == "posed_rgb":
        r = vg.downsample_frames((s["xyz"], s["offsets"]), s["leaves"], poses=s["poses"],
                                 z_limits=s["bands"], attrs=s["rgb"],
                                 min_count=case["min_count"])
        return (r.offsets, r.origins) + _keep(s, r.keys, r.centroids, r.counts, r.attrs)
    if k == "batch":
        st = s["stream"]
        st.wait_stream(torch.cuda.current_stream())
        s["plan"].run(s["xyz"], s["offsets_dev"], case["frames"], s["origins"], s["leaves"],
                      s["keys"], s["centroids"], s["counts"], s["rows"], s["error"], stream=st)
        torch.cuda.current_stream().wait_stream(st)
        return s["rows"], s["origins"], s["error"], s["keys"], s["centroids"], s["counts"]
    m = s["map"]
    m.clear()
    m.insert((s["xyz"], s["offsets"]), s["poses"], s["bands"])
    r = m.extract()
    return _keep(s, r.keys, r.centroids, r.counts)


# ---- what a pass cannot do without -----------------------------------------------------
def _cells(area, leaf, n):
    """Expected occupied cells of n points spread over `area` square metres."""
    k = area / (leaf * leaf)
    return k * -math.expm1(-n / k)


def work(case):
    k = case["kind"]
    leaf = case.get("leaf", 0.05)
    row = 24  # key, centroid, count
    if k in ("batch", "voxel_map"):
        n = case["frames"] * (case["n_min"] + case["n_max"]) // 2
        per = n / case["frames"]
        if k == "batch":
            v = case["frames"] * sum(_cells(86.0, lf, 0.9 * per) for lf in (0.02, 0.05, 0.1)) / 3
        else:
            v = 0.4 * case["frames"] * _cells(86.0, leaf, 0.9 * per)
        return {"bytes": 12 * n + row * v, "flops": 20 * n + 6 * v}
    if k in ("scan", "map"):
        n = case["n"]
        if k == "map":
            v = _cells(20000.0, leaf, 0.69 * n) + _cells(16000.0 / leaf, leaf, 0.29 * n)
        else:
            v = 0.9 * n
        return {"bytes": 12 * n + row * v, "flops": 20 * n + 6 * v}
    if k == "crop":
        n = case["n"]
        return {"bytes": 12 * n + row * _cells(29.0, leaf, 0.9 * n), "flops": 20 * n}
    n = case["width"] * case["height"] * case.get("frames", 1)
    area = 29.0 * max(1.0, case["width"] * case["height"] / 307_200) * case.get("frames", 1)
    v = _cells(area, leaf, 0.9 * n)
    b, fl = 12 * n + row * v, 20 * n + 6 * v
    if k == "autograd":  # the points' gradient out, the centroids' in, the point's row between
        b += 12 * n + 12 * v + 2 * 4 * n
        fl += 3 * n
    elif k == "pyramid":
        b += sum(row * _cells(area, leaf * 2 ** i, 0.9 * n) for i in range(1, case["levels"]))
    elif k == "posed_rgb":
        b += 3 * n + 12 * v
        fl += 18 * n
    elif k == "thin":  # priority in, keep flag out; every pair of near neighbours once
        b = 12 * n + 4 * n + n
        fl = 9 * n * case["threshold"]
    return {"bytes": b, "flops": fl}


# ---- the outputs in 64 bits --------------------------------------------------------------
def _spread(v):
    x = v & 0x1FFFFF
    for s, m in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F),
                 (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        x = (x | (x << s)) & m
    return x


def _posed(xyz, pose, band):
    r = pose.reshape(3, 4)
    x, y, z = xyz[:, 0], xyz[:, 1], xyz[:, 2]
    p = torch.stack([((r[a, 0] * x + r[a, 1] * y) + r[a, 2] * z) + r[a, 3] for a in range(3)],
                    dim=1)
    keep = (p[:, 2] >= band[0]) & (p[:, 2] <= band[1])
    return torch.where(keep[:, None], p, math.nan)


def _decimate(xyz, leaf, origin=None):
    """Keys (the voxel index is defined in 32-bit arithmetic), 64-bit means, counts, origin
    and each point's row (-1 for an invalid point)."""
    ok = torch.isfinite(xyz).all(dim=1)
    p = xyz[ok]
    o = p.min(dim=0).values if origin is None else origin
    i = torch.floor((p - o) / leaf.reshape(1).expand(3)).to(torch.int64)
    key = _spread(i[:, 0]) | (_spread(i[:, 1]) << 1) | (_spread(i[:, 2]) << 2)
    keys, inv, counts = torch.unique(key, return_inverse=True, return_counts=True)
    sums = torch.zeros((keys.shape[0], 3), dtype=torch.float64, device=DEV)
    sums.index_add_(0, inv, p.to(torch.float64))
    row = torch.full((xyz.shape[0],), -1, dtype=torch.int64, device=DEV)
    row[ok] = inv
    return keys, sums / counts[:, None], counts, o, row


def _padded(t, n):
    out = torch.zeros((n,) + tuple(t.shape[1:]), dtype=t.dtype, device=DEV)
    out[:t.shape[0]] = t
    return out


def exact(case, seed):
    k = case["kind"]
    if k == "thin":  # whole numbers only
        return None
    s = _inputs(case, seed)
    xyz = s["xyz"]
    n = xyz.shape[0]
    leaf = torch.tensor(case.get("leaf", 0.0), dtype=torch.float32, device=DEV)
    if k in ("crop", "frame", "scan", "map"):
        o = torch.tensor(FIXED_ORIGIN, device=DEV) if k == "crop" else None
        keys, cents, counts, o, _ = _decimate(xyz, leaf, o)
        return (_padded(keys, n), _padded(cents, n), _padded(counts, n),
                torch.tensor([keys.shape[0]], device=DEV), o,
                torch.zeros(1, dtype=torch.int32, device=DEV))
    if k == "default":
        keys, cents, counts, o, _ = _decimate(xyz, leaf)
        return _padded(keys, n), _padded(cents, n), _padded(counts, n), o
    if k == "autograd":
        keys, cents, counts, _, row = _decimate(xyz, leaf)
        g = s["grad"][:keys.shape[0]].to(torch.float64) / counts[:, None]
        g = torch.where((row >= 0)[:, None], g[row.clamp_min(0)], 0.0)
        return _padded(keys, n), _padded(cents, n), _padded(counts, n), g
    if k == "pyramid":
        keys, cents, counts, _, _ = _decimate(xyz, leaf)
        out = [(keys, cents, counts)]
        for _ in range(1, case["levels"]):
            up, inv = torch.unique(keys >> 3, return_inverse=True)
            nn = torch.zeros(up.shape[0], dtype=torch.int64, device=DEV).index_add_(0, inv, counts)
            sm = torch.zeros((up.shape[0], 3), dtype=torch.float64, device=DEV)
            sm.index_add_(0, inv, cents * counts[:, None])
            keys, cents, counts = up, sm / nn[:, None], nn
            out.append((keys, cents, counts))
        offsets = [0]
        for level in out:
            offsets.append(offsets[-1] + level[0].shape[0])
        return (torch.tensor(offsets, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)) + \
            tuple(_padded(torch.cat(c), n * case["levels"]) for c in zip(*out))
    if k == "voxel_map":
        p = torch.cat([_posed(xyz[a:b], s["poses"][f], s["bands"][f]) for f, (a, b) in
                       enumerate(zip(s["offsets"], s["offsets"][1:]))])
        keys, cents, counts, _, _ = _decimate(p, leaf, torch.tensor(MAP_ORIGIN, device=DEV))
        return tuple(_padded(t, min(n, case["capacity"])) for t in (keys, cents, counts))
    rows, origins, parts = [0], [], []
    for f, (a, b) in enumerate(zip(s["offsets"], s["offsets"][1:])):
        p = xyz[a:b]
        if k == "posed_rgb":
            p = _posed(p, s["poses"][f], s["bands"][f])
        if not bool(torch.isfinite(p).all(dim=1).any()):
            origins.append(torch.zeros(3, device=DEV))
            rows.append(rows[-1])
            continue
        keys, cents, counts, o, row = _decimate(p, s["leaves"][f])
        part = [keys, cents, counts]
        if k == "posed_rgb":
            rgb = torch.zeros((keys.shape[0], 3), dtype=torch.float64, device=DEV)
            rgb.index_add_(0, row[row >= 0], s["rgb"][a:b][row >= 0].to(torch.float64))
            part.append(rgb / counts[:, None])
            kept = counts >= case["min_count"]
            part = [t[kept] for t in part]
        parts.append(part)
        origins.append(o)
        rows.append(rows[-1] + part[0].shape[0])
    cols = [torch.cat(c) for c in zip(*parts)]
    if k == "posed_rgb":
        return (rows, torch.stack(origins)) + tuple(_padded(c, n) for c in cols)
    return (torch.tensor(rows, device=DEV), torch.stack(origins),
            torch.zeros(1, dtype=torch.int32, device=DEV)) + tuple(_padded(c, n) for c in cols)
