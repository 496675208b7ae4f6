"""The work that users of this render library have it do, as cases that can be timed.

Every case goes through the public binding (paper_2502_11618_gb300.Renderer, or the C entry
lnr_filter_static): whole frames in each precision from a thumbnail to a batch of eight
1920x1080 views, the served loop, the soft z-buffer, the depth filter alone, a training pair
and the gridding of a new cloud.  Sizes are those of the library's workloads (200k points at
256x256, multi-room scans at 1920x1080, mixed resolutions served) and ragged ones between.

Nothing is autotuned: the choice of kernels, and with it the rounding of the BF16 and FP8
networks, would then depend on a timing, and two runs of one program could not be compared.

The clouds are ray-cast multi-scanner scans of rooms with furniture, made on the GPU from the
seed: density falls with distance, surfaces behind others stay empty.  Depth images of the
filter case come from such a scan too.  exact() computes the frame with plain torch: the
projection and the filter with the FP32 operations that define them (their results are
decisions: which pixel, which point, kept or not), the network in 64 bits.
"""
import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F

import paper_2502_11618_gb300 as lnr

CH3 = "16,32,64"
CH4 = "32,64,128,256"
INF = float("inf")


def listed():
    return [
        # the method as stated, in FP32, on a small room: the smallest whole frame
        frame("room_256_fp32", "fp32", 256, 256, points=200_000, room=1, cell=0.5, levels=3, ch=CH3),
        # the same at full size: one 1080p frame per call, the accuracy reference users start from
        frame("frame_1080p_fp32", "fp32", 1920, 1080, points=5_000_000, levels=5, ch=CH4),
        # an odd frame size, a net with batch norm, a few views per call
        frame("ragged_3x_bn_fp32", "fp32", 616, 424, points=1_000_000, views=3, levels=4, fs=0.5, ch=CH3, bn=True),
        # a thumbnail or preview on the tensor cores: latency and launches count
        frame("thumb_256_bf16", "bf16", 256, 256, points=200_000, room=1, cell=0.5, levels=3, ch=CH4),
        # an interactive viewer: one 1080p frame per call
        frame("frame_1080p_bf16", "bf16", 1920, 1080, points=5_000_000, levels=5, ch=CH4),
        # offline rendering of a path through a 20M-point scan: eight 1080p views per call
        frame("batch8_1080p_bf16", "bf16", 1920, 1080, points=20_000_000, views=8, levels=5, ch=CH4),
        # the fastest precision, calibrated, at 720p
        frame("batch4_720p_fp8", "fp8", 1280, 720, points=5_000_000, views=4, levels=5, fs=0.5, ch=CH4),
        # the paper's averaging of colours at similar depth
        frame("soft_720p_bf16", "bf16", 1280, 720, points=5_000_000, levels=4, ch=CH4, soft=0.01),
        # requests of mixed resolution through the serving loop, results in page-locked memory
        dict(name="served_mix_bf16", kind="serve", W=1920, H=1080, points=5_000_000, requests=12, levels=6,
             slots=3, batch=4, ch=CH4),
        # the depth filter in a host application's own frame loop
        dict(name="filter_1080p", kind="filter", W=1920, H=1080, points=2_000_000, levels=5, fs=1.0),
        # the network input of one synthetic training pair, from a ground-truth photo
        dict(name="train_pair_1080p", kind="train", W=1920, H=1080, points=2_000_000, levels=5, fs=1.0,
             unfiltered=False),
        # a new cloud or cell size: grid build, then the first z-buffer from it
        dict(name="grid_20M", kind="grid", W=320, H=240, points=20_000_000, cell=0.25),
    ]


def frame(name, prec, W, H, points, views=1, room=3, cell=0.25, levels=5, fs=1.0, ch=CH4, bn=False, soft=0.0):
    """A case of whole frames: `views` views per call, room x room rooms, `levels` filter levels."""
    return dict(name=name, kind="frame", prec=prec, W=W, H=H, points=points, views=views, room=room, cell=cell,
                levels=levels, fs=fs, ch=ch, bn=bn, soft=soft)


def draw(rng):
    """One more case of the same ranges (no larger than the largest listed)."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def size():
        px = math.exp(rng.uniform(math.log(200 * 140), math.log(1920 * 1080)))
        W = max(64, 8 * round(math.sqrt(px * rng.uniform(1.0, 1.9)) / 8))
        return W, max(64, 8 * round(px / W / 8))

    kind = rng.choice(["fp32", "fp32", "bf16", "bf16", "bf16", "fp8", "filter", "filter", "train", "grid"])
    W, H = size()
    levels = rng.randint(0 if rng.random() < 0.15 else 2, 6)
    levels = min(levels, int(math.log2(min(W, H))))
    points = log(200_000, 5_000_000)
    fs = round(rng.uniform(0.5, 1.5), 3)
    if kind == "filter":
        W, H = W - rng.randint(0, 7), H - rng.randint(0, 7)  # the filter takes any size
        return dict(kind="filter", W=W, H=H, points=points, levels=min(levels, int(math.log2(min(W, H)))), fs=fs)
    if kind == "train":
        return dict(kind="train", W=W, H=H, points=points, levels=levels, fs=fs, unfiltered=rng.random() < 0.5)
    if kind == "grid":
        return dict(kind="grid", W=320, H=240, points=log(100_000, 20_000_000), cell=rng.choice([0.125, 0.25, 0.5, 1.0]))
    most = max(1, min(8, int((4 if kind == "fp32" else 16) * 1e6 / (W * H))))
    c = frame("", kind, W, H, points, views=rng.randint(1, most), room=rng.choice([1, 2, 3]),
              cell=rng.choice([0.25, 0.5]), levels=levels, fs=fs, ch=CH4 if kind == "fp8" else rng.choice([CH3, CH4]),
              bn=rng.random() < 0.3, soft=rng.choice([0.0, 0.0, 0.01]))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs ----


def make_cloud(points, rooms, seed, dev):
    """A scan of rooms x rooms rooms (4 m each side; one room: 8 x 6 x 3 m): FP64 world
    coordinates on a 2^-12 m lattice with a georeferencing offset, colours, scanner ids, the
    boxes and the enclosure."""
    rng = np.random.Generator(np.random.PCG64(seed))
    ext = np.array([8.0, 6.0, 3.0]) if rooms == 1 else np.array([4.0 * rooms, 4.0 * rooms, 4.0])
    off = np.zeros(3) if rooms == 1 else np.array([512000.0, 5600000.0, 100.0])
    lo, hi = [], []
    for i in range(1, rooms):  # interior walls along both axes, one doorway per room side
        for ax in (0, 1):
            for j in range(rooms):
                door = 4.0 * j + rng.uniform(0.4, 2.6)
                for a, b, z0 in ((4.0 * j, door, 0.0), (door + 1.0, 4.0 * (j + 1), 0.0), (door, door + 1.0, 2.0)):
                    l, h = np.zeros(3), np.array([0.0, 0.0, ext[2]])
                    l[ax], h[ax], l[1 - ax], h[1 - ax], l[2] = 4.0 * i - 0.05, 4.0 * i + 0.05, a, b, z0
                    lo.append(l)
                    hi.append(h)
    for _ in range(10 if rooms == 1 else 3 * rooms * rooms):  # furniture
        s = rng.uniform(0.3, 1.5, 3)
        p = np.array([rng.uniform(0.15, ext[0] - 0.15 - s[0]), rng.uniform(0.15, ext[1] - 0.15 - s[1]), 0.0])
        lo.append(p)
        hi.append(p + s)
    lo, hi = np.array(lo), np.array(hi)
    scanners = free_places(rng, ext, lo, hi, 2 if rooms == 1 else 2 * rooms, (1.5, 1.5))
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    albedo = torch.as_tensor(rng.uniform(40.0, 220.0, (6 + len(lo), 3)), device=dev, dtype=torch.float32)
    blo, bhi = torch.as_tensor(lo, device=dev).float(), torch.as_tensor(hi, device=dev).float()
    e32 = torch.as_tensor(ext, device=dev).float()
    xyz, rgb, sid = [], [], []
    for s, o in enumerate(scanners):
        n = points // len(scanners) + (s < points % len(scanners))
        o32 = torch.as_tensor(o, device=dev).float()
        bright = float(rng.integers(-8, 9))
        for part in range(0, n, 1 << 20):
            m = min(1 << 20, n - part)
            u = torch.rand((3, m), generator=g, device=dev)
            z = -0.866 + 1.866 * u[0]
            az, r = 2 * math.pi * u[1], torch.sqrt(torch.clamp(1 - z * z, min=0))
            d = torch.stack([r * torch.cos(az), r * torch.sin(az), z], 1)
            d = torch.where(d.abs() < 1e-6, torch.full_like(d, 1e-6), d)
            t, face = ((torch.where(d > 0, e32, torch.zeros_like(d)) - o32) / d).min(1)  # the enclosure
            surf = 2 * face + (d.gather(1, face[:, None])[:, 0] > 0)
            for b in range(len(lo)):
                t1, t2 = (blo[b] - o32) / d, (bhi[b] - o32) / d
                near, far = torch.minimum(t1, t2).amax(1), torch.maximum(t1, t2).amin(1)
                hit = (near <= far) & (near > 1e-6) & (near < t)
                t = torch.where(hit, near, t)
                surf = torch.where(hit, torch.full_like(surf, 6 + b), surf)
            p = o32 + t[:, None] * d
            tex = torch.where(torch.floor(p / 0.25).sum(1).long() % 2 == 1, 0.82, 1.0) * (0.95 + 0.1 * u[2])
            rgb.append((albedo[surf] * tex[:, None] + bright).round().clamp(0, 255).to(torch.uint8))
            xyz.append(torch.round(p.double() * 4096) / 4096)
            sid.append(torch.full((m,), s, dtype=torch.uint8, device=dev))
    xyz = torch.cat(xyz) + torch.as_tensor(off, device=dev)
    return SimpleNamespace(xyz=xyz, rgb=torch.cat(rgb), sid=torch.cat(sid), ext=ext, off=off, lo=lo, hi=hi)


def free_places(rng, ext, lo, hi, n, z):
    """n places in the rooms, away from walls and boxes."""
    out = []
    while len(out) < n:
        p = np.array([rng.uniform(0.4, ext[0] - 0.4), rng.uniform(0.4, ext[1] - 0.4), rng.uniform(*z)])
        if not np.any(np.all((p > lo - 0.3) & (p < hi + 0.3), axis=1)):
            out.append(p)
    return out


def make_views(c, n, seed):
    """n camera poses: height 1.2 to 1.8 m, any yaw, pitch up to 15 degrees."""
    rng = np.random.Generator(np.random.PCG64(seed + 77))
    views = []
    for p in free_places(rng, c.ext, c.lo, c.hi, n, (1.2, 1.8)):
        yaw, pitch = rng.uniform(0, 2 * math.pi), math.radians(rng.uniform(-15, 15))
        f = np.array([math.cos(pitch) * math.cos(yaw), math.cos(pitch) * math.sin(yaw), math.sin(pitch)])
        right = np.array([math.sin(yaw), -math.cos(yaw), 0.0])
        views.append(SimpleNamespace(R=np.stack([right, np.cross(f, right), f]), C=np.round((p + c.off) * 4096) / 4096))
    return views


def make_intr(W, H):
    f = float(np.float32(W / 2 / math.tan(math.radians(30.0))))
    return SimpleNamespace(fx=f, fy=f, cx=W / 2, cy=H / 2, znear=0.05, zfar=100.0)


def channels(case):
    return tuple(int(x) for x in case["ch"].split(","))


def net_shapes(ch):
    """(output, input) channels of every 3x3 convolution in network order."""
    L, cin, out = len(ch), 5, []
    for c in ch:
        out += [(c, cin), (c, c)]
        cin = c
    for l in range(L - 2, -1, -1):
        out += [(ch[l], ch[l] + ch[l + 1]), (ch[l], ch[l])]
    return out


def make_weights(ch, seed, bn):
    """He-normal weights, small biases, batch-norm statistics near identity, in file order."""
    rng = np.random.Generator(np.random.PCG64(seed + 5))
    parts = []
    for co, ci in net_shapes(ch):
        parts += [rng.normal(0.0, math.sqrt(2 / (9 * ci)), co * ci * 9), rng.uniform(-0.05, 0.05, co)]
    parts += [rng.normal(0.0, math.sqrt(2 / ch[0]), 3 * ch[0]), rng.uniform(-0.05, 0.05, 3)]
    if bn:
        for c in ch:
            for _ in range(2):
                parts += [rng.uniform(0.8, 1.2, c), rng.uniform(-0.05, 0.05, c), rng.uniform(-0.1, 0.1, c),
                          rng.uniform(0.5, 1.5, c)]
    return np.concatenate(parts).astype(np.float32)


def inputs(case, seed):
    """What both the library and exact() start from."""
    dev = torch.device("cuda", 0)
    k = case["kind"]
    s = SimpleNamespace(case=case, cloud=make_cloud(case["points"], case.get("room", 3), seed, dev), cell=case.get("cell", 0.25))
    W, H = case["W"], case["H"]
    if k == "serve":
        rng = np.random.Generator(np.random.PCG64(seed + 3))
        views = make_views(s.cloud, case["requests"], seed)
        s.requests = []
        for i, v in enumerate(views):  # a third of the requests at each of three resolutions
            w, h = ((W, H), (W * 2 // 3, H * 2 // 3), (W // 3, H // 3))[i % 3]
            s.requests.append((v, make_intr(w, h), w, h, int(rng.integers(4, case["levels"] + 1)),
                               float(np.float32(rng.uniform(0.5, 1.5)))))
    else:
        s.views = make_views(s.cloud, case.get("views", 1), seed)
        s.intr = make_intr(W, H)
    if k in ("frame", "serve"):
        s.ch = channels(case)
        s.weights = make_weights(s.ch, seed, case.get("bn", False))
    if k == "train":
        g = torch.Generator(device=dev)
        g.manual_seed(seed + 9)
        s.photo = torch.rand((H, W, 3), generator=g, device=dev).cpu().numpy()
    return s


def renderer(s):
    r = lnr.Renderer(0)
    r.load_cloud(s.cloud.xyz.cpu().numpy(), s.cloud.rgb.cpu().numpy(), s.cloud.sid.cpu().numpy())
    r.build_grid(s.cell)
    return r


def prepare(case, seed):
    s = inputs(case, seed)
    k, W, H = case["kind"], case["W"], case["H"]
    dev = torch.device("cuda", 0)
    if k == "filter":
        s.depth = project(s, s.views[0], s.intr, W, H)[0]
        s.kept = torch.empty_like(s.depth)
        s.fn, s.stream = lnr.lib().lnr_filter_static, torch.cuda.current_stream().cuda_stream
    else:
        s.r = renderer(s)
    if k == "frame":
        fp8 = case["prec"] == "fp8"
        s.r.set_unet(s.ch, s.weights, "bf16" if fp8 else case["prec"], has_bn=case["bn"])
        s.r.set_soft_zbuffer(case["soft"])
        if fp8:  # static scales from two other views
            s.r.calibrate(make_views(s.cloud, 2, seed + 1000), s.intr, W, H, case["levels"], case["fs"])
            s.r.set_precision("fp8")
        s.out = torch.empty((case["views"], H, W, 3), dtype=torch.float32, device=dev)
    elif k == "serve":
        s.r.set_unet(s.ch, s.weights, "bf16")
        s.out = [torch.empty((h, w, 3), dtype=torch.float32).pin_memory() for _, _, w, h, _, _ in s.requests]
        s.r.serve_start(max_batch=case["batch"], slots=case["slots"])
    s.cloud.xyz = s.cloud.rgb = s.cloud.sid = None  # the library holds the cloud
    return s


def run(s):
    c = s.case
    k, W, H = c["kind"], c["W"], c["H"]
    if k == "frame":
        return s.r.render_batch(s.views, s.intr, W, H, c["levels"], c["fs"], out=s.out)
    if k == "serve":
        tickets = [s.r.submit_into(*q, o) for q, o in zip(s.requests, s.out)]
        while tickets:
            tickets = [t for t in tickets if s.r.poll(t)[1] is None]
        return s.out
    if k == "filter":
        st = s.fn(ctypes.c_void_p(s.depth.data_ptr()), W, H, c["levels"], ctypes.c_float(c["fs"]),
                  ctypes.c_void_p(s.kept.data_ptr()), ctypes.c_void_p(s.stream))
        if st:
            raise RuntimeError("lnr_filter_static: %d" % st)
        return s.kept
    if k == "train":
        return s.r.training_input(s.views[0], s.intr, W, H, c["levels"], c["fs"], s.photo, c["unfiltered"])
    s.r.build_grid(c["cell"])
    g0, dims = s.r.grid_info()
    return {"g0": g0, "dims": dims, "keys": s.r.render_stage(s.views[0], s.intr, W, H, 0, 0.0, lnr.STAGE_KEYS)}


# ------------------------------------------------------------------ work ----


def work(case):
    """Bytes and operations a pass cannot do without.  A view sees about a sixth of the points
    (12 bytes each) and gathers a colour per pixel; frames come out as three floats per pixel."""
    k, px, n = case["kind"], case["W"] * case["H"], case["points"]
    if k == "filter":
        return {"bytes": 8 * px, "flops": 20 * px}
    if k == "train":
        return {"bytes": 2 * n + (12 + 20 + 4) * px, "flops": 20 * px}
    if k == "grid":  # coordinates, colours and scanner ids in; offsets, colours and keys out
        return {"bytes": (24 + 4 + 16) * n + 8 * px, "flops": 12 * n}
    ch = channels(case)
    per_px = sum(2 * 9 * co * ci / 4 ** l for (co, ci), l in zip(net_shapes(ch), net_levels(ch))) + 2 * 3 * ch[0]
    params = 4 * sum(9 * co * ci + co for co, ci in net_shapes(ch))
    if k == "serve":
        px, views = px * case["requests"] * (1 + 4 / 9 + 1 / 9) / 3, case["requests"]
    else:
        px, views = px * case["views"], case["views"]
    return {"bytes": 2 * n * views + (4 + 12) * px + params, "flops": per_px * px + 30 * n / 6 * views}


def net_levels(ch):
    L = len(ch)
    return [l for l in range(L) for _ in (0, 1)] + [l for l in range(L - 2, -1, -1) for _ in (0, 1)]


# ----------------------------------------------------------------- exact ----


def fma32(a, b, c):
    """a * b + c with one rounding to FP32 (the product of two FP32 values is exact in FP64)."""
    return (a.double() * b.double() + c.double()).float()


def f32(x, dev):
    return torch.tensor(float(np.float32(x)), dtype=torch.float32, device=dev)


def grid_of(s):
    """Points sorted stably by cell: cell indices, FP32 offsets to the cells' origins, colours."""
    c, cell = s.cloud, s.cell
    lo, hi = c.xyz.amin(0), c.xyz.amax(0)
    g0 = torch.floor(lo / cell) * cell
    dims = torch.floor((hi - g0) / cell) + 1
    ijk = torch.minimum(torch.floor((c.xyz - g0) / cell).clamp(min=0), dims - 1).long()
    d = dims.long()
    order = torch.sort((ijk[:, 2] * d[1] + ijk[:, 1]) * d[0] + ijk[:, 0], stable=True)[1]
    ijk = ijk[order]
    offs = (c.xyz[order] - (g0 + ijk.double() * cell)).float()
    return g0.cpu().numpy(), dims.cpu().numpy(), ijk, offs, c.rgb[order].long()


def project(s, view, intr, W, H, soft=0.0):
    """(depth, rgb) of the 1x1-pixel z-buffer: +inf and 0 where no point falls."""
    if not hasattr(s, "grid"):
        s.grid = grid_of(s)
    g0, dims, ijk, offs, rgb = s.grid
    dev = offs.device
    anchor = np.clip(np.floor((view.C - g0) / s.cell), 0, dims - 1)
    rel = (g0 + anchor * s.cell) - view.C
    di = (ijk - torch.as_tensor(anchor, device=dev).long()).float()
    p = []
    for r in range(3):
        R = view.R[r]
        o = f32((R[0] * rel[0] + R[1] * rel[1]) + R[2] * rel[2], dev).expand(len(di))
        for a in range(3):
            o = fma32(di[:, a], f32(R[a] * s.cell, dev), o)
        for a in (2, 1, 0):
            o = fma32(f32(R[a], dev), offs[:, a], o)
        p.append(o)
    z = p[2]
    u = (f32(intr.fx, dev) * p[0]) / z + f32(intr.cx, dev)
    v = (f32(intr.fy, dev) * p[1]) / z + f32(intr.cy, dev)
    ok = (z > f32(intr.znear, dev)) & (z < f32(intr.zfar, dev)) & (u >= 0) & (u < W) & (v >= 0) & (v < H)
    at = ok.nonzero()[:, 0]
    pix = torch.floor(v[at]).long() * W + torch.floor(u[at]).long()
    key = (z[at].view(torch.int32).long() << 32) | at
    most = torch.iinfo(torch.int64).max
    keys = torch.full((W * H,), most, dtype=torch.int64, device=dev).scatter_reduce(0, pix, key, "amin")
    filled = keys != most
    depth = torch.full((W * H,), INF, device=dev)
    depth[filled] = (keys[filled] >> 32).int().view(torch.float32)
    col = torch.zeros((W * H, 3), dtype=torch.int64, device=dev)
    if soft > 0:
        limit = depth * (np.float32(1) + np.float32(soft))
        near = z[at] <= limit[pix]
        n = torch.zeros(W * H, dtype=torch.int64, device=dev).index_add(0, pix[near], torch.ones_like(pix[near]))
        total = col.index_add(0, pix[near], rgb[at[near]])
        col[filled] = ((total + (n // 2)[:, None]) // n.clamp(min=1)[:, None])[filled]
    else:
        col[filled] = rgb[keys[filled] & 0xFFFFFFFF]
    return depth.view(H, W), col.view(H, W, 3)


def depth_filter(depth, levels, fs):
    """Kept depth, +inf where empty or filtered out."""
    if not levels:
        return depth
    M = [depth]
    for _ in range(levels):
        m = M[-1]
        m = F.pad(m, (0, m.shape[1] & 1, 0, m.shape[0] & 1), value=INF)
        M.append(torch.minimum(torch.minimum(m[::2, ::2], m[::2, 1::2]), torch.minimum(m[1::2, ::2], m[1::2, 1::2])))
    S = float(np.float32(1) + np.float32(fs) * np.float32(0.05))
    U = M[levels]

    def around(x):
        return F.pad(x[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]

    for l in range(levels - 1, -1, -1):
        fine, d = M[l], M[l + 1]
        (h, w), (H, W) = d.shape, fine.shape
        D, V = around(d), around(U)
        t = [torch.where(n == INF, torch.zeros_like(d), n - d)
             for n in (D[1:-1, :-2], D[1:-1, 2:], D[:-2, 1:-1], D[2:, 1:-1])]
        lap = (t[0] + t[1]) + (t[2] + t[3])
        edge = (d != INF) & (lap.abs() > float(np.float32(0.1)) * d)
        least = torch.stack([V[b:b + h, a:a + w] for b in range(3) for a in range(3)]).amin(0)
        thr = torch.where(edge, least, U) * S
        up = lambda x: x.repeat_interleave(2, 0).repeat_interleave(2, 1)[:H, :W]  # noqa: E731
        keep = (fine <= up(thr)) & (fine != INF)
        val = torch.where(keep, fine, torch.full_like(fine, INF))
        if l:  # empty pixels of non-final levels: bilinear from the taps that are not empty
            num, den = torch.zeros_like(fine), torch.zeros_like(fine)
            y, x = torch.arange(H, device=d.device)[:, None], torch.arange(W, device=d.device)[None]
            ys, xs, yf, xf = y // 2 + 1, x // 2 + 1, y // 2 + 2 * (y % 2), x // 2 + 2 * (x % 2)
            for a, b, wt in ((ys, xs, 0.5625), (ys, xf, 0.1875), (yf, xs, 0.1875), (yf, xf, 0.0625)):
                tap = V[a, b]
                num = num + torch.where(tap == INF, torch.zeros_like(tap), tap * wt)
                den = den + torch.where(tap == INF, torch.zeros_like(tap), torch.full_like(tap, wt))
            val = torch.where(~keep & (den > 0), num / den, val)
        U = val
    return U


def conv64(x, w, b):
    """3x3 convolution, zero padding, ReLU in FP64: nine matrix products."""
    C, H, W = x.shape
    p = F.pad(x, (1, 1, 1, 1))
    y = b[:, None].expand(-1, H * W).clone()
    for ky in range(3):
        for kx in range(3):
            y.addmm_(w[:, :, ky, kx].contiguous(), p[:, ky:ky + H, kx:kx + W].reshape(C, H * W))
    return y.clamp_(min=0).view(-1, H, W)


def net64(x, ch, weights, bn):
    """The U-Net in FP64: x (5, H, W) -> (H, W, 3)."""
    flat = torch.as_tensor(weights, device=x.device).double()
    at = [0]

    def take(*shape):
        n = math.prod(shape)
        at[0] += n
        return flat[at[0] - n:at[0]].view(*shape)

    convs = [(take(co, ci, 3, 3), take(co)) for co, ci in net_shapes(ch)]
    head = take(3, ch[0]), take(3)
    if bn:
        for i in range(2 * len(ch)):
            g, be, mu, var = (take(ch[i // 2]) for _ in range(4))
            sc = g / torch.sqrt(var + 1e-5)
            convs[i] = convs[i][0] * sc[:, None, None, None], (convs[i][1] - mu) * sc + be
    skips, i, L = [], 0, len(ch)
    for l in range(L):
        x = conv64(conv64(x, *convs[i]), *convs[i + 1])
        i += 2
        if l < L - 1:
            skips.append(x)
            x = F.max_pool2d(x[None], 2)[0]
    for l in range(L - 2, -1, -1):
        x = torch.cat([skips[l], x.repeat_interleave(2, 1).repeat_interleave(2, 2)])
        x = conv64(conv64(x, *convs[i]), *convs[i + 1])
        i += 2
    y = torch.addmm(head[1][:, None].expand(-1, x[0].numel()), head[0], x.view(ch[0], -1))
    return torch.sigmoid(y).T.reshape(x.shape[1], x.shape[2], 3)


def net_input(depth, kept, rgb, zfar):
    on = kept != INF
    chans = [rgb[..., k].double() / 255 for k in range(3)] + [depth.double() / zfar, torch.ones_like(depth).double()]
    return torch.stack([torch.where(on, v, torch.zeros_like(v)) for v in chans])


def exact(case, seed):
    k, W, H = case["kind"], case["W"], case["H"]
    if k == "grid":
        return None  # whole numbers, and a grid frame of exact multiples of the cell
    s = inputs(case, seed)

    def whole_frame(view, intr, w, h, levels, fs, soft=0.0):
        depth, rgb = project(s, view, intr, w, h, soft)
        x = net_input(depth, depth_filter(depth, levels, fs), rgb, intr.zfar)
        return net64(x, s.ch, s.weights, case.get("bn", False))

    if k == "frame":
        return torch.stack([whole_frame(v, s.intr, W, H, case["levels"], case["fs"], case["soft"]) for v in s.views])
    if k == "serve":
        return [whole_frame(*q) for q in s.requests]
    depth, rgb = project(s, s.views[0], s.intr, W, H)
    kept = depth_filter(depth, case["levels"], case["fs"])
    if k == "filter":
        return kept.double()
    fg, filled = kept != INF, depth != INF
    photo = torch.as_tensor(s.photo, device=depth.device).double()
    use = filled if case["unfiltered"] else fg
    col = torch.where(fg[..., None], photo, rgb.double() / 255)
    out = torch.cat([col, (depth.double() / s.intr.zfar)[..., None], torch.ones_like(depth).double()[..., None]], -1)
    return torch.where(use[..., None], out, torch.zeros_like(out))
