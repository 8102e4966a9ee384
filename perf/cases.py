"""Workloads of the reconstruction library, for timing and for comparing two builds.

Every case goes through the public entry points of ``paper_1712_03084_gb300``
(the C-named calls of ``ftr`` and the slots of ``serve``) on seeded synthetic
inputs made on the GPU: a capsule body seen by a ring of depth cameras, a
sphere, a field of smooth blobs, or an ellipsoid mesh.  Kinds:

  points    oriented points in device memory -> splat, solve, mesh (host waits
            for the level and the mesh, the plain synchronous use)
  frame     the queued frame: every camera's points, then solve + mesh +
            texture as one graph replay
  rgbd      the same from depth maps only (Sec. III-A on the device)
  batch     serving slots: frames of mixed grids copied in from page-locked
            host memory, all queued at once, results copied out
  solve     splat + transforms + level with the indicator read out, in FP32 or
            in the split-precision arithmetic
  mesh      marching cubes of a given indicator
  texture   per-vertex texture data of given vertices
  evaluate  rendering and the objective metrics of Sec. III-E
  level     the allocation-free iso-level
"""

import math

import numpy as np
import torch

from paper_1712_03084_gb300 import ftr, serve

DEV = "cuda"
CENTRE = (0.0, 0.95, 0.0)
CUBE = (-1.0, -0.05, -1.0, 1.0, 1.95, 1.0)            # 2 m cube around the body
TALL = (-0.8, -0.05, -0.8, 0.8, 1.95, 0.8)            # elongated grids 2^r x 2^(r+1) x 2^r
SPHERE = (-1.2, -1.2, -1.2, 1.2, 1.2, 1.2)
PREC = {"fp32": ftr.FTR_PREC_FP32, "bf16x3": ftr.FTR_PREC_BF16X3, "fp16x3": ftr.FTR_PREC_FP16X3}


def listed():
    return [
        # the smallest use: 20,000 points of a sphere on 64^3, plain synchronous calls
        dict(name="points_sphere_64", kind="points", source="sphere", nx=64, ny=64, nz=64, points=20000, simple=False),
        # the paper's largest grid (2^r x 2^(r+1) x 2^r, r = 7) with the simple nearest-node splat
        dict(name="points_simple_r7", kind="points", source="body", nx=128, ny=256, nz=128, cams=4, dw=512, dh=424,
             simple=True),
        # the headline: one textured frame, four cameras, 256^3
        dict(name="frame_256", kind="frame", nx=256, ny=256, nz=256, cams=4, dw=512, dh=424),
        # the largest grid that live sessions use
        dict(name="frame_384", kind="frame", nx=384, ny=384, nz=384, cams=5, dw=512, dh=424),
        # a live RGB-D session: depth maps in, confidence maps, mesh and texture out; six cameras
        dict(name="rgbd_192", kind="rgbd", nx=192, ny=192, nz=192, cams=6, dw=512, dh=424),
        # concurrent sessions of mixed grids and rigs, inputs and results in host memory
        dict(name="batch_mixed", kind="batch", grids="128,192,256", cams=4, dw=512, dh=424),
        # the split-precision transforms at the two grids they are used on
        dict(name="solve_256_fp16x3", kind="solve", nx=256, ny=256, nz=256, cams=4, dw=512, dh=424, prec="fp16x3"),
        dict(name="solve_384_bf16x3", kind="solve", nx=384, ny=384, nz=384, cams=4, dw=512, dh=424, prec="bf16x3"),
        # marching cubes alone, on a surface much larger than one body's
        dict(name="mesh_blobs_256", kind="mesh", nx=256, ny=256, nz=256, blobs=40),
        # texture data of a large mesh seen by six cameras
        dict(name="texture_300k", kind="texture", verts=300007, cams=6, dw=512, dh=424),
        # objective evaluation of a mesh in two views: renders, geometry and appearance metrics
        dict(name="evaluate_2_views", kind="evaluate", nu=240, nv=320, cams=2, dw=512, dh=424, rw=1920, rh=1080),
        # the level of a given indicator under a latency budget (no allocation)
        dict(name="level_200k", kind="level", nx=256, ny=256, nz=256, points=200003),
    ]


def draw(rng):
    kind = rng.choice(["points", "points", "frame", "frame", "rgbd", "batch", "solve", "solve", "mesh", "texture",
                       "evaluate", "level"])
    s = math.exp(rng.uniform(math.log(0.5), math.log(1.4)))
    cam = dict(cams=rng.randint(3, 6), dw=int(512 * s) + rng.randint(0, 3), dh=int(424 * s) + rng.randint(0, 3))
    n = rng.choice([64, 96, 128, 192, 256])
    shape = rng.choice([(n, n, n), (n, n, n), (n // 2, n, n // 2)]) if n > 64 else (n, n, n)
    grid = dict(nx=shape[0], ny=shape[1], nz=shape[2])
    if kind == "points":
        if rng.random() < 0.5:
            return dict(kind=kind, source="sphere", points=int(math.exp(rng.uniform(math.log(2000), math.log(400000)))),
                        simple=rng.random() < 0.3, **grid)
        return dict(kind=kind, source="body", simple=rng.random() < 0.3, **grid, **cam)
    if kind in ("frame", "rgbd"):
        return dict(kind=kind, **grid, **cam)
    if kind == "batch":
        g = [rng.choice([64, 96, 128, 192, 256]) for _ in range(rng.randint(2, 3))]
        return dict(kind=kind, grids=",".join(str(v) for v in g), **cam)
    if kind == "solve":
        prec = rng.choice(["fp32", "bf16x3", "fp16x3"])
        n = rng.choice([64, 128, 256] if prec != "fp32" else [48, 96, 192, 256, 384])
        return dict(kind=kind, nx=n, ny=n, nz=n, prec=prec, **cam)
    if kind == "mesh":
        return dict(kind=kind, blobs=rng.randint(3, 40), **grid)
    if kind == "texture":
        return dict(kind=kind, verts=int(math.exp(rng.uniform(math.log(3000), math.log(300000)))), **cam)
    if kind == "evaluate":
        r = rng.uniform(0.4, 1.0)
        return dict(kind=kind, nu=rng.randint(60, 240), nv=rng.randint(80, 320), cams=rng.randint(1, 2), dw=cam["dw"],
                    dh=cam["dh"], rw=int(1920 * r), rh=int(1080 * r))
    return dict(kind=kind, points=int(math.exp(rng.uniform(math.log(2000), math.log(1000000)))), **grid)


# ------------------------------------------------------------------- inputs

def _t(v):
    return torch.as_tensor(v, dtype=torch.float64, device=DEV)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 2 + 1)
    return g


def _grid(case):
    return case["nx"], case["ny"], case["nz"]


def _box(case):
    if case.get("source") == "sphere":
        return SPHERE
    return CUBE if case["nx"] == case["ny"] else TALL


def _capsules(rng):
    """Segments and radii of a ~1.8 m body in a random pose (joint angles within 40 degrees)."""
    def rot(axis):
        a = math.radians(rng.uniform(-40.0, 40.0))
        c, s = math.cos(a), math.sin(a)
        return np.array([[1, 0, 0], [0, c, -s], [0, s, c]] if axis == 0 else [[c, -s, 0], [s, c, 0], [0, 0, 1]])
    segs = [((0, .95, 0), (0, 1.32, 0), .15), ((-.12, 1.33, 0), (.12, 1.33, 0), .11),
            ((-.07, .92, 0), (.07, .92, 0), .13), ((0, 1.4, 0), (0, 1.5, 0), .05), ((0, 1.6, 0), (0, 1.67, 0), .1)]
    for side in (-1.0, 1.0):
        for start, bones, down in (((side * .2, 1.36, 0), ((.28, .05), (.25, .042), (.08, .045)), (side * .5, -1, 0)),
                                   ((side * .1, .88, 0), ((.4, .075), (.38, .055), (.1, .05)), (side * .08, -1, 0))):
            p, R = np.array(start), rot(0) @ rot(2)
            d = np.array(down) / np.linalg.norm(down)
            for length, r in bones:
                q = p + length * (R @ d)
                segs.append((tuple(p), tuple(q), r))
                p, R = q, R @ rot(0)
    yaw = rng.uniform(0.0, 2.0 * math.pi)
    c, s = math.cos(yaw), math.sin(yaw)
    Y = np.array([[c, 0, s], [0, 1, 0], [-s, 0, c]])
    out = [(Y @ np.array(a), Y @ np.array(b), r) for a, b, r in segs]
    low = min(min(a[1], b[1]) - r for a, b, r in out)
    return [(a - (0, low - .05, 0), b - (0, low - .05, 0), r) for a, b, r in out]


def _raycast(segs, o, d):
    """Distance along the unit rays o + t d to the capsules (inf on a miss)."""
    best = torch.full(d.shape[:-1], math.inf, dtype=torch.float64, device=DEV)
    inf = torch.full_like(best, math.inf)

    def ball(c, r):
        m = o - c
        b = d @ m
        h = b * b - (m @ m - r * r)
        return torch.where(h >= 0, -b - torch.sqrt(h.clamp(min=0)), inf)
    for a, b, r in segs:
        a, b = _t(a), _t(b)
        best = torch.minimum(best, torch.minimum(ball(a, r), ball(b, r)))
        u = (b - a) / (b - a).norm()
        length = (b - a).norm()
        du, m = d @ u, o - a
        mu = m @ u
        dp, mp = d - du[..., None] * u, m - mu * u
        A, B, C = (dp * dp).sum(-1), dp @ mp, mp @ mp - r * r
        h = B * B - A * C
        t = (-B - torch.sqrt(h.clamp(min=0))) / A.clamp(min=1e-300)
        y = mu + t * du
        best = torch.minimum(best, torch.where((h >= 0) & (A > 1e-12) & (y >= 0) & (y <= length), t, inf))
    return best


def _cameras(case, rng, ring):
    """Depth cameras on a ring looking at the body: (K, world_to_cam, K_rgb, world_to_rgb), float32."""
    k, w, h = case["cams"], case["dw"], case["dh"]
    f = 365.0 * w / 512.0
    rw, rh = case.get("rw", 1920), case.get("rh", 1080)
    fr = 1060.0 * rw / 1920.0
    out, phase = [], rng.uniform(0.0, 2.0 * math.pi / k)
    for i in range(k):
        a = phase + 2.0 * math.pi * i / k
        pos = np.array([ring * math.cos(a), 1.2, ring * math.sin(a)])
        z = np.array(CENTRE) - pos
        z /= np.linalg.norm(z)
        x = np.cross(z, (0, 1, 0))
        x /= np.linalg.norm(x)
        R = np.stack([x, np.cross(z, x), z])
        RT = np.concatenate([R, (-R @ pos)[:, None]], 1).astype(np.float32)
        RTr = RT.copy()
        RTr[0, 3] -= np.float32(0.05)                   # the RGB camera sits 5 cm beside the depth camera
        K = np.array([[f, 0, (w - 1) / 2], [0, f, (h - 1) / 2], [0, 0, 1]], np.float32)
        Kr = np.array([[fr, 0, (rw - 1) / 2], [0, fr, (rh - 1) / 2], [0, 0, 1]], np.float32)
        out.append((K, RT, Kr, RTr))
    return out


def _pixel_rays(K, w, h):
    K = K.astype(np.float64)
    v, u = torch.meshgrid(_t(np.arange(h)), _t(np.arange(w)), indexing="ij")
    return torch.stack([(u - K[0, 2]) / K[0, 0], (v - K[1, 2]) / K[1, 1], torch.ones_like(u)], -1)


def _raw(depth, K, RT):
    """Points, normals (camera space), validity and confidence of a depth map in
    float64: two triangles per 2 x 2 quad, dropped across depth steps (Sec. III-A)."""
    D = depth.double()
    h, w = D.shape
    X = _pixel_rays(K, w, h) * D[..., None]
    acc = torch.zeros_like(X)
    cnt = torch.zeros_like(D)
    s0, s1 = slice(0, -1), slice(1, None)
    for tri in (((s0, s0), (s0, s1), (s1, s0)), ((s0, s1), (s1, s1), (s1, s0))):
        z = [D[a] for a in tri]
        p = [X[a] for a in tri]
        top = torch.maximum(torch.maximum(z[0], z[1]), z[2])
        gap = torch.maximum(torch.maximum((z[0] - z[1]).abs(), (z[1] - z[2]).abs()), (z[0] - z[2]).abs())
        n = torch.linalg.cross(p[1] - p[0], p[2] - p[0])
        ln = n.norm(dim=-1)
        ok = (z[0] > 0) & (z[1] > 0) & (z[2] > 0) & (gap <= 0.03 + 3 * 0.0012 * top * top) & (ln > 0)
        n = torch.where(ok[..., None], n / torch.where(ln > 0, ln, 1.0)[..., None], 0.0)
        n = torch.where(((n * (p[0] + p[1] + p[2])).sum(-1) > 0)[..., None], -n, n)
        for a in tri:
            acc[a] += n
            cnt[a] += ok
    ln = acc.norm(dim=-1)
    valid = (D > 0) & (cnt > 0) & (ln > 0)
    N = torch.where(valid[..., None], acc / torch.where(ln > 0, ln, 1.0)[..., None], 0.0)
    w1 = (-(X * N).sum(-1) / X.norm(dim=-1).clamp(min=1e-300)).clamp(min=0)
    w2 = torch.nn.functional.avg_pool2d((D > 0).double()[None, None], 21, 1, 10)[0, 0]
    return X, N, valid, torch.where(valid, w1 * w2, 0.0)


def _views(case, seed, ring=2.5, rgb=True):
    """RGB-D views of a body (device tensors) and, per camera, its points, normals, weights."""
    rng, g = np.random.default_rng(seed), _gen(seed)
    segs = _capsules(rng)
    views, sets = [], []
    for K, RT, Kr, RTr in _cameras(case, rng, ring):
        w, h = case["dw"], case["dh"]
        R, t = _t(RT[:, :3]), _t(RT[:, 3])
        rays = _pixel_rays(K, w, h)
        ln = rays.norm(dim=-1)
        z = _raycast(segs, -(t @ R), (rays / ln[..., None]) @ R) / ln
        noise = torch.randn(z.shape, generator=g, device=DEV, dtype=torch.float64)
        depth = torch.where(torch.isfinite(z), z + 0.0012 * z * z * noise, 0.0).float().contiguous()
        X, N, valid, W = _raw(depth, K, RT)
        v = dict(depth=depth, conf=W.float().contiguous(), K=K, world_to_cam=RT, K_rgb=Kr, world_to_rgb=RTr)
        if rgb:
            v["rgb"] = _pattern(rng, case.get("rw", 1920), case.get("rh", 1080))
        views.append(v)
        sets.append((((X[valid] - t) @ R).float().contiguous(), (N[valid] @ R).float().contiguous(),
                     W[valid].float().contiguous()))
    return views, sets


def _pattern(rng, w, h):
    """A smooth RGB image with a seeded pattern."""
    v, u = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
    chan = []
    for _ in range(3):
        a, b, p = rng.uniform(0.01, 0.05), rng.uniform(0.01, 0.05), rng.uniform(0, 6.28)
        chan.append(128 + 100 * torch.sin(a * u + p) * torch.cos(b * v - p))
    return torch.stack(chan, -1).round().to(torch.uint8).contiguous()


def _sphere(case, seed):
    g = _gen(seed)
    n = torch.randn((case["points"], 3), generator=g, device=DEV, dtype=torch.float64)
    n = n / n.norm(dim=1, keepdim=True)
    p = n + 0.005 * torch.randn(n.shape, generator=g, device=DEV, dtype=torch.float64)
    return p.float().contiguous(), n.float().contiguous(), torch.ones(case["points"], device=DEV)


def _field(case, seed):
    """An indicator of smooth blobs (value about 1 inside) and its level."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = _grid(case)
    k = case["blobs"]
    c, s = _t(rng.uniform(0.15, 0.85, (3, k, 1))), _t(rng.uniform(0.05, 0.11, (k, 1)))
    e = [torch.exp(-(((torch.arange(n, device=DEV) + 0.5) / n - c[a]) / s) ** 2) for a, n in enumerate((nx, ny, nz))]
    A = torch.einsum("kz,ky,kx->zyx", e[2], e[1], e[0])
    return A.float().contiguous(), 0.45


def _surface(case, seed):
    """A rippled ellipsoid mesh with vertex colours, and the smooth ellipsoid behind it."""
    rng = np.random.default_rng(seed)
    nu, nv = case["nu"], case["nv"]
    th = _t((np.arange(nu) + 0.5) / nu * math.pi)[:, None]
    ph = _t(np.arange(nv) / nv * 2 * math.pi)[None, :]
    d = torch.stack([torch.sin(th) * torch.cos(ph), torch.cos(th) * torch.ones_like(ph), torch.sin(th) * torch.sin(ph)], -1)
    radii, a, b = _t((0.35, 0.85, 0.3)), int(rng.integers(3, 9)), int(rng.integers(3, 9))
    bump = 1.0 + 0.02 * torch.sin(a * th + float(rng.uniform(0, 6))) * torch.sin(b * ph + float(rng.uniform(0, 6)))
    verts = (d * radii * bump[..., None] + _t(CENTRE)).reshape(-1, 3).float().contiguous()
    i, j = torch.meshgrid(torch.arange(nu - 1, device=DEV), torch.arange(nv, device=DEV), indexing="ij")
    p00, p01 = i * nv + j, i * nv + (j + 1) % nv
    p10, p11 = p00 + nv, p01 + nv
    tris = torch.stack([torch.stack([p00, p01, p10], -1), torch.stack([p01, p11, p10], -1)], 2)
    colour = (128 + 100 * torch.sin(9 * d + float(rng.uniform(0, 6)))).reshape(-1, 3).round().to(torch.uint8)
    return verts, tris.reshape(-1, 3).to(torch.int32).contiguous(), colour.contiguous(), radii


# ------------------------------------------------------------ prepare and run

def _tol(grid, box):
    h = max((box[3 + a] - box[a]) / grid[a] for a in range(3))
    return float(np.float32(max(3.0 * h, 0.02)))


def _cap(grid):
    """Vertices that the buffers of a grid hold; what a mesh leaves free stays zero."""
    return max(1 << 15, 4 * grid[0] * max(grid[1:]))


def _mesh_buffers(cap):
    return (torch.zeros((cap, 3), device=DEV), torch.zeros((cap, 3), device=DEV),
            torch.zeros((2 * cap, 3), dtype=torch.int32, device=DEV))


def prepare(case, seed):
    state = _PREPARE[case["kind"]](case, seed)
    state["kind"] = case["kind"]
    torch.cuda.synchronize()
    return state


def run(state):
    return _RUN[state["kind"]](state)


def _context(case, **kw):
    return ftr.Context(_grid(case), _box(case), **kw)


def _prepare_points(case, seed):
    if case["source"] == "sphere":
        sets = [_sphere(case, seed)]
    else:
        sets = _views(case, seed, rgb=False)[1]
    ctx = _context(case, splat_mode=ftr.FTR_SPLAT_SIMPLE if case["simple"] else ftr.FTR_SPLAT_WEIGHTED)
    st = dict(ctx=ctx, sets=sets, mesh=_mesh_buffers(_cap(_grid(case))))
    torch.cuda.synchronize()
    _run_points(st)                      # a resident context: its buffers have their size, its plans are chosen
    ctx.autotune()
    return st


def _run_points(st):
    ctx = st["ctx"]
    ctx.reset()
    for s in st["sets"]:
        ctx.splat(*s)
    level = ctx.solve()
    return dict(_mesh_out(ctx, ctx.extract_mesh(), st["mesh"]), level=level)


def _mesh_out(ctx, m, buf):
    v, n, t = buf
    if m.n_vertices > len(v) or m.n_tris > len(t):
        raise RuntimeError("the mesh does not fit its buffers")
    ftr.ftr_mesh_copy_async(ctx.h, v, n, t)
    return dict(vertices=v, normals=n, tris=t, counts=[m.n_vertices, m.n_tris])


def _prepare_frame(case, seed):
    views, sets = _views(case, seed)
    grid, k = _grid(case), case["cams"]
    cap = _cap(grid)
    ctx = _context(case)
    st = dict(ctx=ctx, views=views, sets=sets, mesh=_mesh_buffers(cap), tol=_tol(grid, _box(case)), cap=cap,
              tex=(torch.zeros((cap, k), device=DEV), torch.zeros((cap, k, 2), device=DEV),
                   torch.zeros((cap, 3), dtype=torch.uint8, device=DEV),
                   torch.zeros((cap,), dtype=torch.uint8, device=DEV)))
    if case["kind"] == "rgbd":
        st["conf"] = [torch.empty_like(v["depth"]) for v in views]
        for v, c in zip(views, st["conf"]):
            v["conf"] = c                # written by the raw reconstruction
    torch.cuda.synchronize()
    _run_frame(st)                       # a resident session: buffers sized, plans chosen, the graph captured
    ctx.autotune()
    _run_frame(st)
    return st


def _run_frame(st):
    ctx = st["ctx"]
    ctx.reset()
    if "conf" in st:
        ftr.ftr_splat_depth(ctx.h, st["views"], conf_out=st["conf"], wait=False)
    else:
        ctx.splat_sets(st["sets"])
    w, uv, rgb, tex = st["tex"]
    ftr.ftr_frame_launch(ctx.h, st["views"], st["tol"], w, uv, rgb, tex, st["cap"])
    out = dict(_mesh_out(ctx, ftr.ftr_frame_finish(ctx.h), st["mesh"]), weights=w, uv=uv, rgb=rgb, textured=tex)
    if "conf" in st:
        out["conf"] = st["conf"]
    return out


def _prepare_batch(case, seed):
    slots = []
    for i, n in enumerate(int(v) for v in case["grids"].split(",")):
        rig = dict(case, cams=3 + (case["cams"] + i) % 4)
        views, sets = _views(rig, seed * 16 + i, ring=2.0 + 0.5 * (i % 3))
        start, per = 0, []
        for s in sets:
            per.append((start, len(s[0])))
            start += len(s[0])
        pin = [torch.cat([s[a] for s in sets]).cpu().pin_memory() for a in range(3)]
        for v in views:
            for key in ("depth", "conf", "rgb"):
                v[key] = v[key].cpu().pin_memory()
        fin = serve.FrameInput(pin[0], pin[1], pin[2], per, views, start)
        slot = serve.Slot((n, n, n), CUBE, fin, start)
        host = slot.host_buffers()
        for b in host.values():
            b.zero_()
        slots.append((slot, fin, host))
    torch.cuda.synchronize()
    st = dict(slots=slots)
    for _ in range(2):                   # buffers sized, then the final graphs captured, as admission does
        _run_batch(st)
    return st


def _run_batch(st):
    for slot, fin, _ in st["slots"]:
        slot.submit(fin)
    out = []
    for slot, _, host in st["slots"]:
        counts = slot.finish()
        slot.fetch_async(host)
        out.append(dict(host, counts=list(counts)))
    return out


def _prepare_solve(case, seed):
    sets = _views(case, seed, rgb=False)[1]
    nx, ny, nz = _grid(case)
    ctx = _context(case, precision=PREC[case["prec"]])
    st = dict(ctx=ctx, sets=sets, A=torch.empty((nz, ny, nx), device=DEV))
    torch.cuda.synchronize()
    _run_solve(st)
    ctx.autotune()
    return st


def _run_solve(st):
    ctx = st["ctx"]
    ctx.reset()
    ctx.splat_sets(st["sets"])
    level = ctx.solve()
    ftr.ftr_get_field_A(ctx.h, st["A"])
    return dict(A=st["A"], level=level)


def _prepare_mesh(case, seed):
    A, level = _field(case, seed)
    st = dict(ctx=_context(case), A=A, level=level)
    torch.cuda.synchronize()
    st["mesh"] = _mesh_buffers(3 * _cap(_grid(case)))
    _run_mesh(st)
    return st


def _run_mesh(st):
    ftr.ftr_set_indicator(st["ctx"].h, st["A"], st["level"])
    return _mesh_out(st["ctx"], st["ctx"].extract_mesh(), st["mesh"])


def _prepare_texture(case, seed):
    views, sets = _views(case, seed)
    g, n, k = _gen(seed + 7), case["verts"], case["cams"]
    P = torch.cat([s[0] for s in sets])
    P = P[torch.randint(len(P), (n,), generator=g, device=DEV)] + 0.004 * torch.randn((n, 3), generator=g, device=DEV)
    cell = ((P + 2.0) * 64).long()       # mesh vertices come in grid order: z, then y, then x
    P = P[torch.argsort((cell[:, 2] * 512 + cell[:, 1]) * 512 + cell[:, 0])].contiguous()
    return dict(ctx=ftr.Context((32, 32, 32), CUBE), views=views, verts=P, tol=_tol((256,) * 3, CUBE),
                w=torch.empty((n, k), device=DEV), uv=torch.empty((n, k, 2), device=DEV),
                rgb=torch.empty((n, 3), dtype=torch.uint8, device=DEV),
                tex=torch.empty((n,), dtype=torch.uint8, device=DEV))


def _run_texture(st):
    ftr.ftr_texture_vertices(st["ctx"].h, st["views"], st["tol"], st["verts"], st["w"], st["uv"], st["rgb"], st["tex"])
    return dict(weights=st["w"], uv=st["uv"], rgb=st["rgb"], textured=st["tex"])


def _prepare_evaluate(case, seed):
    rng, g = np.random.default_rng(seed + 3), _gen(seed + 3)
    verts, tris, colour, radii = _surface(case, seed)
    w, h, rw, rh = case["dw"], case["dh"], case["rw"], case["rh"]
    views = []
    for K, RT, Kr, RTr in _cameras(case, rng, 2.5):
        R, t = _t(RT[:, :3]), _t(RT[:, 3])
        rays = _pixel_rays(K, w, h) @ R / radii
        o = (-(t @ R) - _t(CENTRE)) / radii                # the sensor's view of the smooth ellipsoid
        a, b, c = (rays * rays).sum(-1), rays @ o, o @ o - 1.0
        disc = b * b - a * c
        z = (-b - torch.sqrt(disc.clamp(min=0))) / a
        z = z + 0.0012 * z * z * torch.randn(z.shape, generator=g, device=DEV, dtype=torch.float64)
        views.append(dict(cam=ftr.make_camera(K, RT, w, h), rgb_cam=ftr.make_camera(Kr, RTr, rw, rh),
                          sensor=torch.where(disc > 0, z, 0.0).float().contiguous(), photo=_pattern(rng, rw, rh),
                          depth=torch.empty((h, w), device=DEV), rgb_depth=torch.empty((rh, rw), device=DEV),
                          rgb=torch.empty((rh, rw, 3), dtype=torch.uint8, device=DEV)))
    return dict(ctx=ftr.Context((32, 32, 32), CUBE), verts=verts, tris=tris, colour=colour, views=views)


def _run_evaluate(st):
    h, out = st["ctx"].h, []
    for v in st["views"]:
        ftr.ftr_render(h, st["verts"], st["tris"], v["cam"], v["depth"])
        geo = ftr.ftr_eval_geometry(h, v["cam"], v["depth"], v["sensor"])
        ftr.ftr_render(h, st["verts"], st["tris"], v["rgb_cam"], v["rgb_depth"], v["rgb"], vertex_rgb=st["colour"])
        app = ftr.ftr_eval_appearance(h, v["rgb_depth"], v["rgb"], v["photo"])
        out.append(dict(depth=v["depth"], rgb_depth=v["rgb_depth"], rgb=v["rgb"], geometry=geo, appearance=app))
    return out


def _prepare_level(case, seed):
    A, _ = _field(dict(case, blobs=12), seed)
    g, box = _gen(seed + 5), _box(case)
    lo, hi = torch.tensor(box[:3], device=DEV), torch.tensor(box[3:], device=DEV)
    n = case["points"]                   # samples of a closed surface in scan order, a few voxels thick
    th = torch.acos(1 - 2 * (torch.arange(n, device=DEV) + 0.5) / n)
    ph = 2 * math.pi * torch.rand((n,), generator=g, device=DEV)
    d = torch.stack([torch.sin(th) * torch.cos(ph), torch.cos(th), torch.sin(th) * torch.sin(ph)], 1)
    P = (lo + hi) / 2 + (hi - lo) * (0.35 + 0.01 * torch.randn((n, 1), generator=g, device=DEV)) * d
    st = dict(A=A, grid=_grid(case), box=box, P=P.contiguous())
    torch.cuda.synchronize()
    _run_level(st)                       # the first call of a process looks up the scratch array
    return st


def _run_level(st):
    return ftr.ftr_iso_level_noalloc(st["A"], st["grid"], st["box"], st["P"])


_PREPARE = dict(points=_prepare_points, frame=_prepare_frame, rgbd=_prepare_frame, batch=_prepare_batch,
                solve=_prepare_solve, mesh=_prepare_mesh, texture=_prepare_texture, evaluate=_prepare_evaluate,
                level=_prepare_level)
_RUN = dict(points=_run_points, frame=_run_frame, rgbd=_run_frame, batch=_run_batch, solve=_run_solve, mesh=_run_mesh,
            texture=_run_texture, evaluate=_run_evaluate, level=_run_level)


# ------------------------------------------------------------------ the work

def work(case):
    """Bytes of the inputs read once and the outputs written once, and the
    operations of the transforms (5/2 M log2 M per real transform of M nodes,
    four of them), the splat and the metrics."""
    kind = case["kind"]

    def solve(nx, ny, nz, pts):
        m = nx * ny * nz
        return 10.0 * m * math.log2(m) + 64.0 * 20 * pts

    def surface(nx, ny, nz):             # vertices of a body about as wide as the box
        return 0.65 * (nx * ny * nz) ** (2.0 / 3.0)
    px = case.get("dw", 0) * case.get("dh", 0)
    if kind in ("points", "solve", "frame", "rgbd", "batch"):
        if kind == "batch":
            grids = [(int(v),) * 3 for v in case["grids"].split(",")]
        else:
            grids = [_grid(case)]
        total = dict(bytes=0.0, flops=0.0)
        for g in grids:
            k = case.get("cams", 0)
            pts = case["points"] if case.get("source") == "sphere" else 0.055 * px * k
            nv = surface(*g)
            mesh = nv * (24 + 24)
            if kind == "solve":
                mesh = 4.0 * g[0] * g[1] * g[2]
            b = 28.0 * pts + mesh
            if kind in ("frame", "rgbd", "batch"):
                b += nv * (12 * k + 4) + nv * k * 20          # texture data out, the pixels it samples in
            if kind == "rgbd":
                b += 8.0 * px * k - 28.0 * pts
            if kind == "batch":
                b += k * (8.0 * px + 3 * 1920 * 1080)         # the views cross from host memory whole
            total["bytes"] += b
            total["flops"] += solve(*g, pts)
        return total
    if kind == "mesh":
        nx, ny, nz = _grid(case)
        return dict(bytes=4.0 * nx * ny * nz + 48.0 * case["blobs"] * 20 * (0.08 * max(nx, ny, nz)) ** 2, flops=1.0 * nx * ny * nz)
    if kind == "texture":
        n, k = case["verts"], case["cams"]
        return dict(bytes=n * (12.0 + k * 12 + 4 + k * 20), flops=n * k * 80.0)
    if kind == "evaluate":
        rpx, mesh = case["rw"] * case["rh"], case["nu"] * case["nv"] * (15.0 + 24)
        return dict(bytes=case["cams"] * (2 * mesh + 8.0 * px + 10.0 * rpx), flops=case["cams"] * (484.0 * rpx + 8 * (0.13 * px) ** 2))
    return dict(bytes=case["points"] * (12.0 + 32), flops=case["points"] * 20.0)


# ------------------------------------------------------------------ 64 bits

def exact(case, seed):
    """What run() returns, from plain torch in float64 (None where that does not exist)."""
    kind = case["kind"]
    if kind == "points":
        sets = [_sphere(case, seed)] if case["source"] == "sphere" else _views(case, seed, rgb=False)[1]
        A, level = _exact_solve(case, sets, case["simple"])
        return dict(_exact_mesh(A, level, _box(case), _cap(_grid(case))), level=level)
    if kind == "solve":
        A, level = _exact_solve(case, _views(case, seed, rgb=False)[1], False)
        return dict(A=A, level=level)
    if kind == "frame":
        return _exact_mesh(*_exact_solve(case, _views(case, seed, rgb=False)[1], False), _box(case),
                           _cap(_grid(case)))
    if kind == "rgbd":
        views = _views(case, seed, rgb=False)[0]
        return dict(conf=[_raw(v["depth"], v["K"], v["world_to_cam"])[3] for v in views])
    if kind == "mesh":
        A, level = _field(case, seed)
        return _exact_mesh(A.double(), level, _box(case), 3 * _cap(_grid(case)))
    if kind == "texture":
        st = _prepare_texture(case, seed)
        return _exact_texture(st["views"], st["verts"], st["tol"])
    if kind == "level":
        st = _prepare_level(case, seed)
        return _exact_level(st["A"].double(), *_nodes(case, st["P"].double()))
    return None


def _nodes(case, P):
    """floor(t), t - floor(t) of the accepted points, t = (X - b_min) / h - 1/2, and the mask of accepted points."""
    n = _t(_grid(case))
    box = _t(np.array(_box(case), np.float32))
    t = (P - box[:3]) / ((box[3:] - box[:3]) / n) - 0.5
    ok = ((t >= 1) & (t < n - 2)).all(1)
    b = t[ok].floor()
    return b.long(), t[ok] - b, ok


def _exact_level(A, b, f, ok):
    total = torch.zeros(len(b), dtype=torch.float64, device=DEV)
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                w = 1.0
                for a, d in enumerate((dx, dy, dz)):
                    w = w * (f[:, a] if d else 1 - f[:, a])
                total += w * A[b[:, 2] + dz, b[:, 1] + dy, b[:, 0] + dx]
    return float(total.mean()) if len(b) else 0.0


def _exact_solve(case, sets, simple):
    nx, ny, nz = n = _grid(case)
    box = _t(np.array(_box(case), np.float32))
    h = (box[3:] - box[:3]) / _t(n)
    P, N, W = (torch.cat([s[a] for s in sets]).double() for a in range(3))
    b, f, ok = _nodes(case, P)
    N, W = N[ok], W[ok]
    acc = torch.zeros((4, nz * ny * nx), dtype=torch.float64, device=DEV)
    s1 = float((h * h).sum()) * 0.25                                     # sigma1^2, sigma2^2 = 1.5 sigma1^2
    steps = [(0, 0, 0)] if simple else [(x, y, z) for z in range(-1, 3) for y in range(-1, 3) for x in range(-1, 3)]
    for step in steps:
        o = _t(step)
        q = b + o.long() if not simple else b + (f >= 0.5).long()
        i = (q[:, 2] * ny + q[:, 1]) * nx + q[:, 0]
        r2 = (((f - o) * h) ** 2).sum(1)
        g1 = torch.ones_like(r2) if simple else torch.exp(-r2 / s1) * W
        g2 = torch.ones_like(r2) if simple else torch.exp(-r2 / (1.5 * s1)) * W
        for a in range(3):
            acc[a].index_add_(0, i, g1 * N[:, a])
        acc[3].index_add_(0, i, g2)
    scale = 1.0 if simple else math.sqrt(1.5)
    total, w2 = None, 0.0
    for a in range(3):
        V = torch.where(acc[3] > 0, scale * acc[a] / acc[3].clamp(min=1e-300), 0.0).reshape(nz, ny, nx)
        S = torch.fft.rfftn(V)
        del V
        m = n[a]
        k = torch.fft.fftfreq(m, 1.0 / m, dtype=torch.float64, device=DEV)
        w = 2 * math.pi * k / (m * float(h[a]))
        num = torch.where(k.abs() == m // 2, 0.0, w)
        if a == 0:
            num, w = num[: nx // 2 + 1], w[: nx // 2 + 1]
        shape = [(1, 1, -1), (1, -1, 1), (-1, 1, 1)][a]
        S *= 1j * num.reshape(shape)
        total = S if total is None else total.add_(S)
        w2 = w2 + (w * w).reshape(shape)
        del S
    w2[0, 0, 0] = 1.0
    total /= w2
    total[0, 0, 0] = 0
    A = torch.fft.irfftn(total, s=(nz, ny, nx))
    return A, _exact_level(A, b, f, ok)


def _exact_mesh(A, level, box, cap):
    """Vertices in (node, axis) order and their normals, float64, in buffers of ``cap``."""
    n = (A.shape[2], A.shape[1], A.shape[0])
    box = _t(np.array(box, np.float32))
    h = (box[3:] - box[:3]) / _t(n)
    inside = A >= level
    cross = torch.zeros((*A.shape, 3), dtype=torch.bool, device=DEV)
    cross[:, :, :-1, 0] = inside[:, :, 1:] != inside[:, :, :-1]
    cross[:, :-1, :, 1] = inside[:, 1:] != inside[:, :-1]
    cross[:-1, :, :, 2] = inside[1:] != inside[:-1]
    z, y, x, a = cross.nonzero(as_tuple=True)
    q0 = torch.stack([x, y, z], 1)
    q1 = q0 + torch.nn.functional.one_hot(a, 3)

    def at(q):
        return A[q[:, 2], q[:, 1], q[:, 0]]

    def grad(q):
        out = []
        for c in range(3):
            e = torch.zeros(3, dtype=torch.long, device=DEV)
            e[c] = 1
            hi, lo = torch.minimum(q[:, c] + 1, torch.full_like(x, n[c] - 1)), torch.maximum(q[:, c] - 1, torch.zeros_like(x))
            qh, ql = q.clone(), q.clone()
            qh[:, c], ql[:, c] = hi, lo
            out.append((at(qh) - at(ql)) / ((hi - lo) * h[c]))
        return torch.stack(out, 1)
    t = ((level - at(q0)) / (at(q1) - at(q0)))[:, None]
    nrm = -((1 - t) * grad(q0) + t * grad(q1))
    room = (0, 0, 0, cap - len(t))
    return dict(vertices=torch.nn.functional.pad(box[:3] + (q0 + t * (q1 - q0) + 0.5) * h, room),
                normals=torch.nn.functional.pad(nrm / nrm.norm(dim=1, keepdim=True), room), tris=None, counts=None)


def _exact_texture(views, verts, tol):
    X, ws, uvs = verts.double(), [], []

    def project(K, RT):
        c = X @ _t(RT[:, :3]).T + _t(RT[:, 3])
        K = K.astype(np.float64)
        return K[0, 0] * c[:, 0] / c[:, 2] + K[0, 2], K[1, 1] * c[:, 1] / c[:, 2] + K[1, 2], c[:, 2]
    for v in views:
        h, w = v["depth"].shape
        u, y, z = project(v["K"], v["world_to_cam"])
        pu, py = torch.floor(u + 0.5), torch.floor(y + 0.5)
        ok = (z > 0) & (pu >= 0) & (pu < w) & (py >= 0) & (py < h)
        i = torch.where(ok, py * w + pu, 0.0).long()
        D = v["depth"].reshape(-1)[i].double()
        wk = torch.where(ok & (D > 0) & ((D - z).abs() <= tol), v["conf"].reshape(-1)[i].double(), 0.0)
        ur, vr, zr = project(v["K_rgb"], v["world_to_rgb"])
        rh, rw = v["rgb"].shape[:2]
        wk = torch.where((zr > 0) & (ur >= 0) & (ur <= rw - 1) & (vr >= 0) & (vr <= rh - 1), wk, 0.0)
        ws.append(wk)
        uvs.append(torch.where((wk > 0)[:, None], torch.stack([ur, vr], 1), -1.0))
    return dict(weights=torch.stack(ws, 1), uv=torch.stack(uvs, 1), rgb=None, textured=None)
