"""The work a user of this library has it do, as measurable cases.

Each case goes through the public autograd entry points (``rasterize_meshes``,
``render_meshes``, ``blend``, ``shade``, ``render_points``, ``knn_points``,
``chamfer_distance``) on seeded synthetic batches of the kind
``workloads.py`` describes.  ``exact`` evaluates the same maths in plain
PyTorch FP64: candidates enumerated face by face over their boxes, a sort per
pixel, autograd for the gradients.
"""
import math

import numpy as np
import torch

from paper_2007_08501_gb300 import autograd as ag
from paper_2007_08501_gb300 import ops, tune, workloads

DEV = "cuda"
BLUR = workloads.BLUR_SIGMA_1E4
SIGMA = GAMMA = 1e-4
MESH_CALLS = ("fragments", "render", "blend", "shade")


def _mesh(name, call, n, low, high, size, K, **kw):
    c = dict(call=call, n=n, low=low, high=high, level_seed=0, noise=0.05, size=size, K=K, blur=True, clip=True,
             persp=True, rgb=False, bin=16, views=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small mesh looked up at thumbnail size, the unbinned form: the smallest call, launch latency
        _mesh("plain_64px_k1", "fragments", 1, 3, 3, 64, 1, blur=False, clip=False, bin=0),
        # the paper's homogeneous training batch: soft colours and silhouettes, forward and backward
        _mesh("rgb_8x5k_256px_k8", "render", 8, 4, 4, 256, 8, rgb=True),
        # the heterogeneous training batch: meshes of 1.3k to 328k faces, soft silhouettes
        _mesh("mixed_32_512px_k4", "render", 32, 3, 7, 512, 4, level_seed=2999, noise=0.03),
        # one scanned-size mesh at full resolution, soft
        _mesh("scan_1m_1024px_k8", "render", 1, 8, 8, 1024, 8, noise=0.02),
        # one scanned-size mesh for a depth map: hard coverage, nearest face only, no gradient
        _mesh("depth_1m_1024px_k1", "fragments", 1, 8, 8, 1024, 1, noise=0.02, blur=False, clip=False),
        # analysis by synthesis: one mesh from 20 cameras, 50 faces a pixel, the largest training step
        _mesh("views_20_512px_k50", "render", 20, 6, 6, 512, 50, noise=0.02, views=True),
        # odd sizes, the stages called one by one (rasterize, then blend), colours
        _mesh("odd_5_225px_k5", "blend", 5, 2, 6, 225, 5, level_seed=7, rgb=True, noise=0.03),
        # Phong-lit training batch: fragments, reflection model, gradients to positions, normals, colours
        _mesh("phong_8x5k_256px_k8", "shade", 8, 4, 4, 256, 8),
        # the point renderer's silhouette benchmark
        dict(name="points_8x200k_k50", call="points", n=8, count=200_000, spread=0, size=256, K=50, radius=0.01, D=1,
             norm=False, bin=8),
        # a small coloured point batch of uneven clouds
        dict(name="points_3_100px_k10", call="points", n=3, count=9_000, spread=6_000, size=100, K=10, radius=0.03,
             D=3, norm=True, bin=16),
        # nearest neighbours between uneven clouds, with gradients
        dict(name="knn_32_k8", call="knn", n=32, count=50_000, spread=40_000, other=50_000, K=8, grad=True),
        # the Chamfer training loss of a predicted cloud against a dense target
        dict(name="chamfer_32_1k_50k", call="chamfer", n=32, count=1_000, spread=0, other=50_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["fragments", "render", "render", "render", "blend", "shade", "points", "knn", "chamfer"])
    while True:
        n = _log(rng, 1, 32)
        if call in MESH_CALLS:
            high = rng.randint(2, 7)
            low = rng.randint(2, high)
            size = _log(rng, 48, 1024)
            K = rng.choice([1, 2, 3, 4, 5, 8, 8, 10, 16, 24, 50])
            rgb = call == "blend" or (call == "render" and rng.random() < 0.5)
            plain = call == "fragments" and rng.random() < 0.3
            blur = K > 1 or rng.random() < 0.5
            c = _mesh(None, call, n, low, high, size, K, level_seed=rng.randrange(1 << 20),
                      noise=rng.choice([0.01, 0.03, 0.05]), rgb=rgb, blur=blur, clip=blur,
                      persp=rng.random() < 0.8, bin=0 if plain else rng.choice([8, 16, 16]),
                      views=n > 1 and rng.random() < 0.2)
            slots = n * size * size * K
            faces = sum(20 * 4 ** int(v) for v in _levels(c))
            heavy = 8_000_000 if call in ("blend", "shade") or rgb else 60_000_000
            if plain and (n > 4 or size > 160 or high > 4):
                continue
            if slots > heavy or faces > 1_400_000:
                continue
            return c
        if call == "points":
            count = _log(rng, 500, 200_000)
            size = _log(rng, 48, 512)
            K = rng.choice([1, 3, 8, 10, 16, 32, 50])
            D = rng.choice([1, 1, 3, 4])
            if n * count > 1_600_000 or n * size * size * K > 26_000_000:
                continue
            return dict(call="points", n=n, count=count, spread=count // 2 if rng.random() < 0.5 else 0, size=size,
                        K=K, radius=rng.choice([0.01, 0.02, 0.03]), D=D, norm=D > 1 and rng.random() < 0.5,
                        bin=rng.choice([8, 16]))
        count, other = _log(rng, 200, 60_000), _log(rng, 200, 60_000)
        if n * count * other > 40_000_000_000:
            continue
        spread = count // 2 if rng.random() < 0.5 else 0
        if call == "chamfer":
            return dict(call="chamfer", n=n, count=count, spread=spread, other=other)
        return dict(call="knn", n=n, count=count, spread=spread, other=other, K=rng.choice([1, 2, 4, 5, 8, 8, 16, 20]),
                    grad=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _levels(case):
    rng = np.random.default_rng(case["level_seed"])
    lv = [int(x) for x in rng.integers(case["low"], case["high"] + 1, size=case["n"])]
    return [lv[0]] * case["n"] if case["views"] else lv


def _sizes(case, which):
    """Points per cloud: uniform in count +- spread, by the case alone."""
    mid, spread = (case["count"], case["spread"]) if which == 0 else (case["other"], 0)
    if which == 1 and case["spread"]:
        spread = case["other"] * case["spread"] // max(1, case["count"])
    rng = np.random.default_rng(100 + which)
    return rng.integers(max(1, mid - spread), mid + spread + 1, size=case["n"])


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _mesh_inputs(case, seed):
    levels, base = _levels(case), int(seed) * 4096
    if case["views"]:
        # several cameras on one mesh: every image's faces index the same vertices
        v, f = workloads.displaced_sphere(levels[0], case["noise"], np.random.default_rng(base))
        rng = np.random.default_rng(base + 1)
        n, F0 = case["n"], f.shape[0]
        b = workloads.pack([(v, f)], [workloads.random_camera(rng)])
        b.faces = np.tile(f.astype(np.int64), (n, 1))
        b.first_face = np.arange(n, dtype=np.int64) * F0
        b.num_faces = np.full(n, F0, np.int64)
        b.cams = np.stack([workloads.look_at_camera(2.7, float(rng.uniform(-30, 30)), 360.0 * i / n)
                           for i in range(n)]).astype(np.float32)
        b.colors = rng.uniform(0.0, 1.0, size=b.verts.shape).astype(np.float32)
    else:
        b = workloads.sphere_batch(levels, case["noise"], base)
    nrm = b.verts / np.maximum(np.linalg.norm(b.verts, axis=1, keepdims=True), 1e-6)
    s = dict(verts=_gpu(b.verts), faces=_gpu(b.faces), ff=_gpu(b.first_face), nf=_gpu(b.num_faces),
             cams=_gpu(b.cams), colors=_gpu(b.colors), normals=_gpu(nrm))
    if case["call"] != "fragments":
        gen = torch.Generator(device=DEV).manual_seed(int(seed) + 17)
        s["grad"] = torch.randn((case["n"], case["size"], case["size"], 4), device=DEV, generator=gen)
    return s


def _raster_settings(case, s):
    """Bins sized the way the tuner sizes them: the occupancy of one forward, with headroom."""
    kw = dict(image_size=case["size"], faces_per_pixel=case["K"], blur_radius=BLUR if case["blur"] else 0.0,
              bin_size=case["bin"], perspective_correct=case["persp"], clip_barycentric_coords=case["clip"])
    if case["bin"] == 0:
        return ag.RasterSettings(**kw)
    n, F, V = case["n"], s["faces"].shape[0], s["verts"].shape[0]
    nb = -(-case["size"] // case["bin"])
    cap = max(256, min(F, 1 << 20))
    entries = min(n * nb * nb * cap, max(1 << 20, 64 * F))
    p = ops.make_rast_params(n, case["size"], 1, kw["blur_radius"], case["bin"], cap, case["persp"], case["clip"],
                             entries)
    ws = ops.alloc_workspace(p, V, F, DEV)
    ops.rast_mesh_fwd(p, s["verts"], s["faces"], s["ff"], s["nf"], s["cams"],
                      *ops.alloc_fragments(n, case["size"], 1, DEV), ws)
    per_bin, entries = tune.capacities(*ops.rast_bin_occupancy(p, V, F, ws))
    return ag.RasterSettings(max_faces_per_bin=per_bin, max_bin_entries=entries, **kw)


def _point_settings(case, s):
    n, P = case["n"], s["points"].shape[0]
    nb = -(-case["size"] // case["bin"])
    cap = max(256, min(P, 1 << 20))
    p = ops.make_pts_params(n, case["size"], 1, case["radius"], case["bin"], cap, min(n * nb * nb * cap, 16 * P + 4096))
    ws = torch.empty(ops.pts_workspace_bytes(p, P), dtype=torch.uint8, device=DEV)
    ops.pts_rasterize_fwd(p, s["points"], s["first"], s["num"], s["cams"],
                          *ops.alloc_pts_fragments(n, case["size"], 1, DEV), ws)
    per_bin, entries = tune.capacities(*ops.pts_bin_occupancy(p, P, ws))
    return ag.PointSettings(case["size"], case["K"], case["radius"], bin_size=case["bin"], max_points_per_bin=per_bin,
                            max_bin_entries=entries, mode=ops.PTS_NORM if case["norm"] else ops.PTS_ALPHA)


def _points_inputs(case, seed):
    b = workloads.point_batch(_sizes(case, 0), int(seed) * 4096, level=4, sigma=0.05, D=case["D"])
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 17)
    S = case["size"]
    return dict(points=_gpu(b.points), first=_gpu(b.first_point), num=_gpu(b.num_points), cams=_gpu(b.cams),
                feats=_gpu(b.features), grad=torch.randn((case["n"], S, S, case["D"]), device=DEV, generator=gen))


def _cloud_inputs(case, seed):
    """Clouds sampled from displaced spheres; candidates and queries from different spheres."""
    rng = np.random.default_rng(int(seed))
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 17)
    s = {}
    for which, key in ((0, "p"), (1, "q")):
        num = _sizes(case, which)
        first = np.concatenate([[0], np.cumsum(num)[:-1]]).astype(np.int64)
        pts = []
        for m in num:
            v, f = workloads.displaced_sphere(4, 0.05, rng)
            tri = _gpu(v.astype(np.float32))[_gpu(f)]
            area = torch.linalg.norm(torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]), dim=1)
            pick = tri[torch.multinomial(area, int(m), replacement=True, generator=gen)]
            u = torch.rand((int(m), 2, 1), device=DEV, generator=gen)
            u = torch.where(u.sum(1, keepdim=True) > 1, 1 - u, u)
            pts.append(pick[:, 0] + u[:, 0] * (pick[:, 1] - pick[:, 0]) + u[:, 1] * (pick[:, 2] - pick[:, 0]))
        s[key] = torch.cat(pts).contiguous()
        s["first_" + key], s["len_" + key] = _gpu(first), _gpu(num.astype(np.int64))
    if case["call"] == "knn":
        s["grad"] = torch.randn((s["p"].shape[0], case["K"]), device=DEV, generator=gen)
    return s


def prepare(case, seed):
    call = case["call"]
    if call in MESH_CALLS:
        s = _mesh_inputs(case, seed)
        s["rs"] = _raster_settings(case, s)
        s["bs"] = ag.BlendSettings(sigma=SIGMA, gamma=GAMMA, rgb=case["rgb"])
        s["ws"] = ag.Workspace(DEV)
        s["light"] = ag.ShadeSettings()
        if call != "fragments":
            s["leaves"] = [s["verts"].requires_grad_(True)]
            if case["rgb"] or call == "shade":
                s["leaves"].append(s["colors"].requires_grad_(True))
            if call == "shade":
                s["leaves"].append(s["normals"].requires_grad_(True))
    elif call == "points":
        s = _points_inputs(case, seed)
        s["ps"] = _point_settings(case, s)
        s["ws"] = ag.Workspace(DEV)
        s["leaves"] = [s["points"].requires_grad_(True), s["feats"].requires_grad_(True)]
    else:
        s = _cloud_inputs(case, seed)
        if call == "chamfer" or case["grad"]:
            s["leaves"] = [s["p"].requires_grad_(True), s["q"].requires_grad_(True)]
    s["case"] = dict(case)
    return s


def run(s):
    case = s["case"]
    call = case["call"]
    if call in MESH_CALLS:
        mesh = (s["verts"], s["faces"], s["ff"], s["nf"], s["cams"])
        if call == "render":
            img = ag.render_meshes(*mesh, s["rs"], s["bs"], colors=s["colors"] if case["rgb"] else None, ws=s["ws"])
        else:
            frags = ag.rasterize_meshes(*mesh, s["rs"], s["ws"])
            if call == "fragments":
                return list(frags)
            if call == "blend":
                img = ag.blend(*frags, s["faces"], s["colors"], s["bs"])
            else:
                img = ag.shade(*frags, s["verts"], s["normals"], s["colors"], s["faces"], s["cams"], s["bs"],
                               s["light"])
        return [img, *torch.autograd.grad(img, s["leaves"], s["grad"])]
    if call == "points":
        img = ag.render_points(s["points"], s["feats"], s["first"], s["num"], s["cams"], s["ps"], s["ws"])
        return [img, *torch.autograd.grad(img, s["leaves"], s["grad"])]
    clouds = (s["p"], s["first_p"], s["len_p"], s["q"], s["first_q"], s["len_q"])
    if call == "knn":
        dists, idx = ag.knn_points(*clouds, case["K"])
        return [dists, idx, *(torch.autograd.grad(dists, s["leaves"], s["grad"]) if case["grad"] else ())]
    loss, per = ag.chamfer_distance(*clouds)
    return [loss, per, *torch.autograd.grad(loss, s["leaves"])]


def work(case):
    """Inputs read once, outputs written once; operations: one evaluation per output slot."""
    call, n = case["call"], case["n"]
    if call in MESH_CALLS:
        lv = _levels(case)
        F = sum(20 * 4 ** v for v in lv)
        V = sum(10 * 4 ** v + 2 for v in (lv[:1] if case["views"] else lv))
        pix = n * case["size"] ** 2
        slots = pix * case["K"]
        if call == "fragments":
            return {"bytes": 12 * V + 24 * F + 28 * slots, "flops": 60 * slots}
        attrs = 1 + int(case["rgb"] or call == "shade") + int(call == "shade")
        return {"bytes": 24 * V * attrs + 24 * F + 32 * pix, "flops": 200 * slots}
    if call == "points":
        P, pix = int(_sizes(case, 0).sum()), n * case["size"] ** 2
        return {"bytes": P * 8 * (3 + case["D"]) + 8 * case["D"] * pix, "flops": 30 * pix * case["K"]}
    P, Q = int(_sizes(case, 0).sum()), int(_sizes(case, 1).sum())
    if call == "knn":
        b = 12 * (P + Q) + 12 * P * case["K"]
        return {"bytes": 2 * b if case["grad"] else b, "flops": 8 * P * case["K"]}
    return {"bytes": 24 * (P + Q), "flops": 16 * (P + Q)}


# ---------------------------------------------------------------------------
# the same results in FP64
# ---------------------------------------------------------------------------
def _f32(x):
    return float(np.float32(x))


def _project(x, cam):
    d = x - cam[9:12]
    v = d @ cam[:9].reshape(3, 3).T
    return cam[12] * v[:, :2] / v[:, 2:], v[:, 2]


def _centres(i, S):
    return 1.0 - (2.0 * i.double() + 1.0) / S


def _cross(a, b):
    return a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]


def _evaluate(P, Z, px, persp, clip):
    """P (M,3,2) NDC corners, Z (M,3) depths, px (M,2): barycentrics, depth, signed squared distance, raw inside."""
    u, w, q = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0], px - P[:, 0]
    A = _cross(u, w)
    b1, b2 = _cross(q, w) / A, _cross(u, q) / A
    b = torch.stack([1 - b1 - b2, b1, b2], 1)
    inside = (b >= 0).all(1)
    best = None
    for i in range(3):
        a, e = P[:, i], P[:, (i + 1) % 3] - P[:, i]
        with torch.no_grad():
            t = (((px - a) * e).sum(1) / (e * e).sum(1).clamp_min(1e-300)).clamp(0, 1)
        r = px - a - t[:, None] * e
        d = (r * r).sum(1)
        best = d if best is None else torch.minimum(best, d)
    if persp:
        t = b / Z
        b = t / t.sum(1, keepdim=True)
    if clip:
        c = torch.where(inside[:, None], b, b.clamp_min(0))
        b = c / c.sum(1, keepdim=True)
    return b, (b * Z).sum(1), torch.where(inside, -best, best), inside


def _rank(pix, z, ids, K, pixels):
    """(pixels, K) ids of the K smallest (z, id) per pixel, -1 where there are fewer."""
    out = torch.full((pixels, K), -1, dtype=torch.int64, device=DEV)
    if pix.numel() == 0:
        return out
    o = torch.argsort(z, stable=True)   # candidates come in ascending id order
    o = o[torch.argsort(pix[o], stable=True)]
    ps = pix[o]
    rank = torch.arange(ps.numel(), device=DEV) - torch.searchsorted(ps, ps)
    keep = rank < K
    out[ps[keep], rank[keep]] = ids[o][keep]
    return out


def _candidates(lo, hi, S, row0, row1, fn):
    """Pairs (box, pixel) of rows [row0, row1), a part at a time: fn(box ids, rows, columns) -> kept pixels, depths, ids."""
    c0 = torch.ceil(((1 - hi[:, 0]) * S - 1) / 2).clamp(0, S).long()
    c1 = torch.floor(((1 - lo[:, 0]) * S - 1) / 2).clamp(-1, S - 1).long()
    r0 = torch.ceil(((1 - hi[:, 1]) * S - 1) / 2).clamp(row0, row1).long()
    r1 = torch.floor(((1 - lo[:, 1]) * S - 1) / 2).clamp(row0 - 1, row1 - 1).long()
    wide = (c1 - c0 + 1).clamp_min(0)
    cnt = wide * (r1 - r0 + 1).clamp_min(0)
    which = torch.nonzero(cnt).squeeze(1)
    got = []
    ends = torch.cumsum(cnt[which], 0)
    at, done = 0, 0
    while at < which.numel():
        to = max(at + 1, int(torch.searchsorted(ends, done + (1 << 24), right=True)))
        sel = which[at:to]
        ids = torch.repeat_interleave(sel, cnt[sel])
        k = torch.arange(ids.numel(), device=DEV) - torch.repeat_interleave(ends[at:to] - cnt[sel] - done, cnt[sel])
        got.append(fn(ids, r0[ids] + k // wide[ids], c0[ids] + k % wide[ids]))
        done, at = int(ends[to - 1]), to
    if not got:
        e = torch.zeros(0, dtype=torch.int64, device=DEV)
        return e, e.double(), e
    return tuple(torch.cat(x) for x in zip(*got))


def _select_faces(case, xy, z, tri, cam):
    """(S*S, K) local face ids of one image."""
    S, K = case["size"], case["K"]
    blur = _f32(BLUR) if case["blur"] else 0.0
    P, Z = xy[tri], z[tri]
    A = _cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
    ok = torch.nonzero((Z >= cam[13]).all(1) & (A.abs() >= 1e-12)).squeeze(1)
    P, Z = P[ok], Z[ok]
    r = math.sqrt(blur)
    lo, hi = P.amin(1) - r, P.amax(1) + r

    def test(i, row, col):
        px = torch.stack([_centres(col, S), _centres(row, S)], 1)
        _, depth, d, inside = _evaluate(P[i], Z[i], px, case["persp"], case["clip"])
        keep = (inside | (d < blur)) & (depth >= cam[13]) & torch.isfinite(depth)
        return (row * S + col)[keep], depth[keep], ok[i[keep]]

    strips = max(1, min(S, (S * S * P.shape[0]) // (1 << 36)))
    out = []
    for k in range(strips):
        a, b = S * k // strips, S * (k + 1) // strips
        pix, depth, ids = _candidates(lo, hi, S, a, b, test)
        out.append(_rank(pix - a * S, depth, ids, K, (b - a) * S))
    return torch.cat(out)


def _softmax_blend(z, d, col, live, bg):
    zfar, znear, eps = 100.0, _f32(0.1), _f32(1e-10)
    sigma, gamma = _f32(SIGMA), _f32(GAMMA)
    prob = torch.where(live, torch.sigmoid(-d / sigma), 0.0)
    zinv = torch.where(live, (zfar - z) / (zfar - znear), 0.0)
    m = torch.where(live, zinv, -math.inf).amax(1).clamp_min(eps).detach()
    w = torch.where(live, prob * torch.exp((zinv - m[:, None]) / gamma), 0.0)
    delta = torch.exp((eps - m) / gamma)
    return ((w[:, :, None] * col).sum(1) + delta[:, None] * bg) / (w.sum(1) + delta)[:, None]


def _phong(x, nrm, a, eye):
    s = ag.ShadeSettings()
    T = lambda v: torch.tensor([_f32(t) for t in v], dtype=torch.float64, device=DEV)  # noqa: E731
    unit = lambda v: v / torch.linalg.norm(v, dim=-1, keepdim=True)  # noqa: E731
    m, l, v = unit(nrm), unit(T(s.light) - x), unit(eye - x)
    c = (m * l).sum(-1, keepdim=True)
    sv = ((2 * c * m - l) * v).sum(-1, keepdim=True)
    on = (c > 0) & (sv > 0)
    shine = torch.where(on, torch.where(on, sv, 1.0) ** s.shininess, 0.0)
    return a * (T(s.ambient) + T(s.diffuse) * c.clamp_min(0)) + T(s.specular) * shine


def _exact_mesh(case, seed):
    s = _mesh_inputs(case, seed)
    S, K, call = case["size"], case["K"], case["call"]
    leaves = [s[k].detach().double().requires_grad_(call != "fragments") for k in ("verts", "colors", "normals")]
    verts, colors, normals = leaves
    cams, bg = s["cams"].double(), torch.ones(3, dtype=torch.float64, device=DEV)
    used = 3 if call == "shade" else 2 if case["rgb"] else 1
    outs, grads = [], [torch.zeros_like(v) for v in leaves[:used]]
    for n in range(case["n"]):
        tri = s["faces"][int(s["ff"][n]):int(s["ff"][n]) + int(s["nf"][n])]
        xy, z = _project(verts, cams[n])
        with torch.no_grad():
            ids = _select_faces(case, xy.detach(), z.detach(), tri, cams[n])
        live = ids >= 0
        pix, slot = torch.nonzero(live, as_tuple=True)
        f = tri[ids[pix, slot]]
        px = torch.stack([_centres(pix % S, S), _centres(pix // S, S)], 1)
        b, depth, d, _ = _evaluate(xy[f], z[f], px, case["persp"], case["clip"])
        fill = lambda v, e: torch.full((S * S, K) + v.shape[1:], e, dtype=torch.float64,  # noqa: E731
                                       device=DEV).index_put((pix, slot), v)
        if call == "fragments":
            outs.append([fill(depth, -1.0).view(S, S, K), fill(b, -1.0).view(S, S, K, 3), fill(d, -1.0).view(S, S, K)])
            continue
        dd = fill(d, 0.0)
        log_keep = torch.where(live, torch.nn.functional.logsigmoid(dd / _f32(SIGMA)), 0.0).sum(1)
        alpha = -torch.expm1(log_keep)
        if call == "shade" or case["rgb"]:
            mix = lambda v: (b[:, :, None] * v[f]).sum(1)  # noqa: E731
            c = _phong(mix(verts), mix(normals), mix(colors), cams[n, 9:12]) if call == "shade" else mix(colors)
            rgb = _softmax_blend(fill(depth, 0.0), dd, fill(c, 0.0), live, bg)
        else:
            rgb = torch.zeros((S * S, 3), dtype=torch.float64, device=DEV)
        img = torch.cat([rgb, alpha[:, None]], 1)
        got = torch.autograd.grad(img, leaves[:used], s["grad"][n].double().view(S * S, 4), allow_unused=True)
        for t, g in zip(grads, got):
            if g is not None:
                t += g
        outs.append(img.detach().view(S, S, 4))
    if call == "fragments":
        return [None] + [torch.stack(x) for x in zip(*outs)]
    return [torch.stack(outs), *grads]


def _exact_points(case, seed):
    s = _points_inputs(case, seed)
    S, K, D = case["size"], case["K"], case["D"]
    pts, feats = (s[k].detach().double().requires_grad_(True) for k in ("points", "feats"))
    cams = s["cams"].double()
    r2 = float(np.float32(case["radius"]) * np.float32(case["radius"]))
    outs, grads = [], [torch.zeros_like(pts), torch.zeros_like(feats)]
    for n in range(case["n"]):
        at, m = int(s["first"][n]), int(s["num"][n])
        xy, z = _project(pts[at:at + m], cams[n])
        with torch.no_grad():
            ok = torch.nonzero(z >= cams[n, 13]).squeeze(1)
            c, zc = xy.detach()[ok], z.detach()[ok]

            def test(i, row, col):
                px = torch.stack([_centres(col, S), _centres(row, S)], 1)
                keep = ((px - c[i]) ** 2).sum(1) < r2
                return (row * S + col)[keep], zc[i[keep]], ok[i[keep]]

            r = math.sqrt(r2)
            ids = _rank(*_candidates(c - r, c + r, S, 0, S, test), K, S * S)
        live = ids >= 0
        pix, slot = torch.nonzero(live, as_tuple=True)
        i = ids[pix, slot]
        px = torch.stack([_centres(pix % S, S), _centres(pix // S, S)], 1)
        d = ((px - xy[i]) ** 2).sum(1)
        zero = torch.zeros((S * S, K), dtype=torch.float64, device=DEV)
        q = torch.ones_like(zero).index_put((pix, slot), d / r2)
        fv = torch.zeros((S * S, K, D), dtype=torch.float64, device=DEV).index_put((pix, slot), feats[at + i])
        al = 1 - q
        if case["norm"]:
            tot = al.sum(1, keepdim=True)
            img = torch.where(tot > 0, (al[:, :, None] * fv).sum(1) / torch.where(tot > 0, tot, 1.0), 0.0)
        else:
            T, img = torch.ones_like(q[:, 0]), 0.0
            for k in range(K):
                img = img + (al[:, k] * T)[:, None] * fv[:, k]
                T = T * q[:, k]
        got = torch.autograd.grad(img, [pts, feats], s["grad"][n].double().view(S * S, D), allow_unused=True)
        for t, g in zip(grads, got):
            if g is not None:
                t += g
        outs.append(img.detach().view(S, S, D))
    return [torch.stack(outs), *grads]


def _nearest(p, q, K):
    """Rows of the K nearest candidates (FP64 distances) of every query of one cloud."""
    got = []
    step = max(1, (1 << 26) // max(1, q.shape[0]))
    for a in range(0, p.shape[0], step):
        x = p[a:a + step]
        # shortlist in fp32 differences, ranked again in FP64
        d = ((x[:, None, :] - q[None]) ** 2).sum(2)
        short = d.topk(min(K + 8, q.shape[0]), dim=1, largest=False).indices
        e = ((x.double()[:, None, :] - q.double()[short]) ** 2).sum(2)
        got.append(torch.gather(short, 1, e.topk(min(K, q.shape[0]), dim=1, largest=False).indices))
    return torch.cat(got)


def _exact_clouds(case, seed):
    s = _cloud_inputs(case, seed)
    p, q = (s[k].detach() for k in ("p", "q"))
    p64, q64 = p.double().requires_grad_(True), q.double().requires_grad_(True)
    K = case["K"] if case["call"] == "knn" else 1
    rows = [[int(x) for x in s[k]] for k in ("first_p", "len_p", "first_q", "len_q")]
    dists = torch.full((p.shape[0], K), math.inf, dtype=torch.float64, device=DEV)
    per = []
    for fp, lp, fq, lq in zip(*rows):
        i = _nearest(p[fp:fp + lp], q[fq:fq + lq], K)
        d = ((p64[fp:fp + lp, None] - q64[fq:fq + lq][i]) ** 2).sum(2)
        if case["call"] == "knn":
            dists[fp:fp + lp, :i.shape[1]] = d
            continue
        j = _nearest(q[fq:fq + lq], p[fp:fp + lp], 1)[:, 0]
        e = ((q64[fq:fq + lq] - p64[fp:fp + lp][j]) ** 2).sum(1)
        per.append(d.mean() + e.mean())
    if case["call"] == "knn":
        if not case["grad"]:
            return [dists.detach(), None]
        g = torch.where(torch.isfinite(dists), s["grad"].double(), 0.0)
        safe = torch.where(torch.isfinite(dists), dists, 0.0)
        return [dists.detach(), None, *torch.autograd.grad(safe, [p64, q64], g)]
    per = torch.stack(per)
    return [per.mean().detach(), per.detach(), *torch.autograd.grad(per.mean(), [p64, q64])]


def exact(case, seed):
    if case["call"] in MESH_CALLS:
        return _exact_mesh(case, seed)
    if case["call"] == "points":
        return _exact_points(case, seed)
    return _exact_clouds(case, seed)
