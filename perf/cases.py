"""Performance cases of the narrow-band signed distance field: what a program does with the package
through its public entry points, over the range of sizes it is used at.

A case is a dict of plain values; `kind` names the work of one pass:

  forward   sdf_narrow_band of a mesh whose features are kept (a mesh evaluated on a grid), with or
            without winner ids, or with the sign beyond the band (the inside/outside field a flow
            solver's mesh generator reads)
  step      sdf_build_features + sdf_narrow_band of a new soup (a body that changes every time step)
  build     sdf_build_features of a soup and the connectivity tables a program reads from it
  autograd  SDFFunction forward, dense loss, and its backward to the vertices
  fit       update_positions, the forward with a compact band list, and the loss with its vertex
            gradient fused over the list (one step of shape fitting)
  batch     a CUDA graph replay of a batch of meshes of uneven sizes

Meshes are synthetic, closed and seeded: displaced geodesic spheres, displaced tori, noisy torus-knot
tubes, rotated boxes, and a coarse sphere beside a tiny dense one.  exact() is the same field, loss
and gradient in 64 bits, by plain torch: the minimum over all triangles of the point-triangle
distance, signed by the pseudonormal of the closest feature.
"""
import math

import torch

import paper_1903_00353_gb300 as sdf

DEV = "cuda"
F64 = dict(dtype=torch.float64, device=DEV)


# ----------------------------------------------------------------------------- meshes
# Each returns float64 vertices [V, 3] and int64 triangles [T, 3], counter-clockwise seen from
# outside, on the GPU.

def _gen(seed):
    return torch.Generator(device="cpu").manual_seed(seed % (1 << 62))


def _uniform(gen, lo, hi, n=None):
    u = torch.rand(1 if n is None else n, generator=gen, dtype=torch.float64) * (hi - lo) + lo
    return float(u) if n is None else u


def _outward(v, t):
    a, b, c = v[t[:, 0]], v[t[:, 1]], v[t[:, 2]]
    vol = (a * torch.linalg.cross(b, c)).sum()
    return t if float(vol) > 0 else t[:, [0, 2, 1]]


def _quads(nu, nv):
    i, j = torch.meshgrid(torch.arange(nu, device=DEV), torch.arange(nv, device=DEV), indexing="ij")
    i, j = i.reshape(-1), j.reshape(-1)
    i1, j1 = (i + 1) % nu, (j + 1) % nv
    a, b, c, d = i * nv + j, i1 * nv + j, i1 * nv + j1, i * nv + j1
    return torch.cat([torch.stack([a, b, c], 1), torch.stack([a, c, d], 1)])


_T = (1.0 + 5.0 ** 0.5) / 2.0
_ICO_V = [(-1, _T, 0), (1, _T, 0), (-1, -_T, 0), (1, -_T, 0), (0, -1, _T), (0, 1, _T), (0, -1, -_T), (0, 1, -_T),
          (_T, 0, -1), (_T, 0, 1), (-_T, 0, -1), (-_T, 0, 1)]
_ICO_F = [(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2), (10, 7, 6),
          (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5), (2, 4, 11), (6, 2, 10),
          (8, 6, 7), (9, 8, 1)]


def _geodesic(f):
    """Unit directions and triangles of the class-I geodesic sphere of frequency f (20 f^2 triangles)."""
    ico = torch.tensor(_ICO_V, **F64)
    faces = torch.tensor(_ICO_F, device=DEV)
    i, j = torch.meshgrid(torch.arange(f + 1, device=DEV), torch.arange(f + 1, device=DEV), indexing="ij")
    i, j = i.reshape(-1), j.reshape(-1)

    def corner_weights(ii, jj):  # lattice points of every face: weights of its three corners
        return torch.stack([f - ii - jj, ii, jj], 1)[None].expand(20, -1, -1)

    up = i + j < f
    dn = i + j < f - 1
    tri = [(i[up], j[up]), (i[up] + 1, j[up]), (i[up], j[up] + 1)], [(i[dn] + 1, j[dn]), (i[dn] + 1, j[dn] + 1),
                                                                   (i[dn], j[dn] + 1)]
    w = torch.cat([torch.stack([corner_weights(*p) for p in t], 2) for t in tri], 1)  # [20, f^2, 3 corners, 3]
    # a lattice point's key is linear in its weights, so that the faces sharing it agree on it
    gen = _gen(12)
    code = torch.randint(1 << 40, 1 << 62, (12,), generator=gen).to(DEV)
    key = (w * code[faces][:, None, None, :]).sum(-1).reshape(-1)
    _, inv = torch.unique(key, return_inverse=True)
    n = int(inv.max()) + 1
    pos = (w.to(torch.float64)[..., None] * ico[faces][:, None, None]).sum(-2).reshape(-1, 3)
    first = torch.full((n,), pos.shape[0], device=DEV, dtype=torch.int64)
    first.scatter_reduce_(0, inv, torch.arange(pos.shape[0], device=DEV), "amin")
    d = pos[first]
    return d / d.norm(dim=1, keepdim=True), inv.reshape(-1, 3)


def sphere(freq, seed, radius=0.3, displacement=0.02, center=(0.5, 0.5, 0.5)):
    d, t = _geodesic(freq)
    gen = _gen(seed)
    bump = torch.zeros(d.shape[0], **F64)
    for _ in range(6):
        k = torch.randn(3, generator=gen, dtype=torch.float64)
        k = k * (_uniform(gen, 1.0, 3.0) / float(k.norm()))
        bump += _uniform(gen, 0.5, 1.0) * torch.sin(d @ k.to(DEV) + _uniform(gen, 0.0, 2 * math.pi))
    r = radius + displacement * bump / bump.abs().max()
    v = torch.tensor(center, **F64) + d * r[:, None]
    return v, _outward(v, t)


def torus(nu, nv, seed, R=0.3, r=0.1, bump=0.02):
    gen = _gen(seed)
    pu, pv = _uniform(gen, 0, 2 * math.pi), _uniform(gen, 0, 2 * math.pi)
    u, v = torch.meshgrid(torch.arange(nu, **F64) * (2 * math.pi / nu), torch.arange(nv, **F64) * (2 * math.pi / nv),
                          indexing="ij")
    rr = r + bump * torch.sin(5 * u + pu) * torch.sin(7 * v + pv)
    p = torch.stack([(R + rr * torch.cos(v)) * torch.cos(u), (R + rr * torch.cos(v)) * torch.sin(u),
                     rr * torch.sin(v)], -1).reshape(-1, 3)
    edge = min(2 * math.pi * R / nu, 2 * math.pi * r / nv)
    p = p + (min(1e-3, 0.15 * edge) * torch.randn(p.shape, generator=gen, dtype=torch.float64)).to(DEV) + 0.5
    return p, _outward(p, _quads(nu, nv))


def knot(n_along, n_around, seed, radius=0.04, noise=0.005, R=0.3, a=0.12):
    """Tube around the (3, 7) torus knot; its frame is the normal of the torus that carries the curve."""
    gen = _gen(seed)
    t = torch.arange(n_along, **F64) * (2 * math.pi / n_along)
    rho, dr = R + a * torch.cos(7 * t), -7 * a * torch.sin(7 * t)
    c = torch.stack([rho * torch.cos(3 * t), rho * torch.sin(3 * t), a * torch.sin(7 * t)], -1)
    d = torch.stack([dr * torch.cos(3 * t) - 3 * rho * torch.sin(3 * t),
                     dr * torch.sin(3 * t) + 3 * rho * torch.cos(3 * t), 7 * a * torch.cos(7 * t)], -1)
    n = torch.stack([torch.cos(7 * t) * torch.cos(3 * t), torch.cos(7 * t) * torch.sin(3 * t), torch.sin(7 * t)], -1)
    b = torch.linalg.cross(d / d.norm(dim=1, keepdim=True), n)
    s, th = torch.meshgrid(t, torch.arange(n_around, **F64) * (2 * math.pi / n_around), indexing="ij")
    field = torch.zeros_like(s)
    for _ in range(8):
        fs, ft = int(_uniform(gen, 1, 40)), int(_uniform(gen, 1, 9))
        field += _uniform(gen, 0.5, 1.0) * torch.sin(fs * s + ft * th + _uniform(gen, 0, 2 * math.pi))
    q = radius + noise * field / field.abs().max()
    p = c[:, None] + q[..., None] * (torch.cos(th)[..., None] * n[:, None] + torch.sin(th)[..., None] * b[:, None])
    p = p.reshape(-1, 3) + 0.5
    return p, _outward(p, _quads(n_along, n_around))


def box(m, seed):
    """A rotated box, each face m x m quads: flat edges and vertices, as CAD surfaces have."""
    gen = _gen(seed)
    q = torch.randn(4, generator=gen, dtype=torch.float64)
    w, x, y, z = (q / q.norm()).tolist()
    rot = torch.tensor([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                        [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                        [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]], **F64)
    half = _uniform(gen, 0.12, 0.24, 3).to(DEV)
    i, j = torch.meshgrid(torch.arange(m, device=DEV), torch.arange(m, device=DEV), indexing="ij")
    i, j = i.reshape(-1), j.reshape(-1)
    quad = [(i, j), (i + 1, j), (i + 1, j + 1), (i, j + 1)]
    tris = []
    for ax in range(3):
        for side in (0, m):
            p = []
            for a, b in quad:
                l = [None, None, None]
                l[ax], l[(ax + 1) % 3], l[(ax + 2) % 3] = torch.full_like(a, side), a, b
                p.append((l[0] * (m + 1) + l[1]) * (m + 1) + l[2])
            if side == 0:
                p = p[::-1]
            tris += [torch.stack([p[0], p[1], p[2]], 1), torch.stack([p[0], p[2], p[3]], 1)]
    ids, t = torch.unique(torch.cat(tris), return_inverse=True)
    l = torch.stack([ids // ((m + 1) * (m + 1)), ids // (m + 1) % (m + 1), ids % (m + 1)], 1).to(torch.float64)
    v = ((2 * l / m - 1) * half) @ rot.T + 0.5
    return v, _outward(v, t)


def cluster(freq, seed):
    """A coarse sphere of 320 triangles and a dense sphere of radius 2e-4: very uneven triangle sizes."""
    v, t = sphere(4, seed, displacement=0.0)
    gen = _gen(seed + 1)
    c = 0.05 + 0.01 * torch.rand(3, generator=gen, dtype=torch.float64)
    v2, t2 = sphere(freq, seed, radius=2e-4, displacement=0.0, center=c.tolist())
    return torch.cat([v, v2]), torch.cat([t, t2 + v.shape[0]])


def _mesh(case, seed):
    m, p, q = case["mesh"], case["p"], case.get("q", 0)
    if m == "sphere":
        v, t = sphere(p, seed)
    elif m == "torus":
        v, t = torus(p, q, seed)
    elif m == "knot":
        v, t = knot(p, q, seed)
    elif m == "box":
        v, t = box(p, seed)
    else:
        v, t = cluster(p, seed)
    v = v.to(torch.float32)
    # an unordered soup: triangles shuffled, each triangle's corners rotated
    gen = torch.Generator(device=DEV).manual_seed(seed % (1 << 62))
    t = t[torch.randperm(t.shape[0], generator=gen, device=DEV)]
    rot = torch.randint(0, 3, (t.shape[0], 1), generator=gen, device=DEV)
    t = torch.gather(t, 1, (torch.arange(3, device=DEV)[None] + rot) % 3)
    return v, t, v[t].contiguous()


def _n_tri(case):
    p, q = case["p"], case.get("q", 0)
    return {"sphere": 20 * p * p, "torus": 2 * p * q, "knot": 2 * p * q, "box": 12 * p * p,
            "cluster": 320 + 20 * p * p}[case["mesh"]]


_AREA = {"sphere": 1.16, "torus": 1.2, "knot": 1.95, "box": 0.8, "cluster": 1.13}


def _grid(case):
    """Cells of size 1 / (longest side), the box centred on the mesh (a shorter side is a window)."""
    n = (case["nx"], case["ny"], case["nz"])
    h = 1.0 / max(n)
    return sdf.Grid(*n, origin=tuple(0.5 - 0.5 * m * h for m in n), h=h), case["w"] * h


def _batch(case, seed):
    """The problems of a batch: mesh kinds in turn, triangles and grid sides spread over the ranges."""
    gen = torch.Generator().manual_seed(case["count"] * 7919 + case["n_max"])  # the sizes are the case's own
    out = []
    for k in range(case["count"]):
        tris = math.exp(_uniform(gen, math.log(case["t_min"]), math.log(case["t_max"])))
        n = 32 * int(_uniform(gen, 2, case["n_max"] // 32 + 0.999))
        kind = ("sphere", "torus", "box")[k % 3]
        sub = {"mesh": kind, "nx": n, "ny": n, "nz": n, "w": case["w"]}
        if kind == "torus":
            sub["q"] = max(8, round(math.sqrt(tris / 5)))
            sub["p"] = max(8, round(tris / 2 / sub["q"]))
        else:
            sub["p"] = max(2, round(math.sqrt(tris / (20 if kind == "sphere" else 12))))
        out.append((sub, seed * 1009 + k))
    return out


# ----------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest use: a coarse solid on a coarse grid, bound by launches and latency
        dict(name="solid_64", kind="forward", mesh="sphere", p=4, nx=64, ny=64, nz=64, w=3.0, winner=True),
        # a CAD-shaped body moving through a flow solver's grid: rebuilt every time step, inside/outside
        # field wanted
        dict(name="moving_body_128", kind="step", mesh="box", p=30, nx=128, ny=128, nz=96, w=3.0, fill=True),
        # a scanned model of the paper's smaller size on a fine grid
        dict(name="torus_512", kind="forward", mesh="torus", p=250, q=100, nx=512, ny=512, nz=512, w=4.0),
        # the inside/outside field on a grid that fits no tile or vector width
        dict(name="signed_ragged", kind="forward", mesh="knot", p=1024, q=64, nx=333, ny=331, nz=257, w=3.0,
             fill=True),
        # CAD-like triangle sizes: thousands of tiny triangles beside large ones
        dict(name="uneven_256", kind="forward", mesh="cluster", p=60, nx=256, ny=256, nz=256, w=3.0),
        # a mesh far finer than the grid (a large scan on a moderate grid), winners kept for later use
        dict(name="knot_512", kind="forward", mesh="knot", p=8192, q=128, nx=512, ny=512, nz=512, w=3.0, winner=True),
        # the paper's largest model size on a fine grid
        dict(name="knot_1024", kind="forward", mesh="knot", p=8192, q=128, nx=1024, ny=1024, nz=1024, w=3.0),
        # connectivity of a small scan and of the largest one
        dict(name="build_50k", kind="build", mesh="torus", p=250, q=100),
        dict(name="build_2m", kind="build", mesh="knot", p=8192, q=128),
        # a training step through autograd, dense field and gradient
        dict(name="autograd_256", kind="autograd", mesh="torus", p=250, q=100, nx=256, ny=256, nz=256, w=3.0),
        # one step of fitting a shape of 200,000 triangles to a target field
        dict(name="fit_512", kind="fit", mesh="sphere", p=100, nx=512, ny=512, nz=512, w=4.0),
        # many small bodies at once, replayed from a CUDA graph
        dict(name="batch_24", kind="batch", count=24, t_min=1e3, t_max=1e5, n_max=256, w=3.0),
    ]


def draw(rng):
    def log_uniform(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["forward", "forward", "forward", "step", "build", "autograd", "fit", "batch"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 32), t_min=5e2, t_max=log_uniform(4e3, 1e5),
                    n_max=32 * rng.randint(3, 8), w=rng.choice([2.0, 3.0, 4.0]))
    top = {"forward": 900, "step": 512, "autograd": 400, "fit": 600, "build": 900}[kind]
    n = int(log_uniform(48, top))
    sides = [n, max(40, int(n * rng.uniform(0.5, 1.0))), max(40, int(n * rng.uniform(0.4, 1.0)))]
    if rng.random() < 0.4:  # powers of two and their multiples are common
        sides = [max(32, s // 32 * 32) for s in sides]
    rng.shuffle(sides)
    mesh = rng.choice(["sphere", "torus", "knot", "box"])
    # mean triangle edge in cells, from meshes finer than the grid to a few large facets
    edge = log_uniform(0.8, 12.0) / max(sides)
    tris = min(2.0e6, max(400.0 if mesh != "knot" else 2e4, _AREA[mesh] / (0.43 * edge * edge)))
    case = dict(kind=kind, mesh=mesh)
    if mesh in ("sphere", "box"):
        case["p"] = max(4, round(math.sqrt(tris / (20 if mesh == "sphere" else 12))))
    else:
        ratio = 2.5 if mesh == "torus" else 24.0
        case["q"] = max(8, round(math.sqrt(tris / 2 / ratio)))
        case["p"] = max(16, round(tris / 2 / case["q"]))
    if kind == "build":
        return case
    case.update(nx=sides[0], ny=sides[1], nz=sides[2], w=rng.choice([2.0, 2.5, 3.0, 4.0, 5.0]))
    if kind in ("forward", "step"):
        case["fill"] = rng.random() < 0.3
        case["winner"] = rng.random() < 0.3
    return case


# ----------------------------------------------------------------------------- one pass
def _target(case, grid):
    """Target field of the losses: the signed distance to a sphere (FP32)."""
    ax = [torch.arange(n, device=DEV, dtype=torch.float32) * grid.h + (o + 0.5 * grid.h - 0.5)
          for n, o in zip((grid.nx, grid.ny, grid.nz), grid.origin)]
    return (ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2).sqrt_().sub_(0.29)


def _order(feats, t, n_vert):
    """The user's vertex of every vertex of the library, and the reverse."""
    to_user = torch.empty(feats.n_vert, dtype=torch.int64, device=DEV)
    to_user[feats.vertex_map().long()] = t.reshape(-1)
    to_lib = torch.empty(n_vert, dtype=torch.int64, device=DEV)
    to_lib[to_user] = torch.arange(feats.n_vert, device=DEV)
    return to_user, to_lib


def prepare(case, seed):
    s = {"case": case, "kind": case["kind"]}
    if case["kind"] == "batch":
        feats, grids, ws = [], [], []
        for sub, sub_seed in _batch(case, seed):
            grid, w = _grid(sub)
            feats.append(sdf.sdf_build_features(_mesh(sub, sub_seed)[2]))
            grids.append(grid)
            ws.append(w)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            s["batch"] = sdf.sdf_batch_create(feats, grids, ws)
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"], stream=stream):
                s["batch"].run(stream=stream)
        torch.cuda.current_stream().wait_stream(stream)
        return s
    v, t, soup = _mesh(case, seed)
    s["soup"] = soup
    if case["kind"] == "build":
        return s
    s["grid"], s["w"] = _grid(case)
    s["out"] = torch.empty(s["grid"].shape, dtype=torch.float32, device=DEV)
    s["winner"] = torch.empty(s["grid"].shape, dtype=torch.int32, device=DEV) if case.get("winner") else False
    s["flags"] = sdf.FLAG_FILL_SIGN if case.get("fill") else 0
    if case["kind"] == "step":
        return s
    s["feats"] = sdf.sdf_build_features(soup)
    if case["kind"] in ("autograd", "fit"):
        s["verts"], s["target"] = v, _target(case, s["grid"])
        s["to_user"], s["to_lib"] = _order(s["feats"], t, v.shape[0])
    if case["kind"] == "fit":
        # as long as the band may get, so that the unsynchronised forward below has room
        s["list"] = sdf.BandList(2 * int(_band_points(case)) + (1 << 18))
    return s


def run(s):
    kind = s["kind"]
    if kind == "forward":
        return sdf.sdf_narrow_band(s["feats"], s["grid"], s["w"], out=s["out"], winner=s["winner"], flags=s["flags"])
    if kind == "step":
        feats = sdf.sdf_build_features(s["soup"])
        return sdf.sdf_narrow_band(feats, s["grid"], s["w"], out=s["out"], winner=s["winner"], flags=s["flags"])
    if kind == "build":
        feats = sdf.sdf_build_features(s["soup"])
        return {"vertices": feats.vertices(), "vertex_map": feats.vertex_map(), "face_map": feats.face_map(),
                "edges": feats.edges(), "counts": feats.counts}
    if kind == "autograd":
        x = s["verts"].detach().requires_grad_()
        dist = sdf.SDFFunction.apply(x[s["to_user"]], s["feats"], s["grid"], s["w"])
        loss, grad, _ = sdf.band_l2_loss(dist.detach(), s["target"])
        return {"loss": loss, "dist": dist.detach(), "grad": torch.autograd.grad(dist, x, grad)[0]}
    if kind == "fit":
        s["feats"].update_positions(s["verts"][s["to_user"]])
        dist, band = sdf.sdf_narrow_band_list(s["feats"], s["grid"], s["w"], out=s["out"], band_list=s["list"],
                                              flags=sdf.FLAG_NO_SYNC)
        loss, grad, count = sdf.band_list_l2(s["feats"], s["grid"], band, dist, s["target"])
        return {"loss": loss, "dist": dist, "grad": grad[s["to_lib"]], "count": count}
    s["graph"].replay()
    return s["batch"].outs


# ----------------------------------------------------------------------------- unavoidable work
def _band_points(case):
    n = max(case["nx"], case["ny"], case["nz"])
    return min(case["nx"] * case["ny"] * case["nz"], _AREA[case["mesh"]] * 2 * case["w"] * n * n)


def work(case):
    """Bytes: the soup (36 B per triangle) or the feature records a forward reads (face 64 B, edge
    80 B, vertex 48 B, corner planes 16 B), each once; the outputs once.  Flops: a distance (about 30)
    per band point, about 500 per triangle of a build's records, about 60 per point of an adjoint."""
    if case["kind"] == "batch":
        subs = [work(dict(sub, kind="forward")) for sub, _ in _batch(case, 0)]
        return {k: sum(w[k] for w in subs) for k in ("bytes", "flops")}
    t = _n_tri(case)
    v, records = t // 2, t * (64 + 1.5 * 80 + 0.5 * 48 + 3 * 16)
    build = {"bytes": t * 36 + v * 12 + t * (12 + 4 + 1.5 * 16), "flops": 500.0 * t}
    if case["kind"] == "build":
        return build
    points, band = case["nx"] * case["ny"] * case["nz"], _band_points(case)
    if case["kind"] == "step":
        return {"bytes": t * 36 + points * 4 * (2 if case.get("winner") else 1), "flops": build["flops"] + 30 * band}
    out = {"bytes": records + points * 4 * (2 if case.get("winner") else 1), "flops": 30 * band}
    if case["kind"] == "forward":
        return out
    # vertices in, gradient out, the target at the band points (dense: over the whole grid)
    target = points * 4 if case["kind"] == "autograd" else band * 4
    return {"bytes": v * 24 + points * 4 + target, "flops": 500.0 * t + 90 * band}


# ----------------------------------------------------------------------------- the same in 64 bits
def _dot(a, b):
    return a[:, 0] * b[:, 0] + a[:, 1] * b[:, 1] + a[:, 2] * b[:, 2]


def _closest(p, a, b, c):
    """Barycentric weights of the closest point of triangles (a, b, c) to points p, by the Voronoi
    regions of corners, edges and face."""
    ab, ac, ap = b - a, c - a, p - a
    d1, d2 = _dot(ab, ap), _dot(ac, ap)
    d00, d01, d11 = _dot(ab, ab), _dot(ab, ac), _dot(ac, ac)
    d3, d4, d5, d6 = d1 - d00, d2 - d01, d1 - d01, d2 - d11  # the same products seen from b and from c
    va, vb, vc = d3 * d6 - d5 * d4, d5 * d2 - d1 * d6, d1 * d4 - d3 * d2
    den = va + vb + vc
    v, w = vb / den, vc / den
    bc = (d4 - d3) + (d5 - d6)
    t = (d4 - d3) / bc
    on = (va <= 0) & (d4 - d3 >= 0) & (d5 - d6 >= 0)
    v, w = torch.where(on, 1 - t, v), torch.where(on, t, w)
    on = (vb <= 0) & (d2 >= 0) & (d6 <= 0)
    v, w = torch.where(on, 0.0, v), torch.where(on, d2 / d11, w)
    on = (vc <= 0) & (d1 >= 0) & (d3 <= 0)
    v, w = torch.where(on, d1 / d00, v), torch.where(on, 0.0, w)
    for on, vv, ww in (((d6 >= 0) & (d5 <= d6), 0.0, 1.0), ((d3 >= 0) & (d4 <= d3), 1.0, 0.0),
                       ((d1 <= 0) & (d2 <= 0), 0.0, 0.0)):
        v, w = torch.where(on, vv, v), torch.where(on, ww, w)
    return v, w


def _pairs(lo, hi, chunk=6_000_000):
    """Every (triangle, grid point) of the triangles' index boxes, in chunks: triangle, i, j, k."""
    n = (hi - lo + 1).clamp(min=0)
    cnt = n[:, 0] * n[:, 1] * n[:, 2]
    end = cnt.cumsum(0)
    total = int(end[-1])
    for s in range(0, total, chunk):
        q = torch.arange(s, min(s + chunk, total), device=DEV)
        tri = torch.searchsorted(end, q, right=True)
        r = q - (end[tri] - cnt[tri])
        x = r % n[tri, 0]
        r = r // n[tri, 0]
        yield tri, lo[tri, 0] + x, lo[tri, 1] + r % n[tri, 1], lo[tri, 2] + r // n[tri, 1]


def _boxes(v, t, grid, w):
    o = torch.tensor([float(torch.tensor(x, dtype=torch.float32)) for x in grid.origin], **F64)
    h = float(torch.tensor(grid.h, dtype=torch.float32))
    c = v[t]
    top = torch.tensor([grid.nx, grid.ny, grid.nz], device=DEV) - 1
    lo = torch.ceil((c.amin(1) - w - o) / h - 0.5).long().clamp(min=0)
    hi = torch.minimum(torch.floor((c.amax(1) + w - o) / h - 0.5).long(), top)
    return lo, hi, o, h


def _exact(v32, t, grid, w, limit):
    """The field in 64 bits and, for every band point, its triangle, closest-point weights and the
    direction s (p - q) / |p - q|; None where it would take too long."""
    v = v32.to(torch.float64)
    w = float(torch.tensor(w, dtype=torch.float32))
    lo, hi, o, h = _boxes(v, t, grid, w)
    if float((hi - lo + 1).clamp(min=0).to(torch.float64).prod(1).sum()) > limit:
        return None
    a, b, c = v[t[:, 0]], v[t[:, 1]], v[t[:, 2]]
    n = torch.linalg.cross(b - a, c - a)
    n = n / n.norm(dim=1, keepdim=True)
    # pseudonormals: n1 + n2 of the edges, the angle-weighted sum of the vertices
    nv = torch.zeros_like(v)
    for k in range(3):
        e, f = v[t[:, (k + 1) % 3]] - v[t[:, k]], v[t[:, (k + 2) % 3]] - v[t[:, k]]
        ang = torch.atan2(torch.linalg.cross(e, f).norm(dim=1), _dot(e, f))
        nv.index_add_(0, t[:, k], ang[:, None] * n)
    edge = torch.stack([torch.minimum(t, t.roll(-1, 1)) * v.shape[0] + torch.maximum(t, t.roll(-1, 1))]).reshape(-1)
    _, eid = torch.unique(edge, return_inverse=True)
    ne = torch.zeros(int(eid.max()) + 1, 3, **F64).index_add_(0, eid, n.repeat_interleave(3, 0))
    eid = eid.reshape(-1, 3)

    best = torch.full((grid.nx * grid.ny * grid.nz,), math.inf, **F64)

    def walk():
        for tri, i, j, k in _pairs(lo, hi):
            p = torch.stack([i, j, k], 1).to(torch.float64).add_(0.5).mul_(h).add_(o)
            wv, ww = _closest(p, a[tri], b[tri], c[tri])
            wa = 1 - wv - ww
            r = p - (wa[:, None] * a[tri] + wv[:, None] * b[tri] + ww[:, None] * c[tri])
            yield tri, (k * grid.ny + j) * grid.nx + i, p, wa, wv, ww, r, _dot(r, r)

    for _, idx, _, _, _, _, _, d2 in walk():
        best.scatter_reduce_(0, idx, d2, "amin")
    kept = []
    for tri, idx, p, wa, wv, ww, r, d2 in walk():
        m = ((d2 == best[idx]) & (d2 < w * w)).nonzero()[:, 0]
        tri, idx, wa, wv, ww, r, d2 = tri[m], idx[m], wa[m], wv[m], ww[m], r[m], d2[m]
        za, zv, zw = wa.abs() < 1e-12, wv == 0, ww == 0
        nrm = n[tri]
        for z, k in ((zw, 0), (za, 1), (zv, 2)):  # a zero weight: on the opposite edge
            nrm = torch.where(z[:, None], ne[eid[tri, k]], nrm)
        for z, k in ((zv & zw, 0), (za & zw, 1), (za & zv, 2)):  # two: at a corner
            nrm = torch.where(z[:, None], nv[t[tri, k]], nrm)
        sgn = torch.where(_dot(r, nrm) < 0, -1.0, 1.0)
        u = torch.where((d2 > 1e-24)[:, None], sgn[:, None] * r / d2.sqrt().clamp(min=1e-12)[:, None], n[tri])
        kept.append((tri, idx, torch.stack([wa, wv, ww], 1), u, sgn * d2.sqrt()))
    tri, idx, lam, u, d = (torch.cat(x) for x in zip(*kept))
    # one entry per point
    first = torch.full((best.shape[0],), idx.shape[0], dtype=torch.int64, device=DEV)
    first.scatter_reduce_(0, idx, torch.arange(idx.shape[0], device=DEV), "amin")
    m = first[first < idx.shape[0]]
    best.fill_(math.inf)
    best[idx[m]] = d[m]
    return best.reshape(grid.shape), tri[m], idx[m], lam[m], u[m], d[m]


def _signed(dist):
    """-inf inside and +inf outside at the points beyond the band: the sign of the nearest band point
    of the row, then of the nearest known row."""
    s = torch.where(torch.isfinite(dist), torch.where(dist < 0, -1, 1), 0).to(torch.int8)
    for axis in (2, 1, 0):
        for back in (False, True):
            q = s.flip(axis) if back else s
            pos = torch.arange(1, q.shape[axis] + 1, device=DEV, dtype=torch.int32)
            pos = pos.reshape([-1 if a == axis else 1 for a in range(3)])
            last = torch.where(q != 0, pos, 0).cummax(axis)[0]
            q = torch.where(last > 0, q.gather(axis, (last - 1).clamp(min=0).long()), q)
            s = q.flip(axis) if back else q
    return torch.where(torch.isfinite(dist), dist, torch.where(s < 0, -math.inf, math.inf))


def exact(case, seed):
    if case["kind"] == "build":
        return None  # tables of whole numbers, and copies of the input's coordinates
    if case["kind"] == "batch":
        out = []
        for sub, sub_seed in _batch(case, seed):
            v, t, _ = _mesh(sub, sub_seed)
            e = _exact(v, t, *_grid(sub), limit=3e8)
            out.append(None if e is None else e[0])
        return out
    v, t, _ = _mesh(case, seed)
    grid, w = _grid(case)
    e = _exact(v, t, grid, w, limit=4e9)
    if e is None:
        return None
    dist, tri, idx, lam, u, d = e
    if case["kind"] in ("forward", "step"):
        dist = _signed(dist) if case.get("fill") else dist
        return (dist, None) if case.get("winner") else dist
    diff = d - _target(case, grid).reshape(-1)[idx].to(torch.float64)
    grad = torch.zeros(v.shape[0], 3, **F64)
    for k in range(3):
        grad.index_add_(0, t[tri, k], (-2 * diff * lam[:, k])[:, None] * u)
    return {"loss": (diff * diff).sum(), "dist": dist, "grad": grad}
