"""Performance cases: what a program that uses this library has it do.

The library renders oblique city scenes (a low-resolution feature grid, three
feature planes, an occupancy plane and a small deferred MLP), trains them and
extracts the real-time scene.  Each case is one such call or group of calls
through the public Python entry points, on seeded synthetic scenes of the
repository's own shapes: a "field" (dense grid, low heightfield: the small
render and training scene) and a "city" (brick grid, buildings in a void).

A scene is given by `res`, the grid's vertices per side:
  field  grid res^2 x res/4 dense, planes (4 res)^2 and 4 res x res/2,
         occupancy (res/2)^2, step 1/256, n_max 128          (res 64)
  city   grid res^2 x res/16 in 8^3 bricks, planes (4 res)^2 and 4 res x res/4,
         occupancy (res/2)^2, step 1/2048, n_max 512         (res 512; BF16 1024)
"""
import math

import numpy as np
import torch

import paper_2404_09531_gb300 as om

DEV = "cuda"
NCH = 8
MLP_NPARAM = 883


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest render: a preview of a small scene, with its sample counts
        {"name": "field_64x64_f32", "kind": "render", "scene": "field", "res": 64, "dtype": "f32", "cams": 1,
         "width": 64, "height": 64, "count": True},
        # a list of held-out pixels rendered for an error estimate, with counts
        {"name": "rays_10007_city_f32", "kind": "rays", "scene": "city", "res": 512, "dtype": "f32", "n": 10007},
        # an odd-sized window drawn by a host that owns all device memory
        {"name": "noalloc_641x361_city_f32", "kind": "noalloc", "scene": "city", "res": 512, "dtype": "f32",
         "width": 641, "height": 361},
        # a viewer's frame: pixels alone
        {"name": "frame_1080_city_f32", "kind": "render", "scene": "city", "res": 512, "dtype": "f32", "cams": 1,
         "width": 1920, "height": 1080, "count": False},
        # the headline workload: eight 1080p cameras in one call
        {"name": "frames8_1080_city_f32", "kind": "render", "scene": "city", "res": 512, "dtype": "f32", "cams": 8,
         "width": 1920, "height": 1080, "count": False},
        # a 4K viewer's frame of the large BF16 scene
        {"name": "frame_4k_city_bf16", "kind": "render", "scene": "city", "res": 1024, "dtype": "bf16", "cams": 1,
         "width": 3840, "height": 2160, "count": False},
        # a small ragged batch through autograd, several smoothness directions
        {"name": "autograd_5003_field_f32", "kind": "autograd", "scene": "field", "res": 64, "dtype": "f32",
         "n": 5003, "k": 3},
        # the training step: loss and gradients of 2^18 rays
        {"name": "train_2p18_field_f32", "kind": "train", "scene": "field", "res": 64, "dtype": "f32",
         "n": 1 << 18, "k": 1},
        # the large training step: 2^20 rays of a city with BF16 features
        {"name": "train_2p20_city_bf16", "kind": "train", "scene": "city", "res": 512, "dtype": "bf16",
         "n": 1 << 20, "k": 1},
        # a whole training iteration: step, both regularisers, Adam, hull update
        {"name": "iteration_2p14_field_f32", "kind": "iteration", "scene": "field", "res": 64, "dtype": "f32",
         "n": 1 << 14, "k": 1, "points": 1 << 14, "erays": 1 << 10},
        # the optimiser alone at a city's size: FP32 masters with BF16 shadows
        {"name": "adam_city_bf16", "kind": "adam", "res": 512, "bricks": 2453, "dtype": "bf16"},
        # extraction after training: bricks, occupancy grid, cropped planes
        {"name": "export_512_city_f32", "kind": "export", "scene": "city", "res": 512, "dtype": "f32",
         "voxels": 2048},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("render", "render", "render", "rays", "noalloc", "autograd", "train", "train", "iteration",
                       "adam", "export"))
    scene = rng.choice(("field", "city"))
    dtype = rng.choice(("f32", "bf16"))
    res = _log_int(rng, 40, 128) if scene == "field" else _log_int(rng, 256, 512 if dtype == "f32" else 1024)
    base = {"kind": kind, "scene": scene, "res": res, "dtype": dtype}
    if kind == "render":
        width = _log_int(rng, 64, 3840)
        height = max(48, int(width * rng.uniform(0.5, 1.0)))
        cams = rng.randint(1, 8)
        while cams > 1 and cams * width * height > 8 * 1920 * 1080:
            cams -= 1
        return dict(base, cams=cams, width=width, height=height, count=width * height * cams <= 1 << 17)
    if kind == "rays":
        return dict(base, n=_log_int(rng, 1000, 1 << 20))
    if kind == "noalloc":
        width = _log_int(rng, 64, 1920)
        return dict(base, width=width, height=max(48, int(width * rng.uniform(0.5, 1.0))))
    if kind in ("autograd", "train"):
        return dict(base, n=_log_int(rng, 1000, 1 << 20), k=rng.choice((0, 1, 1, 2, 3)))
    if kind == "iteration":
        return dict(base, scene="field", res=_log_int(rng, 40, 128), dtype="f32", n=_log_int(rng, 2000, 1 << 17),
                    k=rng.choice((1, 2)), points=_log_int(rng, 2000, 1 << 15), erays=_log_int(rng, 200, 1 << 12))
    if kind == "adam":
        res = _log_int(rng, 64, 512)
        return {"kind": kind, "res": res, "bricks": _log_int(rng, 100, 2500), "dtype": dtype}
    return dict(base, scene="city", res=_log_int(rng, 256, 512), voxels=_log_int(rng, 256, 2048))


# ------------------------------------------------------------------ scenes
def _torch_dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


class _Heights:
    """Four seeded sines, and 64 box buildings for a city (float64)."""

    def __init__(self, rng, city):
        self.city = city
        self.base = -0.03 if city else 0.0
        self.a = rng.uniform(0.001, 0.0025, 4) if city else rng.uniform(0.01, 0.02, 4)
        self.u, self.v = rng.uniform(-2.0, 2.0, 4), rng.uniform(-2.0, 2.0, 4)
        self.phi = rng.uniform(0.0, 2.0 * math.pi, 4)
        self.c = rng.uniform(-0.55, 0.55, (64, 2))
        self.s = rng.uniform(0.02, 0.1, (64, 2))
        self.h = rng.uniform(0.005, 0.04, 64)

    def ground(self, x, y):
        h = torch.full_like(x, self.base)
        for k in range(4):
            h = h + self.a[k] * torch.sin(2.0 * math.pi * (self.u[k] * x + self.v[k] * y) + self.phi[k])
        return h

    def surface(self, x, y):
        g = self.ground(x, y)
        if not self.city:
            return g
        top = torch.zeros_like(g)
        for c, s, h in zip(self.c, self.s, self.h):
            inside = ((x - c[0]).abs() <= 0.5 * s[0]) & ((y - c[1]).abs() <= 0.5 * s[1])
            top = torch.where(inside, top.clamp(min=h), top)
        return g + top


def _shape(case):
    res, city = case["res"], case["scene"] == "city"
    M = res // 2
    if city:
        return dict(aabb=(-1.0, 1.0, -1.0, 1.0, -0.0625, 0.0625), L=(res, res, max(res // 16, 8)),
                    R=(4 * res, 4 * res, res // 4), M=M, brick=8, step=1.0 / 2048, n_max=512, eps=0.002, margin=0.006,
                    radius=0.555 if res < 768 else 0.63, look=0.25, dist=0.6, fov=50.0)
    return dict(aabb=(-1.0, 1.0, -1.0, 1.0, -0.125, 0.125), L=(res, res, res // 4), R=(4 * res, 4 * res, res // 2),
                M=M, brick=0, step=1.0 / 256, n_max=128, eps=0.01, margin=0.03, radius=None, look=0.5, dist=2.5,
                fov=45.0)


def _features(gen, shape, dtype):
    t = torch.empty((*shape, NCH), dtype=torch.float32, device=DEV).normal_(0.0, 0.5, generator=gen)
    t[..., 0].mul_(0.2)  # densities N(0, 0.1)
    return t.to(dtype)


def _axis(lo, hi, n, idx):
    return lo + idx.double() * (hi - lo) / (n - 1)


def _dense_grid(gen, sh, heights, dtype):
    L, box = sh["L"], sh["aabb"]
    x, y, z = torch.meshgrid(*(_axis(box[2 * a], box[2 * a + 1], L[a], torch.arange(L[a], device=DEV))
                               for a in range(3)), indexing="ij")
    grid = _features(gen, L, torch.float32)
    grid[..., 0] += torch.where(z < heights.surface(x[:, :, :1], y[:, :, :1]), 5.0, -5.0).float()
    return grid.to(dtype)


def _brick_pool(gen, sh, heights, table, n, dtype):
    L, box, B = sh["L"], sh["aabb"], sh["brick"]
    pool = _features(gen, (n, B, B, B), torch.float32)
    at = (table >= 0).nonzero()
    at = at[torch.argsort(table[table >= 0])]
    li = torch.arange(B, device=DEV)
    i, j, k = (at[:, a, None] * B + li for a in range(3))  # [n, B] vertex indices
    x, y, z = (_axis(box[2 * a], box[2 * a + 1], L[a], v) for a, v in enumerate((i, j, k)))
    surf = heights.surface(x[:, :, None].expand(n, B, B), y[:, None, :].expand(n, B, B))
    pool[..., 0] += torch.where(z[:, None, None, :] < surf[..., None], 5.0, -5.0).float()
    out = (i >= L[0])[:, :, None, None] | (j >= L[1])[:, None, :, None] | (k >= L[2])[:, None, None, :]
    pool[out] = 0.0
    return pool.to(dtype)


def _occupancy(sh, heights):
    M, box = sh["M"], sh["aabb"]
    hx, hy = (box[1] - box[0]) / M, (box[3] - box[2]) / M
    c = torch.arange(M, device=DEV, dtype=torch.float64) + 0.5
    x, y = torch.meshgrid(box[0] + c * hx, box[2] + c * hy, indexing="ij")
    if not heights.city:
        h = heights.surface(x, y)
        return torch.stack([h - sh["margin"], h + sh["margin"]], -1).float().contiguous()
    lo, hi = torch.full_like(x, math.inf), torch.full_like(x, -math.inf)
    for a in (-0.45, 0.0, 0.45):
        for b in (-0.45, 0.0, 0.45):
            lo = torch.minimum(lo, heights.ground(x + a * hx, y + b * hy))
            hi = torch.maximum(hi, heights.surface(x + a * hx, y + b * hy))
    void = x * x + y * y > sh["radius"] ** 2
    z0 = torch.where(void, 1.0, lo - sh["margin"])  # z_max < z_min marks an empty cell
    z1 = torch.where(void, -1.0, hi + sh["margin"])
    return torch.stack([z0, z1], -1).float().contiguous()


def _make_scene(case, seed, dense=False):
    """The arrays of a seeded scene and an om.Scene over them.  The ground and
    the buildings are the same for every seed (so that every seed stores the
    same number of bricks); features, weights, cameras and rays are the seed's."""
    sh = _shape(case)
    rng = np.random.default_rng([seed, 1])
    gen = torch.Generator(device=DEV).manual_seed(seed)
    heights = _Heights(np.random.default_rng(20240415), case["scene"] == "city")
    dt = _torch_dtype(case)
    occ = _occupancy(sh, heights)
    table = None
    if sh["brick"] and not dense:
        table, n = om.build_brick_table(sh["aabb"], sh["L"], sh["brick"], occ)
        grid = _brick_pool(gen, sh, heights, table, int(n.item()), dt)
    else:
        grid = _dense_grid(gen, sh, heights, dt)
    R = sh["R"]
    mlp = torch.empty(MLP_NPARAM, device=DEV).normal_(0.0, 0.3, generator=gen)
    scene = om.Scene(aabb=sh["aabb"], grid=grid.contiguous(), p_xy=_features(gen, (R[0], R[1]), dt),
                     p_xz=_features(gen, (R[0], R[2]), dt), p_yz=_features(gen, (R[1], R[2]), dt), occ=occ, mlp=mlp,
                     step=sh["step"], eps=sh["eps"], n_max=sh["n_max"], table=table,
                     brick=sh["brick"] if table is not None else 0, grid_res=sh["L"])
    return scene, sh, rng, gen


def _cameras(rng, sh, n, width, height):
    """Oblique cameras: pitch 30-60 degrees, any yaw, near the middle."""
    f = 0.5 * height / math.tan(0.5 * math.radians(sh["fov"]))
    cams = []
    for _ in range(n):
        p, y = math.radians(rng.uniform(30.0, 60.0)), rng.uniform(0.0, 2.0 * math.pi)
        target = np.append(rng.uniform(-sh["look"], sh["look"], 2), 0.0)
        fwd = np.array([math.cos(p) * math.cos(y), math.cos(p) * math.sin(y), -math.sin(p)])
        right = np.cross(fwd, [0.0, 0.0, 1.0])
        right /= np.linalg.norm(right)
        c2w = np.stack([right, np.cross(right, fwd), -fwd, target - sh["dist"] * fwd], 1).astype(np.float32)
        cams.append({"c2w": c2w, "fx": np.float32(f), "fy": np.float32(f), "cx": np.float32(0.5 * width),
                     "cy": np.float32(0.5 * height), "width": width, "height": height})
    return cams


def _rays(rng, gen, sh, n):
    """Rays through random image points of 16 (field) or 64 (city) cameras."""
    city = sh["brick"] > 0
    width, height = (1920, 1080) if city else (256, 256)
    cams = _cameras(rng, sh, 64 if city else 16, width, height)
    c2w = torch.tensor(np.stack([c["c2w"] for c in cams]), device=DEV).double()
    ci = torch.randint(0, len(cams), (n,), device=DEV, generator=gen)
    uv = torch.rand((n, 2), device=DEV, generator=gen, dtype=torch.float64)
    f = float(cams[0]["fx"])
    u = (uv[:, 0] * width - 0.5 * width) / f
    v = -(uv[:, 1] * height - 0.5 * height) / f
    d = torch.einsum("nij,nj->ni", c2w[ci, :, :3], torch.stack([u, v, -torch.ones_like(u)], 1))
    d = d / d.norm(dim=1, keepdim=True)
    return torch.cat([c2w[ci, :, 3], d], 1).float().contiguous()


def _batch(case, rng, gen, sh):
    n, k = case["n"], case["k"]
    rays = _rays(rng, gen, sh, n)
    target = torch.rand((n, 3), device=DEV, generator=gen)
    dirs = None
    if k:
        dirs = rays[:, None, 3:] + torch.empty((n, k, 3), device=DEV).normal_(0.0, math.sqrt(0.3), generator=gen)
    return rays, target, dirs


def _top_down(gen, sh, n):
    """Rays from above the box to the ground (the entropy term's ray set)."""
    x0, x1, y0, y1, z0, z1 = sh["aabb"]
    r = torch.rand((n, 4), device=DEV, generator=gen)
    o = torch.stack([x0 + r[:, 0] * (x1 - x0), y0 + r[:, 1] * (y1 - y0), torch.full((n,), 1.5 * z1 - 0.5 * z0, device=DEV)], 1)
    d = torch.stack([0.4 * r[:, 2] - 0.2, 0.4 * r[:, 3] - 0.2, -torch.ones(n, device=DEV)], 1)
    return torch.cat([o, d / d.norm(dim=1, keepdim=True)], 1).contiguous()


def _points(gen, sh, occ, n):
    """Points in the occupied space (the sparsity term's point set)."""
    x0, x1, y0, y1 = sh["aabb"][:4]
    M = sh["M"]
    live = (occ[..., 0] < occ[..., 1]).reshape(-1).nonzero()[:, 0]
    cell = live[torch.randint(0, live.numel(), (n,), device=DEV, generator=gen)]
    r = torch.rand((n, 3), device=DEV, generator=gen)
    lo, hi = occ.reshape(-1, 2)[cell].unbind(1)
    x = x0 + (cell // M + r[:, 0]) * (x1 - x0) / M
    y = y0 + (cell % M + r[:, 1]) * (y1 - y0) / M
    return torch.stack([x, y, lo + (0.02 + 0.96 * r[:, 2]) * (hi - lo)], 1).contiguous()


# ------------------------------------------------------------------ a case's state and its pass
LAM = (1.0, 1e-2, 1e-4)  # the training configuration's loss weights


def _adam_sizes(case):
    res = case["res"]
    return {"grid": case["bricks"] * 512 * NCH, "p_xy": 16 * res * res * NCH, "p_xz": res * res * NCH,
            "p_yz": res * res * NCH, "occ": res * res // 2, "mlp": MLP_NPARAM}


def _adam_state(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    groups = []
    for name, n in _adam_sizes(case).items():
        g = {k: torch.empty(n, device=DEV).normal_(0.0, s, generator=gen)
             for k, s in (("param", 0.5), ("grad", 1e-4), ("m", 1e-4), ("v", 1e-4))}
        g["v"].square_()
        g["lr"] = 5e-5 if name == "occ" else 1e-2
        if case["dtype"] == "bf16" and name not in ("occ", "mlp"):
            g["shadow"] = g["param"].to(torch.bfloat16)
        groups.append(g)
    return groups


def prepare(case, seed):
    kind = case["kind"]
    if kind == "adam":
        return {"case": case, "groups": _adam_state(case, seed)}
    scene, sh, rng, gen = _make_scene(case, seed, dense=kind == "export")
    st = {"case": case, "scene": scene, "sh": sh}
    if kind in ("render", "noalloc"):
        st["cams"] = _cameras(rng, sh, case.get("cams", 1), case["width"], case["height"])
        st["rgb"] = torch.empty((case.get("cams", 1) * case["width"] * case["height"], 3), device=DEV)
    elif kind == "rays":
        st["rays"] = _rays(rng, gen, sh, case["n"])
    elif kind in ("train", "autograd", "iteration"):
        st["rays"], st["target"], st["dirs"] = _batch(case, rng, gen, sh)
        if kind == "train":
            st["grads"] = om.zero_grads(scene)
        elif kind == "autograd":
            st["params"] = [getattr(scene, k).requires_grad_(True) for k in _PARAMS]
        else:
            st["points"] = _points(gen, sh, scene.occ, case["points"])
            st["erays"] = _top_down(gen, sh, case["erays"])
            # the usual Adam epsilon (the trainer's 1e-15 turns a gradient that
            # cancels to rounding noise into a full step of either sign)
            st["trainer"] = om.Trainer(scene, eps=1e-8)
    return st


_PARAMS = ("grid", "p_xy", "p_xz", "p_yz", "occ", "mlp")


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "render":
        if case["count"]:
            if case["cams"] == 1:
                return om.render(st["scene"], camera=st["cams"][0])
            return om.render_cameras(st["scene"], st["cams"], out=st["rgb"])
        return om.render_cameras(st["scene"], st["cams"], out=st["rgb"], want_count=False)[0]
    if kind == "noalloc":
        return om.render_noalloc(st["scene"], camera=st["cams"][0], rgb=st["rgb"])[0]
    if kind == "rays":
        return om.render(st["scene"], rays=st["rays"])
    if kind == "train":
        for g in st["grads"].values():
            g.zero_()
        r = om.train_step(st["scene"], st["rays"], st["target"], st["dirs"], lam=LAM, grads=st["grads"])
        return {"loss": r["loss"], "grads": r["grads"]}
    if kind == "autograd":
        loss = om.TrainStep.apply(st["scene"], st["rays"], st["target"], st["dirs"], LAM, *st["params"])
        return {"loss": loss.detach(), "grads": dict(zip(_PARAMS, torch.autograd.grad(loss, st["params"])))}
    if kind == "iteration":
        tr = st["trainer"]
        loss = tr.step(st["rays"], st["target"], st["dirs"], sparsity_points=st["points"], entropy_rays=st["erays"])
        return {"loss": loss, "params": {k: getattr(tr.scene, k) for k in _PARAMS}}
    if kind == "adam":
        om.adam_step(st["groups"], step=100, eps=1e-8)
        return [[g[k] for k in ("param", "m", "v", "shadow") if k in g] for g in st["groups"]]
    # export: the bricks the occupancy plane asks for, the occupancy grid, the cropped planes
    sc, sh = st["scene"], st["sh"]
    table, n = om.build_brick_table(sh["aabb"], sh["L"], 8, sc.occ)
    pool = om.extract_bricks(sh["L"], 8, table, sc.grid, n_bricks=int(n.item()))
    v = case["voxels"]
    bits, count = om.occupancy_grid(sh["aabb"], sc.occ, (v, v, max(v // 16, 1)))
    small = om.crop_planes(sc)
    return {"table": table, "pool": pool, "bits": bits, "count": count, "p_xz": small.p_xz, "p_yz": small.p_yz}


# ------------------------------------------------------------------ what a pass cannot do without
def _scene_bytes(case, grads=False):
    """The stored features, bounds and MLP, each once; with `grads` also the FP32 gradients."""
    sh = _shape(case)
    L, R, M = sh["L"], sh["R"], sh["M"]
    grid = L[0] * L[1] * L[2] * (0.15 if sh["brick"] else 1.0)  # about 15 % of a city's bricks are stored
    texels = grid + R[0] * R[1] + R[0] * R[2] + R[1] * R[2]
    el = 2 if case["dtype"] == "bf16" else 4
    return texels * NCH * (el + (4 if grads else 0)) + M * M * 8 * (2 if grads else 1) + 4 * MLP_NPARAM


def work(case):
    kind = case["kind"]
    if kind == "adam":
        n = sum(_adam_sizes(case).values())
        return {"bytes": n * (30 if case["dtype"] == "bf16" else 28), "flops": 14 * n}
    el = 2 if case["dtype"] == "bf16" else 4
    if kind == "export":
        sh, v = _shape(case), case["voxels"]
        L, R = sh["L"], sh["R"]
        pool = 0.15 * L[0] * L[1] * L[2] * NCH * el
        crop = 2 * R[0] * R[2] * NCH * el * 0.6
        return {"bytes": 2 * pool + v * v * max(v // 16, 1) / 8 + 2 * crop + sh["M"] ** 2 * 8, "flops": 0}
    per_ray = 40 if case["scene"] == "city" else 20  # evaluated samples of a ray
    per_sample = 20 * 2 * NCH + 130  # 20 texels of 8 channels, weights, activations, compositing
    mlp = 2 * 848
    if kind in ("render", "noalloc", "rays"):
        n = case["n"] if kind == "rays" else case.get("cams", 1) * case["width"] * case["height"]
        io = n * (12 + (24 if kind == "rays" else 0) + (4 if kind == "rays" or case.get("count") else 0))
        # a few rays cannot touch the whole scene
        feats = min(_scene_bytes(case), n * per_ray * 20 * NCH * el)
        return {"bytes": feats + io, "flops": n * (per_ray * per_sample + mlp)}
    n, k = case["n"], case["k"]
    feats = min(_scene_bytes(case, True), n * per_ray * 20 * NCH * (el + 4))
    flops = n * (3 * per_ray * per_sample + 3 * (1 + k) * mlp)
    extra = 0
    if kind == "iteration":
        sh = _shape(case)
        params = (sh["L"][0] * sh["L"][1] * sh["L"][2] + 16 * case["res"] ** 2 + 2 * sh["R"][0] * sh["R"][2]) * NCH
        extra = params * 28 + case["points"] * 12 + case["erays"] * 24
    return {"bytes": feats + n * (24 + 12 + 12 * k) + extra, "flops": flops}


# ------------------------------------------------------------------ the same results in 64 bits
# Which lattice samples are evaluated is decided in float32 (the library's
# documented rule); everything computed at them is float64, in plain torch.
class _Field:
    """The scene's arrays in 64 bits, for the reference."""

    def __init__(self, scene, sh, grad=False):
        self.sh, self.occ32, self.table = sh, scene.occ, scene.table
        self.p = {k: getattr(scene, k).detach().double().clone() for k in _PARAMS}
        if grad:
            for v in self.p.values():
                v.requires_grad_(True)
        box = sh["aabb"]
        self.lo, self.hi = ([box[2 * a + b] for a in range(3)] for b in range(2))

    def _coord(self, x, a, n):
        u = ((x - self.lo[a]) * ((n - 1) / (self.hi[a] - self.lo[a]))).clamp(0, n - 1)
        i = u.long().clamp(max=n - 2)
        return i, u - i

    def density_and_colour(self, p):
        """t (8 channels) at the points p [s, 3]."""
        sh = self.sh
        L, R = sh["L"], sh["R"]
        i, f = zip(*(self._coord(p[:, a], a, L[a]) for a in range(3)))
        grid = self.p["grid"].reshape(-1, NCH)
        t = torch.zeros((p.shape[0], NCH), dtype=torch.float64, device=DEV)
        for c in range(8):
            e = [(c >> 2) & 1, (c >> 1) & 1, c & 1]
            v = [i[a] + e[a] for a in range(3)]
            w = math.prod(f[a] if e[a] else 1.0 - f[a] for a in range(3))
            if self.table is None:
                at = (v[0] * L[1] + v[1]) * L[2] + v[2]
            else:
                b = self.table[v[0] >> 3, v[1] >> 3, v[2] >> 3].long()
                w = torch.where(b >= 0, w, torch.zeros_like(w))
                at = ((b.clamp(min=0) * 8 + (v[0] & 7)) * 8 + (v[1] & 7)) * 8 + (v[2] & 7)
            t = t + w[:, None] * grid.index_select(0, at)
        i, f = zip(*(self._coord(p[:, a], a, R[a]) for a in range(3)))
        for name, (u, v) in (("p_xy", (0, 1)), ("p_xz", (0, 2)), ("p_yz", (1, 2))):
            plane = self.p[name].reshape(-1, NCH)
            for c in range(4):
                eu, ev = (c >> 1) & 1, c & 1
                w = (f[u] if eu else 1.0 - f[u]) * (f[v] if ev else 1.0 - f[v])
                t = t + w[:, None] * plane.index_select(0, (i[u] + eu) * R[v] + i[v] + ev)
        return t

    def samples(self, rays):
        """The evaluated lattice samples of float32 rays: ray index, position (float64), occupancy cell."""
        sh = self.sh
        o, d = rays[:, :3], rays[:, 3:]
        live = self.occ32[..., 0] <= self.occ32[..., 1]
        zlo = max(self.lo[2], float(self.occ32[..., 0][live].min()))
        zhi = min(self.hi[2], float(self.occ32[..., 1][live].max()))
        od, dd = o.double(), d.double()
        tin, tout = torch.zeros_like(od[:, 0]), torch.full_like(od[:, 0], math.inf)
        for a, (lo, hi) in enumerate(((self.lo[0], self.hi[0]), (self.lo[1], self.hi[1]), (zlo, zhi))):
            ta, tb = (lo - od[:, a]) / dd[:, a], (hi - od[:, a]) / dd[:, a]
            tin, tout = torch.maximum(tin, torch.minimum(ta, tb)), torch.minimum(tout, torch.maximum(ta, tb))
        k0 = (torch.floor(tin / sh["step"]) - 3).clamp(min=0).long()
        n = torch.where(tin <= tout + 4 * sh["step"], torch.ceil(tout / sh["step"]).nan_to_num(0).long() + 4 - k0, 0).clamp(min=0)
        first = torch.cumsum(n, 0) - n
        ray = torch.repeat_interleave(torch.arange(rays.shape[0], device=DEV), n)
        k = k0[ray] + torch.arange(ray.numel(), device=DEV) - first[ray]
        t = k.float() * sh["step"]
        lo32, hi32 = (torch.tensor(v, dtype=torch.float32, device=DEV) for v in (self.lo, self.hi))
        prod = t[:, None] * d[ray]  # each operation rounded: the decision rule has no fused ones
        p = o[ray] + prod
        ok = ((p >= lo32) & (p <= hi32)).all(1)
        ray, k, p = ray[ok], k[ok], p[ok]
        M = sh["M"]
        c = []
        for a in range(2):
            scale = torch.tensor(float(np.float32(M) / (np.float32(self.hi[a]) - np.float32(self.lo[a]))), dtype=torch.float32, device=DEV)
            c.append(torch.floor((p[:, a] - lo32[a]) * scale).long().clamp(0, M - 1))
        cell = c[0] * M + c[1]
        zb = self.occ32.reshape(-1, 2)[cell]
        ok = (zb[:, 0] < p[:, 2]) & (p[:, 2] < zb[:, 1])
        ray, k, cell = ray[ok], k[ok], cell[ok]
        rank = self._rank(ray, rays.shape[0])
        ok = rank < sh["n_max"]
        ray, k, cell = ray[ok], k[ok], cell[ok]
        return ray, od[ray] + (k.double() * sh["step"])[:, None] * dd[ray], cell

    @staticmethod
    def _rank(ray, n):
        count = torch.bincount(ray, minlength=n)
        return torch.arange(ray.numel(), device=DEV) - (torch.cumsum(count, 0) - count)[ray]

    def opacity(self, p, cell):
        """M alpha and the features t at samples."""
        sh = self.sh
        t = self.density_and_colour(p)
        alpha = -torch.expm1(-torch.exp(t[:, 0]) * sh["step"])
        zb = self.p["occ"].reshape(-1, 2).index_select(0, cell)
        rl, rh = (p[:, 2] - zb[:, 0]) / sh["eps"], (zb[:, 1] - p[:, 2]) / sh["eps"]
        M = torch.minimum(torch.minimum(rl * rl, rh * rh), torch.ones_like(rl))
        return M * alpha, t

    def march(self, rays, thr=1e-4):
        """F [n, 7], T [n], sample count [n] of rays."""
        n = rays.shape[0]
        with torch.no_grad():
            ray, p, cell = self.samples(rays)
            ah, _ = self.opacity(p, cell)
            lg = torch.log1p(-ah)
            before = self._before(lg, ray, n)
            keep = torch.exp(before) >= thr  # a ray stops after the sample that takes T below the threshold
            ray, p, cell = ray[keep], p[keep], cell[keep]
        ah, t = self.opacity(p, cell)
        lg = torch.log1p(-ah)
        w = torch.exp(self._before(lg, ray, n)) * ah
        F = torch.zeros((n, 7), dtype=torch.float64, device=DEV).index_add(0, ray, w[:, None] * torch.sigmoid(t[:, 1:]))
        T = torch.exp(torch.zeros(n, dtype=torch.float64, device=DEV).index_add(0, ray, lg))
        return F, T, torch.bincount(ray, minlength=n)

    @staticmethod
    def _before(lg, ray, n):
        """log T before each sample (samples in ray order)."""
        if lg.numel() == 0:
            return lg
        c = torch.cumsum(lg, 0) - lg
        count = torch.bincount(ray, minlength=n)
        first = torch.cumsum(count, 0) - count
        return c - c[first.clamp(max=lg.numel() - 1)[ray]]

    def mlp(self, F, d):
        W = self.p["mlp"]
        x = [F, d]
        for k in range(4):
            x += [torch.sin(2.0 ** k * d), torch.cos(2.0 ** k * d)]
        h = torch.relu(torch.cat(x, 1) @ W[:544].view(16, 34).T + W[544:560])
        h = torch.relu(h @ W[560:816].view(16, 16).T + W[816:832])
        return torch.sigmoid(h @ W[832:880].view(3, 16).T + W[880:883])

    def pixels(self, rays):
        F, T, count = self.march(rays)
        live = (count > 0)[:, None]
        return F[:, :3] + torch.where(live, self.mlp(F, rays[:, 3:].double()), torch.zeros_like(F[:, :3])), F, T, count


def _camera_rays(cam):
    """Pinhole rays in float32, every operation rounded (the library's documented rule)."""
    w, h = cam["width"], cam["height"]
    c2w = torch.tensor(cam["c2w"], device=DEV)
    f = {k: torch.tensor(float(cam[k]), dtype=torch.float32, device=DEV) for k in ("fx", "fy", "cx", "cy")}
    px = torch.arange(w, device=DEV).float().repeat(h)
    py = torch.arange(h, device=DEV).float().repeat_interleave(w)
    u, v = (px + 0.5 - f["cx"]) / f["fx"], -((py + 0.5 - f["cy"]) / f["fy"])
    d = []
    for a in range(3):
        x, y = c2w[a, 0] * u, c2w[a, 1] * v
        d.append((x + y) + c2w[a, 2] * -1.0)
    q = [x * x for x in d]
    norm = torch.sqrt((q[0] + q[1]) + q[2])
    return torch.stack([c2w[a, 3].expand(w * h) for a in range(3)] + [x / norm for x in d], 1)


CHUNK = 1 << 16


def _exact_loss(f, rays, target, dirs, lam):
    """Adds the gradients of the training loss to f.p's; the four loss values."""
    n = rays.shape[0]
    total = torch.zeros(4, dtype=torch.float64, device=DEV)
    for c in range(0, n, CHUNK // 4):
        r, tg = rays[c:c + CHUNK // 4], target[c:c + CHUNK // 4].double()
        d = r[:, 3:].double()
        rgb, F, _, count = f.pixels(r)
        l_rgb = lam[0] / n * torch.sqrt((rgb - tg).square().sum(1) + 1e-6).sum()
        l_s = torch.zeros((), dtype=torch.float64, device=DEV)
        live = count > 0
        yd = f.mlp(F, d)
        for k in range(0 if dirs is None else dirs.shape[1]):
            s = dirs[c:c + CHUNK // 4, k].double()
            cos = (d * s).sum(1) / (d.norm(dim=1) * s.norm(dim=1))
            q = (f.mlp(F, s / s.norm(dim=1, keepdim=True)) - yd).square().sum(1)
            l_s = l_s + lam[1] / n * (cos * q)[live].sum()
        (l_rgb + l_s).backward()
        total[1] += l_rgb.detach()
        total[2] += l_s.detach()
    span = lam[2] * (f.p["occ"][..., 1] - f.p["occ"][..., 0]).square().sum()
    span.backward()
    total[3] = span.detach()
    total[0] = total[1:].sum()
    return total


def _exact_regularisers(f, points, erays, lam_s, lam_e):
    t0 = f.density_and_colour(points.double())[:, 0]
    loss = lam_s * -torch.expm1(-torch.exp(t0) * f.sh["step"]).mean()
    ray, p, cell = f.samples(erays)
    a, _ = f.opacity(p, cell)
    S = torch.zeros(erays.shape[0], dtype=torch.float64, device=DEV).index_add(0, ray, a)
    q = a / S[ray]
    loss = loss + lam_e * -(torch.xlogy(q, q)).sum() / erays.shape[0]
    loss.backward()
    return loss.detach()


def exact(case, seed):
    kind = case["kind"]
    if kind == "adam":
        out = []
        b1, b2, eps, t = 0.9, 0.99, 1e-8, 100
        for g in _adam_state(case, seed):
            p, d, m, v = (g[k].double() for k in ("param", "grad", "m", "v"))
            m, v = b1 * m + (1 - b1) * d, b2 * v + (1 - b2) * d * d
            p = p - g["lr"] / (1 - b1 ** t) * m / (torch.sqrt(v / (1 - b2 ** t)) + eps)
            out.append([p, m, v] + ([p] if "shadow" in g else []))
        return out
    if kind == "export":
        return None  # copies and bits: nothing is rounded
    st = prepare(case, seed)
    if kind in ("render", "noalloc", "rays"):
        f = _Field(st["scene"], st["sh"])
        every = [st["rays"]] if kind == "rays" else [_camera_rays(c) for c in st["cams"]]
        rgb = torch.cat([f.pixels(r[c:c + CHUNK])[0] for r in every for c in range(0, r.shape[0], CHUNK)])
        return (rgb, None) if kind == "rays" or case.get("count") else rgb
    f = _Field(st["scene"], st["sh"], grad=True)
    if kind != "iteration":
        loss = _exact_loss(f, st["rays"], st["target"], st["dirs"], LAM)
        return {"loss": loss if kind == "train" else loss[0], "grads": {k: v.grad for k, v in f.p.items()}}
    loss = _exact_loss(f, st["rays"], st["target"], st["dirs"], (1.0, 0.1, 0.0))
    loss[0] += _exact_regularisers(f, st["points"], st["erays"], 0.05, 1e-3)
    new = {}
    for k, p in f.p.items():
        lr = 5e-5 if k == "occ" else 1e-2
        new[k] = p.detach() - lr * p.grad / (p.grad.abs() + 1e-8)
    return {"loss": loss, "params": new}
