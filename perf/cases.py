"""The work that users of this framework have it do, as measurable cases.

``listed()`` names twelve cases over the paths of the library: whole renders
(single view, panorama, stereo pair, large scene), training steps
(tensor-core and default precision), distillation (whole step in the default
precision, the teacher alone), direct point queries, and the steps around
them (occupancy update, field assignment, compositing).  ``draw(rng)`` gives
another case of the same ranges.  Inputs are made on the GPU from the seed;
``exact`` restates each path in plain FP64 torch.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

import paper_2208_02705_gb300 as roam
from paper_2208_02705_gb300.roaming import stereo_pair

PEX, PED = 63, 27                # encoded position and direction features
PRECISION = {"f32": roam.ROAM_F32, "bf16": roam.ROAM_BF16, "fp8": roam.ROAM_FP8}
SAMPLES_PER_RAY = 20             # composited samples per ray of these scenes, about


def _mapped(grid):
    """Occupied voxels of a mapped floor: most of its surfaces, whatever the furniture."""
    return int(grid ** 2 * (2.5 if grid < 96 else 3.3 if grid < 128 else 6.0 if grid < 192 else 7.6))


def listed():
    return [
        # a thumbnail of one room in the options' default precision (FP32): the
        # smallest render, where launches and latency count
        dict(name="thumbnail_f32", kind="render", grid=32, fields=8, W=32, H=2, model=0, width=128, height=64,
             views=1, precision="f32", n_max=64, graph=False, stereo=False),
        # one panorama of a floor in the tensor-core precision: the ordinary render
        dict(name="panorama_bf16", kind="render", grid=256, fields=512, W=64, H=3, model=0, width=1024, height=512,
             views=1, precision="bf16", n_max=128, graph=False, stereo=False),
        # one frame of stereoscopic roaming: both eyes of a pose at 720p, fields
        # of mixed widths, replayed as a CUDA graph into the same buffers
        dict(name="stereo_frame_mixed", kind="render", grid=256, fields=512, W=0, H=3, model=1, width=1280, height=720,
             views=1, precision="bf16", n_max=128, graph=True, stereo=True),
        # the large scene: thousands of wide fields, the quantised precision
        dict(name="large_panorama_fp8", kind="render", grid=512, fields=4096, W=128, H=4, model=0, width=2048,
             height=1024, views=1, precision="fp8", n_max=192, graph=False, stereo=False),
        # a fine-tuning step on a large ray batch: forward, loss, adjoint, Adam
        dict(name="finetune_bf16", kind="finetune", grid=256, fields=512, W=64, H=3, views=16, width=1024, height=512,
             rays=65536, precision="bf16", n_max=128),
        # a step through torch.autograd with the caller's own optimizer, default
        # precision, the paper's batch of 4096 rays per process
        dict(name="autograd_f32", kind="autograd", grid=256, fields=512, W=64, H=3, views=4, width=512, height=256,
             rays=4096, precision="f32", n_max=128),
        # a distillation step in the default precision: teacher, students, loss,
        # adjoint, Adam
        dict(name="distill_f32", kind="distill", grid=256, fields=512, W=64, H=3, per_field=64, precision="f32"),
        # the teacher alone on the tensor cores, as for targets made ahead
        dict(name="teacher_bf16", kind="teacher", points=131072, precision="bf16"),
        # a ragged set of points queried directly (probing the field)
        dict(name="points_bf16", kind="points", grid=128, fields=64, W=64, H=3, points=20011, precision="bf16"),
        # one occupancy update from four panoramic depth scans
        dict(name="occupancy_scans", kind="occupancy", grid=256, views=4, model=0, width=1024, height=512),
        # the assignment of a floor's voxels to its networks
        dict(name="assign_fields", kind="assign", grid=256, fields=256, voxels=_mapped(256)),
        # compositing of the caller's own samples
        dict(name="composite_rays", kind="composite", rays=100003, n_max=64),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["render", "render", "finetune", "autograd", "distill", "teacher", "points", "occupancy",
                       "assign", "composite"])
    grid = 32 * rng.randint(2, 8)
    fields = log_int(8, 512)
    W, H = rng.choice([(32, 2), (32, 4), (64, 1), (64, 2), (64, 3)])
    if kind == "render":
        prec = rng.choice(["f32", "bf16", "bf16", "fp8"])
        if prec != "f32" and rng.random() < 0.3:
            W, H = rng.choice([(128, 3), (0, 3)])
        model = rng.randint(0, 1)
        width = log_int(64, 512 if prec == "f32" else 1024)
        return dict(kind=kind, grid=grid, fields=fields, W=W, H=H, model=model, width=width,
                    height=max(32, width // 2 + rng.randint(-9, 9)), views=rng.randint(1, 2), precision=prec,
                    n_max=rng.choice([32, 64, 100, 128]), graph=rng.random() < 0.3, stereo=False)
    if kind in ("finetune", "autograd"):
        return dict(kind=kind, grid=grid, fields=fields, W=W, H=H, views=rng.randint(1, 8), width=512, height=256,
                    rays=log_int(500, 10000), precision=rng.choice(["f32", "bf16"]), n_max=rng.choice([64, 128]))
    if kind == "distill":
        return dict(kind=kind, grid=grid, fields=fields, W=W, H=H, per_field=log_int(20, 64),
                    precision=rng.choice(["f32", "bf16"]))
    if kind == "teacher":
        prec = rng.choice(["f32", "bf16"])
        return dict(kind=kind, points=log_int(1000, 30000 if prec == "f32" else 300000), precision=prec)
    if kind == "points":
        W = rng.choice([32, 64, 128])
        return dict(kind=kind, grid=grid, fields=fields, W=W, H=3, points=log_int(1000, 300000),
                    precision=rng.choice(["f32", "bf16", "fp8"]))
    if kind == "occupancy":
        width = log_int(64, 1024)
        return dict(kind=kind, grid=grid, views=rng.randint(1, 4), model=rng.randint(0, 1), width=width,
                    height=max(32, width // 2 + rng.randint(-9, 9)))
    if kind == "assign":
        return dict(kind=kind, grid=grid, fields=log_int(8, 256), voxels=_mapped(grid))
    return dict(kind=kind, rays=log_int(1000, 100000), n_max=rng.choice([16, 50, 64, 128]))


# ---- inputs ----------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float32)


@dataclasses.dataclass
class _Camera:
    model: int
    width: int
    height: int
    fov_h: float
    R: np.ndarray
    o: np.ndarray


class _Scene:
    """A floor of rooms in a cubic grid: slabs, walls with doors, furniture;
    occupied voxels split into fields of equal voxel counts (a kd tree)."""

    def __init__(self, G, n_fields, seed):
        rng = np.random.default_rng([int(seed), G])
        self.G = G
        self.vox = 8.0 / G
        occ = torch.zeros((G, G, G), dtype=torch.bool, device="cuda")       # [z][y][x]
        m = max(2, G // 16)
        wall = 1 if G < 128 else 2
        h = max(G // 3, 12)
        y0, y1 = (G - h) // 2, (G - h) // 2 + h
        nx, nz = (1, 1) if G < 96 else ((2, 2) if G < 192 else ((4, 2) if G < 384 else (5, 4)))
        xs = np.linspace(m, G - m, nx + 1).round().astype(int)
        zs = np.linspace(m, G - m, nz + 1).round().astype(int)
        occ[m:G - m, y1 - wall:y1, m:G - m] = True
        occ[m:G - m, y0:y0 + wall, m:G - m] = True
        for i, x in enumerate(xs):
            a = x if i == 0 else x - wall
            occ[m:G - m, y0:y1, a:a + wall] = True
        for k, z in enumerate(zs):
            a = z if k == 0 else z - wall
            occ[a:a + wall, y0:y1, m:G - m] = True
        door = max(4, G // 24)
        for i in range(1, nx):
            for k in range(nz):
                c = int(rng.integers(zs[k] + wall + door, zs[k + 1] - wall - door))
                occ[c - door // 2:c + door // 2, y1 - wall - int(0.6 * h):y1 - wall, xs[i] - wall:xs[i] + wall] = False
        for k in range(1, nz):
            for i in range(nx):
                c = int(rng.integers(xs[i] + wall + door, xs[i + 1] - wall - door))
                occ[zs[k] - wall:zs[k] + wall, y1 - wall - int(0.6 * h):y1 - wall, c - door // 2:c + door // 2] = False
        self.rooms = []
        for i in range(nx):
            for k in range(nz):
                lo = np.array([xs[i] + wall, y0 + wall, zs[k] + wall])
                hi = np.array([xs[i + 1] - wall, y1 - wall, zs[k + 1] - wall])
                self.rooms.append((lo, hi))
                for _ in range(5):
                    # furniture along the walls: the room's middle stays free
                    s = rng.integers(G // 48 + 2, G // 16 + 3, size=3)
                    ax = int(rng.integers(0, 2)) * 2
                    p = np.array([int(rng.integers(lo[q], max(lo[q] + 1, hi[q] - s[q]))) for q in range(3)])
                    p[ax] = lo[ax] if rng.random() < 0.5 else hi[ax] - min(s[ax], (hi[ax] - lo[ax]) // 5)
                    p[1] = hi[1] - s[1]
                    e = np.minimum(p + s, hi)
                    occ[p[2]:e[2], p[1]:e[1], p[0]:e[0]] = True
                    mid0, mid1 = lo + (hi - lo) // 4, hi - (hi - lo) // 4
                    occ[mid0[2]:mid1[2], mid0[1]:mid1[1], mid0[0]:mid1[0]] = False
        self.occ = occ
        self.rng = rng
        self.pack()
        zyx = occ.nonzero()                                   # linear order, x fastest
        self.xyz = zyx.flip(1).contiguous()                   # [S][3]
        self.fields = n_fields
        S = self.xyz.shape[0]
        # kd labels: split the largest parts along their longest axis until there
        # are n_fields of them, equal shares of voxels (by rank along the axis)
        lab = torch.zeros(S, dtype=torch.int64, device="cuda")
        parts, share = 1, np.array([n_fields])
        while parts < n_fields:
            lo = torch.full((parts, 3), G, device="cuda").scatter_reduce(0, lab[:, None].expand(-1, 3), self.xyz, "amin")
            hi = torch.zeros((parts, 3), dtype=torch.int64, device="cuda").scatter_reduce(
                0, lab[:, None].expand(-1, 3), self.xyz, "amax")
            axis = (hi - lo).argmax(1)
            c = self.xyz.gather(1, axis[lab][:, None])[:, 0]
            key = (lab * G + c) * S + torch.arange(S, device="cuda")
            order = key.argsort()
            count = torch.bincount(lab, minlength=parts)
            start = count.cumsum(0) - count
            pos = torch.empty_like(lab)
            pos[order] = torch.arange(S, device="cuda")
            pos -= start[lab]
            left = share // 2
            cut = count * torch.from_numpy(left).cuda() // torch.from_numpy(share).cuda()
            right = pos >= cut[lab]
            # children of a part keep its place; a part of one field is not split
            n_child = np.where(share > 1, 2, 1)
            first = torch.from_numpy(np.cumsum(n_child) - n_child).cuda()
            split = torch.from_numpy(share > 1).cuda()
            lab = first[lab] + (right & split[lab]).to(torch.int64)
            share = np.concatenate([[s // 2, s - s // 2] if s > 1 else [s] for s in share])
            parts = len(share)
        self.lab = lab
        lo = torch.full((n_fields, 3), G, device="cuda").scatter_reduce(0, lab[:, None].expand(-1, 3), self.xyz, "amin")
        hi = torch.zeros((n_fields, 3), dtype=torch.int64, device="cuda").scatter_reduce(
            0, lab[:, None].expand(-1, 3), self.xyz, "amax") + 1
        lo, hi = lo.double() * self.vox, hi.double() * self.vox
        scale = 2.0 / (hi - lo)
        self.affine = torch.cat([scale, -1.0 - lo * scale], 1).float().contiguous()
        self.delta = self.vox / 4
        # a sample of density logit 0 has opacity 0.3 over one step
        self.sigma = -math.log(0.7) / (self.delta * math.log(2.0))

    def pack(self):
        G = self.G
        words = self.occ.view(G, G, G // 32, 32).to(torch.int64) << torch.arange(32, device="cuda")
        self.bits = words.sum(-1).to(torch.int32).contiguous()

    def keep(self, n, g):
        """Leaves n occupied voxels: a map has holes where no scan saw the surface."""
        gone = self.xyz[torch.randperm(self.xyz.shape[0], generator=g, device="cuda")[n:]]
        self.occ[gone[:, 2], gone[:, 1], gone[:, 0]] = False
        self.pack()

    def camera(self, model, width, height):
        rng = self.rng
        lo, hi = self.rooms[int(rng.integers(len(self.rooms)))]
        o = (lo + (hi - lo) * rng.uniform(0.3, 0.7, 3)) * self.vox
        a, p = rng.uniform(0, 2 * math.pi), rng.uniform(-0.15, 0.15)
        Ry = np.array([[math.cos(a), 0, math.sin(a)], [0, 1, 0], [-math.sin(a), 0, math.cos(a)]])
        Rx = np.array([[1, 0, 0], [0, math.cos(p), -math.sin(p)], [0, math.sin(p), math.cos(p)]])
        # as the library takes them: FP32 values
        return _Camera(model, width, height, math.pi / 2, (Ry @ Rx).astype(np.float32).astype(np.float64),
                       o.astype(np.float32).astype(np.float64))

    def load_geometry(self, r):
        r.load_grid(self.bits, (self.G,) * 3, (0.0, 0.0, 0.0), self.vox)
        r.load_fields(self.lab.to(torch.int16), self.affine)


def _shapes(W, H):
    return [(W, PEX)] + [(W, W)] * (H - 1) + [(1 + W, W), (W, W + PED), (3, W)]


def _teacher_shapes():
    return ([(256, PEX)] + [(256, 256)] * 3 + [(256, 256 + PEX)] + [(256, 256)] * 3 +
            [(1, 256), (256, 256), (128, 256 + PED), (3, 128)])


def _weights(g, shapes, n):
    """[n][P]: Xavier-uniform matrices and small biases, layer after layer."""
    amp = torch.cat([torch.cat([torch.full((o * i,), math.sqrt(6.0 / (o + i))), torch.full((o,), 0.05)])
                     for o, i in shapes]).cuda()
    w = _uniform(g, n, amp.numel())
    return w.mul_(2.0).sub_(1.0).mul_(amp)


def _mixed_widths(seed, n):
    return np.random.default_rng([int(seed), 7]).choice([32, 64, 128], n).astype(np.int32)


def _field_weights(case, seed):
    g = _gen(seed + 1)
    if case["W"]:
        return _weights(g, _shapes(case["W"], case["H"]), case["fields"])
    widths = _mixed_widths(seed, case["fields"])
    by_width = {W: iter(_weights(g, _shapes(W, case["H"]), int((widths == W).sum()))) for W in (32, 64, 128)}
    return [next(by_width[int(W)]) for W in widths]


def _load_weights(r, case, seed, sc):
    if case["W"]:
        w = _field_weights(case, seed)
        r.load_weights(w, case["W"], case["H"], sc.sigma)
        return w
    widths = _mixed_widths(seed, case["fields"])
    r.load_weights_mixed(torch.cat(_field_weights(case, seed)), widths, case["H"], sc.sigma)
    return None


def _points(sc, g, per_voxel_index):
    """Points uniform in the given occupied voxels, uniform directions, their fields."""
    n = per_voxel_index.numel()
    p = (sc.xyz[per_voxel_index].float() + _uniform(g, n, 3)) * sc.vox
    d = torch.randn(n, 3, generator=g, device="cuda")
    d = d / d.norm(dim=1, keepdim=True)
    return p.contiguous(), d.contiguous(), sc.lab[per_voxel_index].to(torch.int16).contiguous()


def _cameras(case, sc):
    cams = [sc.camera(case.get("model", 0), case["width"], case["height"]) for _ in range(case["views"])]
    if case.get("stereo"):
        cams = [e for c in cams for e in stereo_pair(c)]
        for e in cams:
            e.o = e.o.astype(np.float32).astype(np.float64)
    return cams


def _ray_batch(case, seed):
    g = _gen(seed + 2)
    n, pix = case["rays"], case["width"] * case["height"]
    rays = torch.stack([torch.randint(0, case["views"], (n,), generator=g, device="cuda"),
                        torch.randint(0, pix, (n,), generator=g, device="cuda")], 1).to(torch.int32).contiguous()
    return rays, _uniform(g, n, 3)


def _distill_inputs(case, sc, seed):
    g = _gen(seed + 2)
    order = sc.lab.argsort(stable=True)
    count = torch.bincount(sc.lab, minlength=case["fields"])
    start = count.cumsum(0) - count
    u = torch.rand(case["fields"], case["per_field"], generator=g, device="cuda", dtype=torch.float64)
    pick = start[:, None] + (u * count[:, None]).long().clamp_(max=(count - 1).clamp(min=0)[:, None])
    return _points(sc, g, order[pick.reshape(-1)])


def _teacher_inputs(case, seed):
    g = _gen(seed)
    w = _weights(g, _teacher_shapes(), 1)[0]
    aff = np.array([0.25, 0.25, 0.25, -1.0, -1.0, -1.0], dtype=np.float32)
    p = _uniform(g, case["points"], 3) * 8.0
    d = torch.randn(case["points"], 3, generator=g, device="cuda")
    return w, aff, p, (d / d.norm(dim=1, keepdim=True)).contiguous()


def _scan_inputs(case, seed, sc, cams):
    """Depth and opacity maps as a render of the rooms gives them: the way to
    the room's walls, furniture in front of some of it, pixels that saw little."""
    g = _gen(seed + 2)
    depth, opacity = [], []
    for c in cams:
        d = _directions(c, torch.arange(c.width * c.height, device="cuda"))
        o = torch.from_numpy(c.o).cuda()
        lo, hi = next((lo, hi) for lo, hi in sc.rooms if np.all(c.o / sc.vox >= lo) and np.all(c.o / sc.vox <= hi))
        far = torch.where(d > 0, torch.from_numpy(hi).cuda() * sc.vox - o, o - torch.from_numpy(lo).cuda() * sc.vox)
        t = (far / d.abs().clamp(min=1e-9)).amin(1) + 0.5 * sc.vox
        n = t.numel()
        block = torch.rand((c.height + 15) // 16, (c.width + 15) // 16, generator=g, device="cuda")
        block = block.repeat_interleave(16, 0)[:c.height].repeat_interleave(16, 1)[:, :c.width].reshape(-1)
        t = torch.where(block < 0.3, t * (0.5 + block), t)
        a = 1.0 - 0.2 * torch.rand(n, generator=g, device="cuda") ** 2
        a = torch.where(torch.rand(n, generator=g, device="cuda") < 0.05, 0.4 * a, a)
        opacity.append(a.float())
        depth.append((t * a).float())
    return torch.cat(depth).contiguous(), torch.cat(opacity).contiguous()


def _composite_inputs(case, seed):
    g = _gen(seed)
    n, k = case["rays"], case["n_max"]
    count = torch.randint(0, k + 1, (n,), generator=g, device="cuda", dtype=torch.int32)
    sr = _uniform(g, n, k, 4)
    sr[..., 0] = sr[..., 0] ** 3 * 150.0
    t = (torch.cumsum(_uniform(g, n, k), 1) * 0.05).contiguous()
    return count, sr.contiguous(), t


def prepare(case, seed):
    kind = case["kind"]
    r = roam.Roam(0)
    s = {"kind": kind, "roam": r}
    if kind == "teacher":
        w, aff, s["p"], s["d"] = _teacher_inputs(case, seed)
        r.teacher_load(w, aff)
        s["precision"] = PRECISION[case["precision"]]
        return s
    if kind == "composite":
        s["count"], s["sr"], s["t"] = _composite_inputs(case, seed)
        s["opts"] = roam.render_opts(0.01, case["n_max"], bg=(0.1, 0.2, 0.3))
        return s
    sc = _Scene(case["grid"], case.get("fields", 8), seed)
    if kind in ("occupancy", "assign"):
        if kind == "assign":
            sc.keep(case["voxels"], _gen(seed + 2))
        r.load_grid(sc.bits, (sc.G,) * 3, (0.0, 0.0, 0.0), sc.vox)
        s["fields"] = case.get("fields")
        if kind == "occupancy":
            s["cams"] = _cameras(case, sc)
            s["depth"], s["opacity"] = _scan_inputs(case, seed, sc, s["cams"])
            s["logit"] = torch.zeros(sc.G ** 3, device="cuda")
            s["bits"] = torch.zeros(sc.G ** 3 // 32, dtype=torch.int32, device="cuda")
        return s
    sc.load_geometry(r)
    w = _load_weights(r, case, seed, sc)
    s["precision"] = PRECISION[case["precision"]]
    if kind == "render":
        s["cams"] = _cameras(case, sc)
        s["opts"] = roam.render_opts(sc.delta, case["n_max"], precision=s["precision"], use_graph=case["graph"])
        n = sum(c.width * c.height for c in s["cams"])
        s["rgb"] = torch.empty((n, 3), device="cuda")
        s["depth"] = torch.empty(n, device="cuda")
        s["opacity"] = torch.empty(n, device="cuda")
    elif kind in ("finetune", "autograd"):
        s["cams"] = _cameras(case, sc)
        s["rays"], s["target"] = _ray_batch(case, seed)
        s["opts"] = roam.render_opts(sc.delta, case["n_max"], precision=s["precision"])
        s["step"] = 0
        if kind == "autograd":
            s["function"] = roam.render_function()
            s["weights"] = w.requires_grad_(True)
    elif kind == "distill":
        s["p"], s["d"], s["field"] = _distill_inputs(case, sc, seed)
        s["per_field"] = float(case["per_field"])
        tw = _weights(_gen(seed + 3), _teacher_shapes(), 1)[0]
        r.teacher_load(tw, np.array([0.25, 0.25, 0.25, -1.0, -1.0, -1.0], dtype=np.float32))
        s["step"] = 0
    else:
        g = _gen(seed + 2)
        pick = torch.randint(0, sc.xyz.shape[0], (case["points"],), generator=g, device="cuda")
        s["p"], s["d"], s["field"] = _points(sc, g, pick)
    return s


# ---- one pass --------------------------------------------------------------


def run(s):
    kind, r = s["kind"], s["roam"]
    if kind == "render":
        rgb, depth, opacity = r.render(s["cams"], s["opts"], s["rgb"], s["depth"], s["opacity"])
        return {"rgb": rgb, "depth": depth, "opacity": opacity}
    if kind == "finetune":
        s["step"] += 1
        loss, grad = r.local_grad(s["cams"], s["rays"], s["target"], s["opts"], 3.0 * s["rays"].shape[0])
        r.adam_step(grad, lr=1e-6, step=s["step"])
        return {"loss": loss, "grad": grad}
    if kind == "autograd":
        w = s["weights"]
        w.grad = None
        rgb = s["function"].apply(w, r, s["cams"], s["rays"], s["opts"])
        loss = ((rgb - s["target"]) ** 2).mean()
        loss.backward()
        with torch.no_grad():
            w.add_(w.grad, alpha=-1e-4)
        return {"rgb": rgb.detach(), "loss": loss.detach(), "grad": w.grad}
    if kind == "distill":
        s["step"] += 1
        prec = s["precision"]
        t = r.teacher_eval(s["p"], s["d"], prec)
        st = r.mlp_eval(s["p"], s["d"], s["field"], prec)
        loss, dl = r.distill_loss(st, t, s["per_field"])
        grad = r.mlp_backward(s["p"], s["d"], s["field"], dl, precision=prec)
        r.adam_step(grad, lr=1e-6, step=s["step"])
        return {"teacher": t, "student": st, "loss": loss, "grad": grad}
    if kind == "teacher":
        return r.teacher_eval(s["p"], s["d"], s["precision"])
    if kind == "points":
        return r.mlp_eval(s["p"], s["d"], s["field"], s["precision"])
    if kind == "occupancy":
        logit, bits = r.occupancy_update(s["cams"], s["depth"], s["opacity"], s["logit"], s["bits"])
        return {"logit": logit, "bits": bits}
    if kind == "assign":
        labels, boxes = r.assign_fields(s["fields"])
        return {"labels": labels, "boxes": boxes}
    rgb, depth, opacity, used = r.composite(s["count"], s["sr"], s["t"], s["opts"])
    return {"rgb": rgb, "depth": depth, "opacity": opacity, "used": used}


def _macs(W, H):
    return sum(o * i for o, i in _shapes(W, H))


def work(case):
    kind = case["kind"]
    if kind == "teacher":
        return {"bytes": case["points"] * 40 + 4 * 595844,
                "flops": 2 * case["points"] * sum(o * i for o, i in _teacher_shapes())}
    if kind == "composite":
        return {"bytes": case["rays"] * (4 + 24 + 10 * case["n_max"]), "flops": case["rays"] * case["n_max"] * 8}
    vox = case["grid"] ** 3
    if kind == "occupancy":
        pix = case["views"] * case["width"] * case["height"]
        return {"bytes": 8 * pix + 8 * vox + vox // 8, "flops": pix * case["grid"] * 3}
    if kind == "assign":
        return {"bytes": vox // 8 + 2 * case["voxels"] + 24 * case["fields"], "flops": case["voxels"] * 8}
    W, H = case["W"] or 64, case["H"]
    macs = _macs(W, H)
    params = case["fields"] * sum(o * i + o for o, i in _shapes(W, H))
    # every pass over the samples: forward 2, adjoint 2 (weights) + 2 (inputs)
    # + the recomputed forward 2 per multiply
    if kind == "points":
        return {"bytes": case["points"] * 42 + 4 * params, "flops": 2 * macs * case["points"]}
    if kind == "render":
        n = case["views"] * (2 if case["stereo"] else 1) * case["width"] * case["height"]
        return {"bytes": 20 * n + vox // 8 + 4 * params, "flops": 2 * macs * n * SAMPLES_PER_RAY}
    if kind == "distill":
        n = case["fields"] * case["per_field"]
        return {"bytes": n * 42 + 32 * params, "flops": n * (8 * macs + 2 * 595844)}
    n = case["rays"]
    return {"bytes": n * 32 + vox // 8 + (32 if kind == "finetune" else 12) * params,
            "flops": 8 * macs * n * SAMPLES_PER_RAY}


# ---- the same in FP64 ------------------------------------------------------


def _directions(cam, pix):
    """World directions (FP64) of pixels: Eq. 2-3 of the paper, or a pinhole."""
    u, v = (pix % cam.width).double(), (pix // cam.width).double()
    if cam.model == 0:
        phi = 2 * math.pi * ((u + 0.5) / cam.width - 0.5)
        th = math.pi * (0.5 - (v + 0.5) / cam.height)
        d = torch.stack([th.cos() * phi.sin(), -th.sin(), th.cos() * phi.cos()], 1)
    else:
        # (the library's field of view is an FP32 number)
        f = math.tan(0.5 * float(np.float32(cam.fov_h))) / (0.5 * cam.width)
        d = torch.stack([(u + 0.5 - 0.5 * cam.width) * f, (v + 0.5 - 0.5 * cam.height) * f, torch.ones_like(u)], 1)
        d = d / d.norm(dim=1, keepdim=True)
    return d @ torch.from_numpy(np.ascontiguousarray(cam.R.T)).cuda()


def _encode(x, L):
    e = [x]
    for k in range(L):
        a = torch.remainder(x * float(2 ** k), 2.0) * math.pi
        e += [a.sin(), a.cos()]
    return torch.cat(e, 1)


def _split(w, shapes):
    out, at = [], 0
    for o, i in shapes:
        out.append((w[at:at + o * i].view(o, i), w[at + o * i:at + o * i + o]))
        at += o * i + o
    return out


def _mlp64(wf, W, H, x, d, sigma):
    """One field's outputs at local positions x and directions d (all FP64)."""
    L = _split(wf, _shapes(W, H))
    h = _encode(x, 10)
    for A, b in L[:H]:
        h = torch.relu(torch.addmm(b, h, A.T))
    s = torch.addmm(L[H][1], h, L[H][0].T)
    g = torch.relu(torch.addmm(L[H + 1][1], torch.cat([s[:, 1:], _encode(d, 4)], 1), L[H + 1][0].T))
    c = torch.sigmoid(torch.addmm(L[H + 2][1], g, L[H + 2][0].T))
    return torch.cat([sigma * torch.nn.functional.softplus(s[:, :1]), c], 1)


def _fields64(case, w, affine, sigma, p, d, field):
    """Every field's points through its own MLP; keeps autograd's graph."""
    out = torch.empty((p.shape[0], 4), dtype=torch.float64, device="cuda")
    order = field.long().argsort(stable=True)
    ends = torch.bincount(field.long(), minlength=len(w)).cumsum(0).tolist()
    pieces, at, a64 = [], 0, affine.double()
    for f, end in enumerate(ends):
        if end > at:
            i = order[at:end]
            wf = w[f].double()
            W = case["W"] or _width_of(wf.numel(), case["H"])
            pieces.append(_mlp64(wf, W, case["H"], a64[f, :3] * p[i] + a64[f, 3:], d[i], sigma))
        at = end
    if pieces:
        out = out.index_copy(0, order, torch.cat(pieces))
    return out


def _width_of(P, H):
    return next(W for W in (32, 64, 128) if sum(o * i + o for o, i in _shapes(W, H)) == P)


def _teacher64(w, aff, p, d):
    L = _split(w.double(), _teacher_shapes())
    a = torch.from_numpy(aff).cuda().double()
    out = []
    for at in range(0, p.shape[0], 65536):
        x = _encode(a[:3] * p[at:at + 65536].double() + a[3:], 10)
        h = x
        for k in range(8):
            if k == 4:
                h = torch.cat([h, x], 1)
            h = torch.addmm(L[k][1], h, L[k][0].T)
            h = torch.relu(h) if k < 7 else h
        sig = torch.relu(torch.addmm(L[8][1], h, L[8][0].T))
        h = torch.relu(torch.addmm(L[9][1], h, L[9][0].T))
        h = torch.relu(torch.addmm(L[10][1], torch.cat([h, _encode(d[at:at + 65536].double(), 4)], 1), L[10][0].T))
        out.append(torch.cat([sig, torch.sigmoid(torch.addmm(L[11][1], h, L[11][0].T))], 1))
    return torch.cat(out)


def _kept(sc, o, d, n_max):
    """(sample index j, ray) lists of the kept samples, ray after ray, in FP64."""
    n_j = int(math.ceil(sc.G * math.sqrt(3.0) * sc.vox / sc.delta)) + 2
    js, rs = [], []
    step = max(1, 30_000_000 // n_j)
    flat = sc.occ.reshape(-1)
    t = (torch.arange(n_j, device="cuda").double() + 0.5) * float(np.float32(sc.delta))
    vox = float(np.float32(sc.vox))
    for at in range(0, o.shape[0], step):
        idx, inside = None, None
        for a in (2, 1, 0):
            q = torch.floor((o[at:at + step, a:a + 1] + d[at:at + step, a:a + 1] * t) / vox)
            ok = (q >= 0) & (q < sc.G)
            q = q.clamp_(0, sc.G - 1).int()
            idx = q if idx is None else idx * sc.G + q
            inside = ok if inside is None else inside & ok
        keep = inside & flat[idx.long()]
        keep &= keep.cumsum(1, dtype=torch.int32) <= n_max
        r, j = keep.nonzero(as_tuple=True)
        js.append(j)
        rs.append(r + at)
    return torch.cat(js), torch.cat(rs)


def _rays64(case, sc, cams, rays):
    if rays is None:
        o = torch.cat([torch.from_numpy(c.o).cuda().expand(c.width * c.height, 3) for c in cams])
        d = torch.cat([_directions(c, torch.arange(c.width * c.height, device="cuda")) for c in cams])
        return o.contiguous(), d
    o = torch.from_numpy(np.stack([c.o for c in cams])).cuda()[rays[:, 0].long()]
    d = torch.empty_like(o)
    for v, c in enumerate(cams):
        m = rays[:, 0] == v
        d[m] = _directions(c, rays[m, 1].long())
    return o, d


def _render64(case, sc, w, o, d, n_max, t_stop=1e-4, chunk=1 << 18):
    """rgb, depth, opacity per ray (Eq. 4-5 with early termination), FP64."""
    outs = []
    delta, sigma = float(np.float32(sc.delta)), float(np.float32(sc.sigma))
    lab = torch.full((sc.G ** 3,), -1, dtype=torch.int32, device="cuda")
    lab[(sc.xyz[:, 2] * sc.G + sc.xyz[:, 1]) * sc.G + sc.xyz[:, 0]] = sc.lab.int()
    for at in range(0, o.shape[0], chunk):
        oc, dc = o[at:at + chunk], d[at:at + chunk]
        n = oc.shape[0]
        j, r = _kept(sc, oc, dc, n_max)
        count = torch.bincount(r, minlength=n)
        first = count.cumsum(0) - count
        k = torch.arange(r.numel(), device="cuda") - first[r]
        T = torch.ones(n, dtype=torch.float64, device="cuda")
        acc = torch.zeros(n, 5, dtype=torch.float64, device="cuda")
        alive = torch.ones(n, dtype=torch.bool, device="cuda")
        for k0 in range(0, n_max, 32):
            m = (k >= k0) & (k < k0 + 32) & alive[r]
            if not bool(m.any()):
                break
            jm, rm, km = j[m], r[m], k[m] - k0
            t = (jm.double() + 0.5) * delta
            p = oc[rm] + t[:, None] * dc[rm]
            v = torch.floor(p / float(np.float32(sc.vox))).long().clamp_(0, sc.G - 1)
            f = lab[(v[:, 2] * sc.G + v[:, 1]) * sc.G + v[:, 0]].clamp_(min=0)
            out = _fields64(case, w, sc.affine, sigma, p, dc[rm], f)
            tau = torch.zeros(n, 32, dtype=torch.float64, device="cuda").index_put((rm, km), out[:, 0] * delta)
            live = torch.zeros(n, 32, dtype=torch.bool, device="cuda").index_put((rm, km), torch.ones_like(km).bool())
            after = T[:, None] * torch.exp(-tau.cumsum(1))
            before = torch.cat([T[:, None], after[:, :-1]], 1)
            used = live & (before >= t_stop)
            wgt = torch.where(used, before - after, torch.zeros((), dtype=torch.float64, device="cuda"))[rm, km]
            acc = acc.index_add(0, rm, torch.cat([out[:, 1:] * wgt[:, None], (wgt * t)[:, None], wgt[:, None]], 1))
            stop = (after < t_stop)
            # the transmittance after the last composited sample
            T_new = torch.where(stop.any(1), after.gather(1, stop.int().argmax(1, keepdim=True))[:, 0], after[:, -1])
            alive = alive & ~stop.any(1)
            T = T_new
        outs.append(acc)
    acc = torch.cat(outs)
    return acc[:, :3], acc[:, 3], acc[:, 4]


def _scans64(case, sc, cams, depth, opacity):
    """Log-odds after the scans (Eq. 6): exact segment traversal per pixel."""
    G, vox = sc.G, float(np.float32(sc.vox))
    L = torch.zeros(G ** 3, dtype=torch.float64, device="cuda")
    p_hit, p_miss = float(np.float32(0.7)), float(np.float32(0.4))
    at = 0
    for c in cams:
        n = c.width * c.height
        A, D = opacity[at:at + n].double(), depth[at:at + n].double()
        at += n
        m = A >= 0.5
        A, te = A[m], D[m] / A[m]
        d = _directions(c, torch.arange(n, device="cuda"))[m]
        o = torch.from_numpy(c.o).cuda()
        free = torch.zeros(G ** 3, dtype=torch.bool, device="cuda")
        step = torch.sign(d)
        plane = torch.where(d > 0, torch.floor(o / vox) + 1, torch.ceil(o / vox) - 1)
        inf = torch.full((), 1e300, dtype=torch.float64, device="cuda")
        tn = torch.where(d != 0, (plane * vox - o) / d, inf)
        t_cur = torch.zeros_like(te)
        cell = torch.floor((o + 0.5 * torch.minimum(tn.amin(1), te)[:, None] * d) / vox)
        ce = torch.floor((o + te[:, None] * d) / vox)
        ends, eA = ce, A
        while te.numel():
            t1 = torch.minimum(tn.amin(1), te)
            ok = ((t1 - t_cur) >= 1e-9 * vox) & ((cell >= 0) & (cell < G)).all(1)
            q = cell[ok].long()
            free[(q[:, 2] * G + q[:, 1]) * G + q[:, 0]] = True
            go = t1 < te
            cross = (tn == t1[:, None])[go]
            d, step, te, t_cur = d[go], step[go], te[go], t1[go]
            plane = plane[go] + step * cross
            cell = cell[go] + step * cross
            tn = torch.where(d != 0, (plane * vox - o) / d, inf)
        ok = ((ends >= 0) & (ends < G)).all(1)
        q = ends[ok].long()
        hit = torch.zeros(G ** 3, dtype=torch.float64, device="cuda").scatter_reduce(
            0, (q[:, 2] * G + q[:, 1]) * G + q[:, 0], eA[ok], "amax")
        h = hit > 0
        ph = 0.5 + (p_hit - 0.5) * hit[h]
        L[h] += torch.log(ph / (1 - ph))
        f = free & ~h
        L[f] += math.log(p_miss / (1 - p_miss))
        L.clamp_(-2.0, 3.5)
    return L


def exact(case, seed):
    kind = case["kind"]
    if kind == "assign":
        return None
    if kind == "teacher":
        w, aff, p, d = _teacher_inputs(case, seed)
        return _teacher64(w, aff, p, d)
    if kind == "composite":
        count, sr, t = _composite_inputs(case, seed)
        n_max = case["n_max"]
        k = torch.arange(n_max, device="cuda")
        sr, t = sr.double(), t.double()
        tau = torch.where(k < count[:, None], sr[..., 0] * float(np.float32(0.01)), 0.0)
        after = torch.exp(-tau.cumsum(1))
        before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
        used = (k < count[:, None]) & (before >= 1e-4)
        wgt = torch.where(used, before - after, 0.0)
        T = torch.where(used, after, 2.0).amin(1)
        T = torch.where(used.any(1), T, 1.0)
        bg = torch.tensor([0.1, 0.2, 0.3], dtype=torch.float32).double().cuda()
        return {"rgb": (sr[..., 1:] * wgt[..., None]).sum(1) + T[:, None] * bg, "depth": (wgt * t).sum(1),
                "opacity": wgt.sum(1), "used": None}
    sc = _Scene(case["grid"], case.get("fields", 8), seed)
    if kind == "occupancy":
        cams = _cameras(case, sc)
        depth, opacity = _scan_inputs(case, seed, sc, cams)
        return {"logit": _scans64(case, sc, cams, depth, opacity), "bits": None}
    w = _field_weights(case, seed)
    if kind == "points":
        g = _gen(seed + 2)
        pick = torch.randint(0, sc.xyz.shape[0], (case["points"],), generator=g, device="cuda")
        p, d, f = _points(sc, g, pick)
        return _fields64(case, w, sc.affine, float(np.float32(sc.sigma)), p.double(), d.double(), f)
    if kind == "distill":
        p, d, f = _distill_inputs(case, sc, seed)
        tw = _weights(_gen(seed + 3), _teacher_shapes(), 1)[0]
        t = _teacher64(tw, np.array([0.25, 0.25, 0.25, -1.0, -1.0, -1.0], dtype=np.float32), p, d)
        w = w.double().requires_grad_(True)
        st = _fields64(case, w, sc.affine, float(np.float32(sc.sigma)), p.double(), d.double(), f)
        loss = ((st - t) ** 2).sum() / case["per_field"]
        loss.backward()
        return {"teacher": t, "student": st.detach(), "loss": loss.detach().reshape(1), "grad": w.grad}
    cams = _cameras(case, sc)
    if kind == "render":
        o, d = _rays64(case, sc, cams, None)
        with torch.no_grad():
            rgb, depth, opacity = _render64(case, sc, w, o, d, case["n_max"])
        return {"rgb": rgb, "depth": depth, "opacity": opacity}
    rays, target = _ray_batch(case, seed)
    o, d = _rays64(case, sc, cams, rays)
    w = w.double().requires_grad_(True)
    total, grad_rgb = 0.0, []
    for at in range(0, o.shape[0], 8192):
        rgb = _render64(case, sc, w, o[at:at + 8192], d[at:at + 8192], case["n_max"])[0]
        loss = ((rgb - target[at:at + 8192].double()) ** 2).sum() / (3.0 * o.shape[0])
        loss.backward()
        total += loss.detach()
        grad_rgb.append(rgb.detach())
    out = {"loss": total.reshape(1) if kind == "finetune" else total, "grad": w.grad}
    if kind == "autograd":
        out["rgb"] = torch.cat(grad_rgb)
    return out
