"""The occupancy traversal on voxel planes, without allowances.  Cameras on
plane crossings and axis-aligned views, whose rays run along planes, cross two
or three planes at once and turn to FP64 step after step: every voxel of every
scan must have the log-odds of the definition, evaluated here in FP64 from
sorted crossings (the voxel of an interval from its midpoint, intervals below
1e-9 voxel not marked).  A walk that steps one axis at a time without that rule
marks other voxels, as checked here.

Also a camera near the largest admitted distance from the grid (16,384 voxels
from its far corner), where the rounding of the end point is largest, and a
second grid of another size on the same context (the marks are left clear)."""
import math

import numpy as np
import pytest

import fixtures as F

VOX = 0.125
P_HIT, P_MISS, L_MIN, L_MAX, A_MIN = 0.7, 0.4, -2.0, 3.5, 0.5


def _logit(p):
    return math.log(p / (1.0 - p))


def _rays(cam):
    """FP64 directions of a perspective view, from its FP32 parameters."""
    inv = math.tan(0.5 * float(np.float32(cam.fov_h))) / (0.5 * cam.width)
    v, u = np.mgrid[0:cam.height, 0:cam.width]
    x, y = (u + 0.5 - 0.5 * cam.width) * inv, (v + 0.5 - 0.5 * cam.height) * inv
    n = 1.0 / np.sqrt(x * x + y * y + 1.0)
    local = np.stack([x * n, y * n, n], axis=-1).reshape(-1, 3)
    return local @ np.asarray(cam.R, np.float32).astype(np.float64).T


def _scan(dims, cam, depth, op, one_axis_at_a_time=False):
    """(free voxels, hit voxel -> opacity) of one view by the definition."""
    o = np.asarray(cam.o, np.float32).astype(np.float64) / VOX              # (dyadic: exact)
    dims = np.asarray(dims)
    free, hit = set(), {}

    def voxel(q):
        c = np.floor(q).astype(np.int64)
        return tuple(c) if ((c >= 0) & (c < dims)).all() else None

    for d, D, A in zip(_rays(cam) / VOX, depth, op):
        if not A >= np.float32(A_MIN):
            continue
        t_end = float(D) / float(A)
        events = []
        for a in range(3):
            if d[a] != 0.0:
                lo, hi = sorted((o[a], o[a] + t_end * d[a]))
                if not one_axis_at_a_time:                        # (planes outside the grid part no voxels in it)
                    lo, hi = max(lo, -1), min(hi, dims[a] + 1)
                k = np.arange(math.floor(lo), math.ceil(hi) + 1)
                t = (k - o[a]) / d[a]
                events += [(s, a) for s in t[(t > 0.0) & (t < t_end)]]
        events.sort()
        if one_axis_at_a_time:
            c = np.floor(o + 0.5 * (events[0][0] if events else t_end) * d)
            for s, a in events + [(t_end, None)]:
                v = voxel(c)
                if v:
                    free.add(v)
                if a is not None:
                    c[a] += math.copysign(1.0, d[a])
        else:
            ts = np.array([0.0] + [s for s, _ in events] + [t_end])
            length = np.linalg.norm(d)
            for t0, t1 in zip(ts[:-1], ts[1:]):
                if (t1 - t0) * length >= 1e-9:
                    v = voxel(o + 0.5 * (t0 + t1) * d)
                    if v:
                        free.add(v)
        e = o + t_end * d
        v = voxel(e)
        if v:
            assert np.abs(e - np.rint(e))[d != 0.0].min() > 1e-9, "an end point on a plane decides nothing"
            hit[v] = max(hit.get(v, 0.0), float(A))
    return free, hit


def _apply(L, free, hit):
    for v in free - hit.keys():
        L[v[::-1]] = min(max(L[v[::-1]] + _logit(P_MISS), L_MIN), L_MAX)
    for v, A in hit.items():
        L[v[::-1]] = min(max(L[v[::-1]] + _logit(0.5 + (P_HIT - 0.5) * A), L_MIN), L_MAX)


def _maps(cam, reach, seed):
    rng = np.random.default_rng(seed)
    op = rng.uniform(0.4, 1.0, cam.n_pixels).astype(np.float32)
    return (rng.uniform(0.0, reach, cam.n_pixels) * op).astype(np.float32), op


ALONG_X = np.array([[0.0, 0.0, 1.0], [0.0, 1.0, 0.0], [-1.0, 0.0, 0.0]])
CAMERAS = {
    "in_a_plane": F.Camera(F.PERSPECTIVE, 65, 49, math.pi / 2, np.eye(3), np.array([1.0, 2.0625, 0.5])),
    "on_a_corner": F.Camera(F.PERSPECTIVE, 65, 65, math.pi / 2, np.eye(3), np.array([2.0, 2.0, 0.5])),
    "outside_on_planes": F.Camera(F.PERSPECTIVE, 49, 49, math.pi / 2, ALONG_X, np.array([-1.0, 2.0, 2.0])),
}


@pytest.mark.parametrize("name", sorted(CAMERAS))
def test_a_walk_without_the_tie_rule_marks_other_voxels(name):
    cam = CAMERAS[name]
    depth, op = _maps(cam, 7.0, 5)
    free, hit = _scan((32, 32, 32), cam, depth, op)
    naive, _ = _scan((32, 32, 32), cam, depth, op, one_axis_at_a_time=True)
    assert len(free) > 1000 and free <= naive
    # (the kernel is allowed no difference: any voxel tells the two apart)
    assert (naive - free) - hit.keys()


@pytest.fixture(scope="module")
def roam():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    return roam


def _update(r, dims, cam, depth, op, L):
    torch = pytest.importorskip("torch")
    r.occupancy_update([cam], torch.from_numpy(depth).cuda(), torch.from_numpy(op).cuda(), L,
                       torch.zeros(int(np.prod(dims)) // 32, dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    r.check()


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CAMERAS))
def test_every_voxel_on_planes(roam, name):
    torch = pytest.importorskip("torch")
    cam, dims = CAMERAS[name], (32, 32, 32)
    r = roam.Roam(0)
    r.load_grid(np.full(32 ** 3 // 32, 0xffffffff, np.uint32), dims, (0.0, 0.0, 0.0), VOX)
    L = torch.zeros(32 ** 3, dtype=torch.float32, device="cuda")
    ref = np.zeros(dims[::-1])
    for seed in (5, 6):
        depth, op = _maps(cam, 7.0, seed)
        _update(r, dims, cam, depth, op, L)
        _apply(ref, *_scan(dims, cam, depth, op))
        # (a step of the log-odds is at least 0.2; FP32 rounding is below 1e-6)
        assert np.abs(L.cpu().numpy().reshape(ref.shape) - ref).max() <= 1e-5, seed
    r.close()


@pytest.mark.gpu
def test_far_camera_and_grids_of_two_sizes_on_one_context(roam):
    torch = pytest.importorskip("torch")
    r = roam.Roam(0)
    o = np.array([-16200 * VOX, 2.03, 1.97])
    for dims in ((64, 64, 64), (32, 32, 32), (64, 32, 40)):
        cam = F.Camera(F.PERSPECTIVE, 60, 60, 0.004, ALONG_X, o)
        r.load_grid(np.full(int(np.prod(dims)) // 32, 0xffffffff, np.uint32), dims, (0.0, 0.0, 0.0), VOX)
        rng = np.random.default_rng(dims[2])
        op = rng.uniform(0.4, 1.0, cam.n_pixels).astype(np.float32)
        depth = (rng.uniform(16200 * VOX, (16200 + dims[0]) * VOX, cam.n_pixels) * op).astype(np.float32)
        L = torch.zeros(int(np.prod(dims)), dtype=torch.float32, device="cuda")
        _update(r, dims, cam, depth, op, L)
        ref = np.zeros(dims[::-1])
        _apply(ref, *_scan(dims, cam, depth, op))
        assert np.count_nonzero(ref) > 3000
        assert np.abs(L.cpu().numpy().reshape(ref.shape) - ref).max() <= 1e-5, dims
    r.close()
