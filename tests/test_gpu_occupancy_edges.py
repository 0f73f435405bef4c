"""The occupancy traversal where its FP32 steps hand over to FP64 or take a
short cut: a camera on voxel planes and corners, axis-aligned rays along
planes, a camera outside the grid, end points far past the grid, zero depths, several views of both models in one call, and a second call on
the same context (the marks are left clear).  Against the oracle, with the
allowances of the traversal's other tests (ties reported by the oracle)."""
import math

import numpy as np
import pytest

import fixtures as F
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

G, VOX = 32, 0.125


@pytest.fixture(scope="module")
def roam():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    return roam


CAMERAS = {
    "on_a_corner": [F.Camera(F.EQUIRECT, 96, 48, 0.0, F.yaw_pitch(0.4, 0.1), np.array([2.0, 2.0, 2.0]))],
    "along_planes": [F.Camera(F.PERSPECTIVE, 65, 49, math.pi / 2, np.eye(3), np.array([1.0, 2.0625, 0.5]))],
    "outside": [F.Camera(F.PERSPECTIVE, 80, 60, math.pi / 2, F.yaw_pitch(math.pi / 2, 0.05), np.array([-3.0, 2.1, 1.9]))],
    "mixed_views": [F.Camera(F.EQUIRECT, 70, 33, 0.0, F.yaw_pitch(1.0, 0.0), np.array([1.03, 1.9, 2.71])),
                    F.Camera(F.PERSPECTIVE, 51, 40, 1.2, F.yaw_pitch(-2.0, 0.3), np.array([3.3, 2.0, 0.77])),
                    F.Camera(F.EQUIRECT, 64, 20, 0.0, F.yaw_pitch(2.0, -0.2), np.array([2.5, 2.0625, 1.3]))],
}


@pytest.mark.parametrize("name", sorted(CAMERAS))
def test_occupancy_edges(roam, name):
    cams = CAMERAS[name]
    r = roam.Roam(0)
    scene = F.room_scene(1, G, VOX)
    r.load_grid(scene.bits, scene.dims, scene.origin, scene.vox)
    n = sum(c.n_pixels for c in cams)
    rng = np.random.default_rng(len(name))
    op = rng.uniform(0.4, 1.0, n).astype(np.float32)
    depth = (rng.uniform(0.0, 9.0, n) * op).astype(np.float32)      # the grid is 4 wide
    depth[rng.random(n) < 0.05] = 0.0
    L = torch.zeros(G ** 3, dtype=torch.float32, device="cuda")
    bits = torch.zeros(G ** 3 // 32, dtype=torch.int32, device="cuda")
    dt, ot = torch.from_numpy(depth).cuda(), torch.from_numpy(op).cuda()
    Lr = np.zeros(G ** 3)
    thr = math.log(0.97 / 0.03)
    total_ties = 0
    for _ in range(2):
        r.occupancy_update(cams, dt, ot, L, bits)
        torch.cuda.synchronize()
        r.check()
        bits_r, ties = O.occupancy_update(scene.dims, scene.origin, scene.vox, Lr, F.camera_array(cams), depth, op)
        total_ties += ties
        bad = np.abs(L.cpu().numpy().astype(np.float64) - Lr) > 1e-5
        assert np.count_nonzero(Lr) > 100
        assert bad.sum() <= 2 * total_ties, (bad.sum(), total_ties)
        got = np.unpackbits(bits.cpu().numpy().view(np.uint8), bitorder="little").astype(bool)
        ref = np.unpackbits(bits_r.view(np.uint8), bitorder="little").astype(bool)
        sure = (np.abs(Lr - thr) > 1e-4) & ~bad
        assert np.array_equal(got[sure], ref[sure])
    r.close()
