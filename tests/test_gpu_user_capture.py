"""Calls recorded into a CUDA graph of the caller's (after one call outside, which
allocates): the programmatic launches keep their order in it, replays read the
inputs as they are then, and an occupancy update in it, replayed between direct
ones, finds and leaves the marks clear."""
import math

import numpy as np
import pytest

import fixtures as F

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FIELDS = 40


@pytest.fixture(scope="module")
def roam():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    return roam


@pytest.mark.parametrize("prec,W", [("F32", 32), ("F32", 64), ("BF16", 32), ("BF16", 128), ("FP8", 64)])
def test_point_queries(roam, prec, W):
    r = roam.Roam(0)
    r.load_grid(np.full(1024, 0xffffffff, np.uint32), (32, 32, 32), (0.0, 0.0, 0.0), 0.1)
    r.load_fields((np.arange(32 ** 3) % FIELDS).astype(np.uint16),
                  np.tile(np.array([0.5, 0.5, 0.5, 0.0, 0.0, 0.0], np.float32), (FIELDS, 1)))
    r.load_weights(F.xavier_weights(3, F.ROLE_STUDENT, FIELDS, W, 2, bias_scale=0.3), W, 2, 10.0)
    g = torch.Generator(device="cuda")
    g.manual_seed(W)
    n, precision = 30_011, getattr(roam, "ROAM_" + prec)

    def inputs():
        return (torch.rand((n, 3), device="cuda", generator=g) * 2 - 1,
                torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1),
                torch.randint(0, FIELDS, (n,), device="cuda", generator=g).to(torch.int16))

    p, d, f = inputs()
    r.mlp_eval(p, d, f, precision)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = r.mlp_eval(p, d, f, precision)
    for _ in range(3):
        new = inputs()
        for a, b in zip((p, d, f), new):
            a.copy_(b)
        graph.replay()
        assert torch.equal(out, r.mlp_eval(*new, precision))
    r.check()
    r.close()


def test_occupancy_update_between_direct_ones(roam):
    G, vox = 32, 0.125
    r = roam.Roam(0)
    r.load_grid(np.full(G ** 3 // 32, 0xffffffff, np.uint32), (G, G, G), (0.0, 0.0, 0.0), vox)

    def cams(x):
        return [F.Camera(F.EQUIRECT, 96, 48, 0.0, F.yaw_pitch(0.4, 0.1), np.array([x, 2.03, 1.97])),
                F.Camera(F.PERSPECTIVE, 50, 40, math.pi / 3, F.yaw_pitch(x, 0.0), np.array([1.1, x, 2.2]))]

    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    n = sum(c.n_pixels for c in cams(1.0))
    op = torch.rand(n, device="cuda", generator=g) * 0.6 + 0.4
    depth = torch.rand(n, device="cuda", generator=g) * 4 * op
    L = torch.zeros(G ** 3, device="cuda")
    bits = torch.zeros(G ** 3 // 32, dtype=torch.int32, device="cuda")
    Lr, br = L.clone(), bits.clone()
    r.occupancy_update(cams(1.7), depth, op, L, bits)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        r.occupancy_update(cams(1.3), depth, op, L, bits)
    graph.replay()
    torch.cuda.synchronize()
    r.occupancy_update(cams(1.5), depth, op, L, bits)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    q = roam.Roam(0)
    q.load_grid(np.full(G ** 3 // 32, 0xffffffff, np.uint32), (G, G, G), (0.0, 0.0, 0.0), vox)
    for x in (1.7, 1.3, 1.5, 1.3):
        q.occupancy_update(cams(x), depth, op, Lr, br)
    torch.cuda.synchronize()
    assert torch.equal(L, Lr) and torch.equal(bits, br)
    assert torch.count_nonzero(L) > 1000
    q.close()
    r.close()
