"""The FP32 adjoint at the edges of its tiles (128 samples at W = 32, 64 at
W = 64, 32 at W = 64 / H = 4): fields of one sample, just under, at and just
over a tile, several tiles, and none, for every supported shape, against the
oracle's FP64 adjoint.  Samples at a ReLU kink of the oracle (|pre-activation|
< 1e-4, where FP32 may take the other branch) carry no gradient; the rest
agree to FP32 rounding: within 1e-4 of max|g|, the bar of the FP32 adjoint's
other tests."""
import numpy as np
import pytest

import fixtures as F
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIGMA_SCALE = 2.0
COUNTS = (1, 31, 64, 65, 0, 129, 33, 200)


@pytest.fixture(scope="module")
def roam():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    return roam


@pytest.mark.parametrize("W,H", [(32, 1), (32, 2), (32, 3), (32, 4), (64, 1), (64, 2), (64, 3), (64, 4)])
def test_f32_adjoint_at_tile_edges(roam, room32, W, H):
    w = F.xavier_weights(1, F.ROLE_STUDENT, room32.part.n_fields, W, H, bias_scale=0.1)
    r = roam.Roam(0)
    r.load_grid(room32.scene.bits, room32.scene.dims, room32.scene.origin, room32.scene.vox)
    r.load_fields(room32.part.field_of_rank, room32.affine)
    r.load_weights(w, W, H, SIGMA_SCALE)
    p, d, f = F.distill_points(room32.scene, room32.part, 5, max(COUNTS))
    keep = np.concatenate([np.flatnonzero(f == k)[:n] for k, n in enumerate(COUNTS)])
    keep = np.random.default_rng(W + H).permutation(keep)
    p, d, f = p[keep], d[keep], f[keep]
    dl = (np.random.default_rng(W * H).normal(size=(p.shape[0], 4)) * 0.05).astype(np.float32)
    _, margin = O.mlp_grad_points(w, room32.affine, W, H, SIGMA_SCALE, p, d, f, dl)
    dl[margin < 1e-4] = 0.0
    g_o, _ = O.mlp_grad_points(w, room32.affine, W, H, SIGMA_SCALE, p, d, f, dl)
    g = r.mlp_backward(torch.from_numpy(p).cuda(), torch.from_numpy(d).cuda(),
                       torch.from_numpy(f.astype(np.int16)).cuda(), torch.from_numpy(dl).cuda())
    torch.cuda.synchronize()
    r.check()
    g = g.cpu().numpy()
    assert not g[4].any()                                # the field without samples
    for k in range(len(COUNTS)):
        if COUNTS[k]:
            assert np.abs(g[k] - g_o[k]).max() <= 1e-4 * np.abs(g_o[k]).max(), (k, COUNTS[k])
    r.close()
