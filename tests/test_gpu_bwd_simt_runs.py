"""The FP32 adjoint with several tiles per block: one long field of more than
two tiles per SM between many fields of one or two tiles, so that a block's run
of tiles starts and ends inside fields and crosses field changes (the weight
ring carries over into the next tile and field, the shared gradient is flushed
and cleared, a field's gradient comes from many blocks).  Every sample is one of
a few points of its field, so the oracle's gradient of a point times its count
is exact; samples at a ReLU kink of the oracle carry no gradient, and the bar is
the FP32 adjoint's, 1e-4 of max|g|."""
import numpy as np
import pytest

import fixtures as F
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIGMA_SCALE = 2.0
FIELDS, LONG = 220, 97


@pytest.mark.parametrize("W,H", [(32, 1), (32, 4), (64, 1), (64, 2), (64, 3), (64, 4)])
def test_runs_of_tiles_across_fields(W, H):
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    tile = 128 if W == 32 else (64 if H <= 3 else 32)
    rng = np.random.default_rng(10 * W + H)
    counts = np.array([(1, 3, tile - 1, tile, tile + 1)[k % 5] for k in range(FIELDS)])
    counts[LONG] = (2 * n_sm + 40) * tile + 7
    counts[[5, 6, FIELDS - 2]] = 0
    uniq = np.where(np.arange(FIELDS) == LONG, 48, 3)                # distinct points per field
    uf = np.repeat(np.arange(FIELDS), uniq)
    p = rng.uniform(-0.9, 0.9, (uf.size, 3)).astype(np.float32)
    d = rng.normal(size=(uf.size, 3))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    dl = (rng.normal(size=(uf.size, 4)) * 0.05).astype(np.float32)
    w = F.xavier_weights(1, F.ROLE_STUDENT, FIELDS, W, H, bias_scale=0.1)
    aff = np.tile(np.array([0.5, 0.5, 0.5, 0.1, -0.1, 0.0], np.float32), (FIELDS, 1))
    _, margin = O.mlp_grad_points(w, aff, W, H, SIGMA_SCALE, p, d, uf, dl)
    dl[margin < 1e-4] = 0.0
    # samples: each field's points in turn, shuffled over all fields
    start = np.concatenate([[0], np.cumsum(uniq)])
    pick = np.concatenate([start[k] + np.arange(counts[k]) % uniq[k] for k in range(FIELDS)])
    times = np.bincount(pick, minlength=uf.size)
    pick = rng.permutation(pick)
    g_o, _ = O.mlp_grad_points(w, aff, W, H, SIGMA_SCALE, p, d, uf, dl.astype(np.float64) * times[:, None])
    r = roam.Roam(0)
    r.load_grid(np.full(1024, 0xffffffff, np.uint32), (32, 32, 32), (0.0, 0.0, 0.0), 0.1)
    r.load_fields((np.arange(32 ** 3) % FIELDS).astype(np.uint16), aff)
    r.load_weights(w, W, H, SIGMA_SCALE)
    args = [torch.from_numpy(a[pick]).cuda() for a in (p, d, uf.astype(np.int16), dl)]
    g = r.mlp_backward(*args).cpu().numpy()
    torch.cuda.synchronize()
    r.check()
    r.close()
    for k in range(FIELDS):
        if counts[k] == 0:
            assert not g[k].any(), k
        else:
            assert np.abs(g[k] - g_o[k]).max() <= 1e-4 * np.abs(g_o[k]).max(), (k, counts[k])
