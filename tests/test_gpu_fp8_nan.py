"""FP8 forward with inputs that make NaNs.  A sample whose position is NaN or
infinite has no finite encoding; its first layer's ReLU gives zeros (max(NaN, 0)
is 0), so its outputs are those of the same network with a first layer of
zeros, bit for bit, and the samples beside it are not touched."""
import numpy as np
import pytest

import fixtures as F

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FIELDS = 3


@pytest.fixture(scope="module")
def roam():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    return roam


def _ctx(roam, w, W, H):
    r = roam.Roam(0)
    r.load_grid(np.full(1024, 0xffffffff, np.uint32), (32, 32, 32), (0.0, 0.0, 0.0), 0.1)
    r.load_fields((np.arange(32 ** 3) % FIELDS).astype(np.uint16),
                  np.tile(np.array([0.5, 0.5, 0.5, 0.0, 0.0, 0.0], np.float32), (FIELDS, 1)))
    r.load_weights(w, W, H, 10.0)
    return r


def _points(n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    p = torch.rand((n, 3), device="cuda", generator=g) * 2 - 1
    d = torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1)
    f = torch.randint(0, FIELDS, (n,), device="cuda", generator=g).to(torch.int16)
    return p, d, f


@pytest.mark.parametrize("W,H", [(32, 1), (64, 3), (128, 2)])
def test_positions_without_a_finite_encoding(roam, W, H):
    w = F.xavier_weights(1, F.ROLE_STUDENT, FIELDS, W, H, bias_scale=0.3)
    w0 = w.copy()
    w0[:, :W * 63 + W] = 0.0
    p, d, f = _points(700, W)
    bad = torch.zeros(700, dtype=torch.bool, device="cuda")
    bad[::7] = True
    q = p.clone()
    q[0::21, 0] = float("nan")
    q[7::21, 1] = float("inf")
    q[14::21, 2] = -float("inf")
    r, r0 = _ctx(roam, w, W, H), _ctx(roam, w0, W, H)
    out = r.mlp_eval(q, d, f, roam.ROAM_FP8)
    assert torch.equal(out[~bad], r.mlp_eval(p, d, f, roam.ROAM_FP8)[~bad])
    assert torch.equal(out[bad], r0.mlp_eval(p, d, f, roam.ROAM_FP8)[bad])
    assert torch.isfinite(out).all()
    r.close()
    r0.close()


@pytest.mark.parametrize("W,H", [(32, 2), (64, 2), (128, 2)])
def test_rows_whose_scale_underflows(roam, W, H):
    """An output whose weights are zeros and values below 448 times the smallest
    float: its scale max / 448 would round to 0 and 0 / 0 make its weights NaN.
    Such weights add nothing to a bias that is not as small, so the outputs are
    those of a row of zeros, bit for bit."""
    w = F.xavier_weights(2, F.ROLE_STUDENT, FIELDS, W, H, bias_scale=0.3)
    hidden = W * 63 + W                       # H = 2: one hidden layer, [out][in]
    w0 = w.copy()
    for row in (0, W // 2, W - 1):
        s = slice(hidden + row * W, hidden + (row + 1) * W)
        w0[:, s] = 0.0
        w[:, s] = 0.0
        w[:, hidden + row * W + 3] = np.float32(1e-43)
        w[:, hidden + row * W + 5] = np.float32(-2.8e-45)
    p, d, f = _points(300, W)
    r, r0 = _ctx(roam, w, W, H), _ctx(roam, w0, W, H)
    out, ref = r.mlp_eval(p, d, f, roam.ROAM_FP8), r0.mlp_eval(p, d, f, roam.ROAM_FP8)
    assert torch.isfinite(ref).all()
    assert torch.equal(out, ref)
    r.close()
    r0.close()
