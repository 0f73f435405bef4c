"""The tensor-core forward at W = 32 keeps six tiles in flight where a call has
enough samples per field and per SM, else four.  A sample's outputs depend on
neither the form nor the tiles beside it: every sample of a call large enough
for six equals, bit for bit, the same sample in calls small enough for four,
with one sample fewer than the line (four) and at it (six), with the tile
padding that makes groups without work, and with a field of one sample."""
import numpy as np
import pytest

import fixtures as F

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FIELDS = 5
CHUNK = 40_000


@pytest.fixture(scope="module")
def roam():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    return roam


@pytest.mark.parametrize("prec", ["BF16", "FP8"])
@pytest.mark.parametrize("H", [1, 4])
def test_six_tiles_in_flight_give_the_bits_of_four(roam, H, prec):
    line = 16 * 128 * torch.cuda.get_device_properties(0).multi_processor_count
    r = roam.Roam(0)
    r.load_grid(np.full(1024, 0xffffffff, np.uint32), (32, 32, 32), (0.0, 0.0, 0.0), 0.1)
    r.load_fields((np.arange(32 ** 3) % FIELDS).astype(np.uint16),
                  np.tile(np.array([0.5, 0.5, 0.5, 0.0, 0.0, 0.0], np.float32), (FIELDS, 1)))
    r.load_weights(F.xavier_weights(3, F.ROLE_STUDENT, FIELDS, 32, H, bias_scale=0.3), 32, H, 10.0)
    g = torch.Generator(device="cuda")
    g.manual_seed(H)
    n = line + 129
    p = torch.rand((n, 3), device="cuda", generator=g) * 2 - 1
    d = torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1)
    f = torch.randint(0, FIELDS - 1, (n,), device="cuda", generator=g).to(torch.int16)
    f[line // 2] = FIELDS - 1
    precision = getattr(roam, "ROAM_" + prec)

    def ev(m):
        return r.mlp_eval(p[:m], d[:m], f[:m], precision)

    ref = torch.cat([r.mlp_eval(p[i:i + CHUNK], d[i:i + CHUNK], f[i:i + CHUNK], precision)
                     for i in range(0, n, CHUNK)])
    assert torch.isfinite(ref).all()
    for m in (line - 1, line, n):
        assert torch.equal(ev(m), ref[:m]), m
    for pad in (4, 8):
        r.set_tile_padding(pad)
        assert torch.equal(ev(n), ref), pad
    r.check()
    r.close()
