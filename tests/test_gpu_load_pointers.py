"""Where the weights handed to roam_load_weights may lie.  Device memory of any
alignment is read in place; memory of other kinds handed over as device memory
goes through a copy, which reads it or refuses it, and either way the context
stays usable."""
import numpy as np
import pytest

import fixtures as F

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FIELDS, W, H = 3, 32, 2


@pytest.fixture(scope="module")
def ctx():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    r = roam.Roam(0)
    r.load_grid(np.full(1024, 0xffffffff, np.uint32), (32, 32, 32), (0.0, 0.0, 0.0), 0.1)
    r.load_fields((np.arange(32 ** 3) % FIELDS).astype(np.uint16),
                  np.tile(np.array([0.5, 0.5, 0.5, 0.0, 0.0, 0.0], np.float32), (FIELDS, 1)))
    yield roam, r
    r.close()


def _weights(seed):
    return torch.from_numpy(F.xavier_weights(seed, F.ROLE_STUDENT, FIELDS, W, H, bias_scale=0.3))


@pytest.mark.parametrize("offset", [0, 1, 3])
def test_device_memory_of_any_alignment(ctx, offset):
    _, r = ctx
    w = _weights(1 + offset).cuda()
    room = torch.empty(w.numel() + 8, device="cuda")
    at = room[offset:offset + w.numel()].view_as(w)
    at.copy_(w)
    r.load_weights(at, W, H, 10.0)
    assert torch.equal(r.get_weights(), w)


@pytest.mark.parametrize("pinned", [False, True])
def test_host_memory_handed_over_as_device_memory(ctx, pinned):
    roam, r = ctx
    w = _weights(11 + pinned)
    host = w.pin_memory() if pinned else w
    try:
        r.load_weights(host, W, H, 10.0)
    except roam.RoamError:
        pass
    else:
        assert torch.equal(r.get_weights().cpu(), w)
    again = _weights(20).cuda()
    r.load_weights(again, W, H, 10.0)
    assert torch.equal(r.get_weights(), again)
    torch.cuda.synchronize()
