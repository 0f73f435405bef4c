"""Bucketing of key counts on both sides of the line between its launch shapes
(2^21 keys), against a stable sort: offsets equal, every field's samples those of
the keys (in any order)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FIELDS = 700


@pytest.mark.parametrize("n", [(1 << 21) - 1, 1 << 21, 3_000_001])
def test_bucketing_of_many_keys(n):
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    r = roam.Roam(0)
    r.load_grid(np.full(1024, 0xffffffff, np.uint32), (32, 32, 32), (0.0, 0.0, 0.0), 0.1)
    r.load_fields((np.arange(32 ** 3) % FIELDS).astype(np.uint16), np.ones((FIELDS, 6), np.float32))
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    keys = torch.randint(0, FIELDS - 1, (n,), device="cuda", generator=g).to(torch.int16)
    keys[: n // 3] = 5                                     # one long field beside the others; the last one empty
    perm, offsets = r.bucket(keys)
    r.check()
    count = torch.bincount(keys.long(), minlength=FIELDS)
    want = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(count, 0)])
    assert torch.equal(offsets.long(), want)
    got = keys.long()[perm.long()]
    assert torch.equal(got, torch.sort(keys.long(), stable=True).values)
    assert torch.equal(torch.sort(perm.long()).values, torch.arange(n, device="cuda"))
    r.close()
