"""Both forms of the field assignment beyond the sizes of the other tests,
against the oracle's full sort (labels equal, voxel for voxel; boxes equal):
squared distances past 2^21, where the general form's key takes a fifth
digit; and, from the brick lists, a first anchor so far from the rest that
every brick is a candidate of its network: more than a block's table holds or
just fewer, with a few voxels each or with many."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def roam():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    return roam


def _bits(lin, dims):
    bits = np.zeros(dims[0] * dims[1] * dims[2] // 32, np.uint32)
    np.bitwise_or.at(bits, lin >> 5, np.uint32(1) << (lin & 31).astype(np.uint32))
    return bits


def _box(dims, lo, hi):
    z, y, x = np.meshgrid(*(np.arange(a, b) for a, b in zip(lo[::-1], hi[::-1])), indexing="ij")
    return ((z * dims[1] + y) * dims[0] + x).reshape(-1)


def _check(roam, dims, lin, n):
    lin = np.unique(lin)
    r = roam.Roam(0)
    r.load_grid(_bits(lin, dims), dims, (0.0, 0.0, 0.0), 0.1)
    labels, boxes = r.assign_fields(n)
    torch.cuda.synchronize()
    got = labels.cpu().numpy().view(np.uint16).astype(np.int32)
    assert np.array_equal(got, O.assign_fields(dims, lin, n))
    xyz = np.stack([lin % dims[0], (lin // dims[0]) % dims[1], lin // (dims[0] * dims[1])], axis=1)
    lo = np.full((n, 3), 1 << 30)
    hi = np.zeros((n, 3), dtype=np.int64)
    np.minimum.at(lo, got, xyz)
    np.maximum.at(hi, got, xyz + 1)
    assert np.array_equal(boxes.cpu().numpy(), np.concatenate([lo, hi], axis=1))
    r.close()


@pytest.mark.parametrize("n", [2, 3, 40])
def test_clusters_far_apart(roam, n):
    """A first cluster smaller than a network, the rest 2,700 voxels away (n = 2
    and 3: networks above 65,536 voxels; 40: small ones)."""
    dims = (2048, 2048, 8)
    lin = np.concatenate([_box(dims, (0, 0, 0), (90, 90, 8)), _box(dims, (1900, 1880, 0), (2040, 2030, 8))])
    _check(roam, dims, lin, n)


@pytest.mark.parametrize("x1,count,n", [
    (2040, 60_000, 25),       # past the table, 2 voxels per brick
    (2040, 300_000, 20),      # past the table, 9 voxels per brick
    (1664, 45_000, 25),       # within the table, 4 voxels per brick, too many to keep in registers
    (1664, 150_000, 20),      # within the table, 15 voxels per brick
])
def test_every_brick_a_candidate(roam, x1, count, n):
    dims = (2048, 512, 64)
    rng = np.random.default_rng(count)
    x, y, z = rng.integers(1504, x1, count), rng.integers(0, 512, count), rng.integers(0, 64, count)
    lin = np.concatenate([_box(dims, (0, 0, 0), (5, 4, 3)), (z * dims[1] + y) * dims[0] + x])
    _check(roam, dims, lin, n)


def test_lists_take_memory_only_where_they_are_used(roam):
    """The general form (here: one network, and two of 4.2 M voxels) holds the
    voxels' indices and a few kilobytes; the lists take 6 bytes per voxel more."""
    dims = (256, 256, 128)
    S = dims[0] * dims[1] * dims[2]
    r = roam.Roam(0)
    r.load_grid(np.full(S // 32, 0xffffffff, np.uint32), dims, (0.0, 0.0, 0.0), 0.1)
    del_me = torch.empty(S, dtype=torch.int16, device="cuda")      # (the labels come from torch's cache below)
    del del_me
    torch.empty((600, 6), dtype=torch.int32, device="cuda")

    def held(n):
        free = torch.cuda.mem_get_info()[0]
        r.assign_fields(n)
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0]

    assert held(1) <= 4 * S + (8 << 20)
    assert held(2) <= 8 << 20
    assert held(600) >= 6 * S - (8 << 20)
    r.close()
