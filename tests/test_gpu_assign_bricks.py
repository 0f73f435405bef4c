"""The assignment from brick lists where it can go wrong, against the oracle's
full sort (labels equal, voxel for voxel): networks of one voxel, a solid
block (many equal distances), grids that are not cubes, an anchor far from
the voxels it takes (coarse distance bins: the last bin is narrowed before
its keys are ranked), distances past the bins' range, and networks on both
sides of the size that selects the general form."""
import numpy as np
import pytest

import fixtures as F
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def roam():
    import paper_2208_02705_gb300 as roam
    from paper_2208_02705_gb300 import build
    build.build()
    return roam


def _scattered(gz, gy, gx, share, seed):
    return np.random.default_rng(seed).random((gz, gy, gx)) < share


def _two_clusters(gz, gy, gx, x0, x1):
    occ = np.zeros((gz, gy, gx), dtype=bool)
    occ[2:6, 1:6, 0:5] = True                   # the first anchor's cluster
    occ[:, :, x0:x1] = True
    return occ


CASES = {
    "one_voxel_each": (_scattered(16, 24, 32, 0.02, 1), None),
    "two_voxels": (_scattered(8, 8, 32, 0.3, 2), 300),
    "not_a_cube": (_scattered(40, 24, 64, 0.2, 3), 37),
    "solid": (np.ones((64, 64, 64), dtype=bool), 5),
    "solid_general": (np.ones((64, 64, 64), dtype=bool), 3),
    "far_anchor": (_two_clusters(64, 64, 512, 440, 504), 50),
    "past_the_bins": (_two_clusters(8, 8, 2048, 1900, 2040), 4),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_assign_from_brick_lists(roam, name):
    occ, n = CASES[name]
    gz, gy, gx = occ.shape
    lin = np.flatnonzero(occ.reshape(-1)).astype(np.int64)
    n = lin.size if n is None else n
    r = roam.Roam(0)
    r.load_grid(F.pack_bits(occ), (gx, gy, gz), (0.0, 0.0, 0.0), 0.1)
    labels, boxes = r.assign_fields(n)
    torch.cuda.synchronize()
    got = labels.cpu().numpy().view(np.uint16).astype(np.int32)
    assert np.array_equal(got, O.assign_fields((gx, gy, gz), lin, n))
    xyz = np.stack([lin % gx, (lin // gx) % gy, lin // (gx * gy)], axis=1)
    lo = np.full((n, 3), 1 << 30)
    hi = np.zeros((n, 3), dtype=np.int64)
    np.minimum.at(lo, got, xyz)
    np.maximum.at(hi, got, xyz + 1)
    assert np.array_equal(boxes.cpu().numpy(), np.concatenate([lo, hi], axis=1))
    r.close()
