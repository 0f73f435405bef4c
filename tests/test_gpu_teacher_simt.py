"""The FP32 teacher over its tile sizes (32, 64, 96 and 128 points, chosen by
the number of points; whole waves, then a rest) and their remainders, against the oracle at the first and
last points and a sample of the others; the bar of the FP32 teacher's other
test (1e-4: FP32 sums of up to 319 terms over 11 layers)."""
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


@pytest.mark.parametrize("n", [1, 31, 33, 4864, 9727, 9800, 14001, 15999, 20011, 32768, 40001])
def test_teacher_f32_tiles(roam, room32, n):
    r = roam.Roam(0)
    w, aff = F.teacher_weights(7, bias_scale=0.1), F.scene_affine(room32.scene)
    r.teacher_load(w, aff)
    rng = np.random.default_rng(n)
    p = rng.uniform(0, 3.2, (n, 3)).astype(np.float32)
    d = rng.normal(size=(n, 3))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    out = r.teacher_eval(torch.from_numpy(p).cuda(), torch.from_numpy(d).cuda(), precision=roam.ROAM_F32)
    torch.cuda.synchronize()
    r.check()
    i = np.unique(np.concatenate([np.arange(min(n, 130)), np.arange(max(0, n - 130), n), rng.integers(0, n, 200)]))
    ref = O.teacher_eval(w, aff, p[i].astype(np.float64), d[i].astype(np.float64))
    got = out.cpu().numpy().astype(np.float64)[i]
    assert np.abs(got[:, 1:] - ref[:, 1:]).max() <= 1e-4
    assert (np.abs(got[:, 0] - ref[:, 0]) / np.maximum(1.0, ref[:, 0])).max() <= 1e-4
    r.close()
