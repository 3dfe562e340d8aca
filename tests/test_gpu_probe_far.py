"""FP64 AO probe from points outside the scene, up to 100,000 times its size away:
each point is placed so that its first sample's ray goes to a random place in the
scene. Counts equal the oracle's brute force (see test_gpu_fp64_filter)."""
import math

import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limited", [False, True])
@pytest.mark.parametrize("away", [0.8, 3.0, 30.0, 1e3, 1e5])
def test_far_points(oracle, away, limited):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
    sc = S.globule(300, 285, 13.0, seed=4)
    sp = sc.spheres.copy()
    sp[:, 3] *= 0.4  # let rays through
    sc = S.Scene(spheres=sp, cylinders=sc.cylinders, color_idx=sc.color_idx, palette=sc.palette, radius=sc.radius)
    n, dist = 2000, 26.0 * away
    rng = np.random.default_rng(int(away * 10))
    nrm = rng.standard_normal((n, 3))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    target = rng.uniform(-9.0, 9.0, (n, 3))
    d = np.array([oracle.cosine_dir(nrm[k], *oracle.ao_uniforms(k, 0, 0, 9)) for k in range(n)])
    pts = target - dist * d - 1e-3 * nrm
    maxdist = dist if limited else math.inf
    p = S.Params(seed=9, precision=S.PRECISION_FP64, eps=1e-3, ao_maxdist=maxdist)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=60.0)
        out = torch.zeros(n, device="cuda")
        G.gbrt_ao_probe(R.ctx, scene, grid, torch.from_numpy(pts).cuda(), torch.from_numpy(nrm).cuda(), 1, p, out)
        G.gbrt_sync(R.ctx)
    ref = np.asarray(oracle.ao_probe(sc, pts, nrm, 1, seed=9, eps=1e-3, maxdist=maxdist, mode="brute"))
    assert 0.05 < ref.mean() < 0.95
    got = out.cpu().numpy().astype(np.float64)
    assert np.array_equal(got, ref), int((got != ref).sum())
