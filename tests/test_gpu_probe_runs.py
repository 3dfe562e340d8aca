"""gbrt_ao_probe hands each warp a run of (point, sample) jobs: counts of points
and samples around the warp's width and the run's length, runs that end inside
a point, several points a refill, no samples at all. Against the oracle's brute
force with the same samples: equal in FP64; in FP32 a sample flips when it
passes within ~1e-6 of a silhouette, so of the at most ~13,000 samples here
more than one flip has a probability below 1e-3."""
import math

import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [S.PRECISION_FP32, S.PRECISION_FP64])
@pytest.mark.parametrize("n,spp,maxdist", [(1, 1, math.inf), (1, 0, math.inf), (3, 31, math.inf), (33, 32, 5.0),
                                           (200, 65, math.inf), (4000, 3, 2.0)])
def test_probe_counts_equal_the_oracle(oracle, prec, n, spp, maxdist):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
    sc = S.globule(300, 285, 13.0, seed=4)
    rng = np.random.default_rng(n + spp)
    k = rng.integers(0, sc.n_spheres, n)
    nrm = rng.standard_normal((n, 3))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    pts = sc.spheres[k, :3].astype(np.float64) + sc.spheres[k, 3:4].astype(np.float64) * nrm
    p = S.Params(seed=9, precision=prec, eps=1e-3, ao_maxdist=maxdist)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=4.0)
        out = torch.full((n,), -1.0, device="cuda")
        G.gbrt_ao_probe(R.ctx, scene, grid, torch.from_numpy(pts).cuda(), torch.from_numpy(nrm).cuda(), spp, p, out)
        G.gbrt_sync(R.ctx)
    got = out.cpu().numpy().astype(np.float64)
    if spp == 0:
        assert np.all(got == 1.0)
        return
    ref = oracle.ao_probe(sc, pts, nrm, spp, seed=9, eps=1e-3, maxdist=maxdist, mode="brute")
    flips = int(np.abs(np.rint(got * spp) - np.rint(np.asarray(ref) * spp)).sum())
    assert flips <= (0 if prec == S.PRECISION_FP64 else 1), flips
