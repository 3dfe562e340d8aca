"""FP64 hit ids where the FP32 walk of the FP64 path is strained, against the
oracle's brute force (equal on every pixel: see test_gpu_fp64_filter)."""
import math

import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt
    return gbrt


def _ids(G, R, scene, grid, cam, W, H, p):
    _, ids, _ = R.render(scene, grid, cam, W, H, S.default_lights(), p, ids=True)
    G.gbrt_sync(R.ctx)
    return ids.cpu().numpy().view(np.uint32).ravel()


def test_the_walk_ends_only_past_the_roots_error(G, oracle):
    """A tube 0.036 off the view direction, seen close to its silhouette: its
    FP32 root is wrong by up to some 1e-3, more than the cells' padding. Small
    balls come out of it just beyond cell boundaries, where a walk that takes
    that root for exact ends one cell early."""
    ext, r, sin, pad = 40.0, 0.5, 0.036, 4e-4
    a = np.array([0.0, sin, math.sqrt(1.0 - sin * sin)])
    lo, E = -0.5 * ext - pad, ext + 2.0 * pad
    N, lam = 63, 200.0
    n = int(math.floor(E * (lam * N / E ** 3) ** (1.0 / 3.0) + 0.5))
    bounds = lo + E / n * np.arange(1, n)
    bounds = bounds[np.abs(bounds) < 14.0]
    rng = np.random.default_rng(1)
    sph = [[-19.5, -19.5, -19.5, 0.5], [19.5, 19.5, 19.5, 0.5]]
    for k in range(N - 3):
        front, half = bounds[k % len(bounds)] - 1.1 * pad, rng.uniform(0.5, 1.2)
        sph.append([math.sqrt(r * r - (half * sin) ** 2), (front - half) * a[1] / a[2], front - 0.05, 0.05])
    sc = S.make_scene(np.array(sph), np.concatenate([-18.0 * a, 18.0 * a, [r]])[None])
    p = S.Params(ao_samples=0, precision=S.PRECISION_FP64)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=lam)
        assert G.gbrt_grid_info(grid)["dims"] == (n, n, n)
        for x, y, _, _ in sph[2:26]:
            cam = S.Camera(eye=(x, y, 60.0), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0), right=(1.0, 0.0, 0.0),
                           half_w=1e-4, half_h=2e-3)
            ids = _ids(G, R, scene, grid, cam, 100, 800, p)
            ref = oracle.render(sc, cam, 100, 800, S.default_lights(), p, mode="brute")
            assert np.array_equal(ids, ref["id"]), int((ids != ref["id"]).sum())
