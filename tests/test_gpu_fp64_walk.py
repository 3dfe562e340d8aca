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


def _far_corners(n, r, gap, phi=None, seed=3):
    """A slab of some 1000 x 1000 x 2, `n` cells a side. Beside corners of its
    far cells, near the diagonal (or in the direction phi from its near corner): small balls (or posts along z) that only the
    cell on one side of the corner lists, `gap` paddings from its faces."""
    ext, pad = 1000.0, 0.01
    lo, E, N = -pad, ext + 2.0 * pad, 602 if phi else 3002
    V = E * E * (2.0 + 2.0 * pad)
    lam = (n / E) ** 3 * V / N
    rng = np.random.default_rng(seed)
    sph, cyl = [[1.5, 1.5, 1.0, 1.0], [ext - 0.5, ext - 0.5, 1.5, 0.5], [0.5, 0.5, 0.5, 0.5]], []
    for k in range(N - 3):
        i = int(rng.integers(n - 150, n - 2))
        j = int(i * math.tan(phi)) + int(rng.integers(-1, 3)) if phi else int(i + rng.integers(-25, 26))
        j = int(np.clip(j, 10, n - 3))
        s, q = (1 if k % 2 else -1), pad * gap + r
        x, y = lo + i * E / n - s * q, lo + j * E / n + s * q
        sph.append([x, y, 1.0, r])
        cyl.append([x, y, 0.1, x, y, 1.9, r])
    if phi:
        return S.make_scene(np.array(sph[:3]), np.array(cyl)), lam
    return S.make_scene(np.array(sph)), lam


@pytest.mark.parametrize("n,r,gap,phi", [(1023, 0.0015, 1.005, 0.7698324332205881),
                                         (1000, 0.002, 1.01, 0.7677444752973936)])
def test_long_walks_keep_to_their_cells(G, oracle, n, r, gap, phi):
    """Rays along the slab's diagonal cross some 2000 cells. Crossings summed up
    in FP32 drift by 2e-5 of the slab, the cells' lists are padded by 1e-5."""
    sc, lam = _far_corners(n, r, gap)
    d, u = (math.cos(phi), math.sin(phi), 0.0), (-math.sin(phi), math.cos(phi), 0.0)
    cam = S.Camera(eye=(500.0 - 900.0 * d[0], 500.0 - 900.0 * d[1], 1.0), dir=d, up=(0.0, 0.0, 1.0), right=u,
                   half_w=25.0, half_h=1e-3)
    p = S.Params(ao_samples=0, precision=S.PRECISION_FP64)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=lam)
        assert G.gbrt_grid_info(grid)["dims"][:2] == (n, n)
        ids = _ids(G, R, scene, grid, cam, 65000, 1, p)
    ref = oracle.render(sc, cam, 65000, 1, S.default_lights(), p, mode="brute")
    assert np.array_equal(ids, ref["id"]), int((ids != ref["id"]).sum())


def test_long_shadow_rays_keep_to_their_cells(G, oracle):
    """The same for shadow rays: from a ball in the near corner to posts in the
    far one."""
    phi = 0.7474635178445264
    sc, lam = _far_corners(1023, 0.0015, 1.005, phi)
    lights = S.Lights(dirs=[(math.cos(phi), math.sin(phi), 0.0)], intensity=[1.0], scale=1.0, skylight=0.0)
    cam = S.Camera(eye=(1.5, 1.5, 5.0), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0), right=(1.0, 0.0, 0.0), half_w=1.0,
                   half_h=1.0)
    p = S.Params(ao_samples=0, shadows=True, precision=S.PRECISION_FP64)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=lam)
        rgb, _, _ = R.render(scene, grid, cam, 600, 600, lights, p)
        G.gbrt_sync(R.ctx)
        got = rgb.cpu().numpy().reshape(-1, 3)
    ref = oracle.render(sc, cam, 600, 600, lights, p, mode="brute")
    wrong = np.abs(got - ref["rgb"]).max(axis=1) > 1e-9
    assert not wrong.any(), int(wrong.sum())
