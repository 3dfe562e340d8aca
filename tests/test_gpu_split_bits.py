"""Row bands small enough for several lanes to share a primary ray give the
pixels of the whole frame, also where a ray's cells do not settle its order:
crosses of tubes some 50,000 units off, where FP32 coordinates are 4e-3 apart, and a tube
nearly along the view, whose FP32 root is wrong by more than the cells' padding,
with small balls coming out of it just beyond cell boundaries. Lanes that look
at the cells behind the one where the whole frame's walk ends must not use what
they find there."""
import math

import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _frames_equal(G, torch, R, scene, grid, cam, w, h, bands, p):
    lights, fp64 = S.default_lights(), p.precision == S.PRECISION_FP64

    def out():
        return [torch.zeros((h, w, 3), device="cuda", dtype=torch.float64 if fp64 else torch.float32)] + \
            [torch.zeros((h, w), dtype=torch.int32, device="cuda") for _ in range(2)]

    got, ref = out(), out()
    G.gbrt_render(R.ctx, scene, grid, cam, w, h, p.ao_samples, lights, p, *ref)
    for k in range(bands):
        G.gbrt_render_batch(R.ctx, [G.make_item(scene, grid, cam, w, h, p.ao_samples, lights, p, *got,
                                                rows=(k * h // bands, (k + 1) * h // bands))])
    G.gbrt_sync(R.ctx)
    return sum(int((u != v).sum()) for u, v in zip(got, ref))


@pytest.mark.parametrize("fp64", [False, True])
def test_far_off_crosses(fp64):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
    p = S.Params(ao_samples=1, seed=1, precision=S.PRECISION_FP64 if fp64 else S.PRECISION_FP32)
    wrong = 0
    with G.Renderer(0) as R:
        for seed in range(250):
            rng = np.random.default_rng(seed)
            off = rng.uniform(-60000.0, 60000.0, 3)
            c = rng.uniform(-12.0, 12.0, (1100, 3)) * [1.0, 0.05, 0.05]
            e = np.eye(3)[rng.integers(0, 3, 1100)] * rng.choice([0.5, 1.0, 2.0])
            m = np.round(c * 8.0) / 8.0 + off
            sc = S.make_scene(np.concatenate([c + off, rng.uniform(0.01, 0.05, (1100, 1))], 1),
                              np.concatenate([m - e, m + e, np.full((1100, 1), rng.choice([0.125, 0.25]))], 1))
            d = rng.standard_normal(3)
            d /= np.linalg.norm(d)
            u = np.cross(d, [0.3, 0.9, 0.1])
            u /= np.linalg.norm(u)
            half = rng.choice([1.4, 13.0])
            at = off if half > 2.0 else m[0]
            cam = S.Camera(eye=tuple(at - 40.0 * d), dir=tuple(d), up=tuple(np.cross(u, d)), right=tuple(u),
                           half_w=half, half_h=half)
            scene, grid = R.upload(sc, lam=8.0)
            wrong += _frames_equal(G, torch, R, scene, grid, cam, 900, 900, int(rng.choice([24, 60, 120])), p)
            R.free(scene, grid)
    assert wrong == 0, wrong


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("bands", [2, 16])
def test_grazing_tube(bands, fp64):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
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
    p = S.Params(ao_samples=2, seed=1, precision=S.PRECISION_FP64 if fp64 else S.PRECISION_FP32)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=lam)
        for x, y, _, _ in sph[2:32]:
            cam = S.Camera(eye=(x, y, 60.0), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0), right=(1.0, 0.0, 0.0),
                           half_w=1e-4, half_h=2e-3)
            assert _frames_equal(G, torch, R, scene, grid, cam, 100, 1600, bands, p) == 0, (x, y)
