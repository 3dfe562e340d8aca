"""The near pass leaves one object out of a hit's candidates: the tube that the
hit lies on. Objects that share that tube's centre stay in: the other arms of a
3-D cross, the outer wall of a pipe seen through its open end, a sleeve around
the middle of a bond, a sphere at a tube's middle, a tube drawn twice. The same
frame in row bands (no near pass) is the reference, bit for bit.

Coordinates are multiples of 1/64, so the middles are the same floats."""
import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu

W, H, BANDS = 1100, 1100, 22


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt
    return gbrt


def _q(x):
    return np.round(np.asarray(x) * 64.0) / 64.0


def _scene(kind):
    rng = np.random.default_rng(29)
    c = _q(rng.uniform(-12.0, 12.0, (260, 3)))
    d = rng.standard_normal((260, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)

    def tube(e, r):
        return np.concatenate([c - e, c + e, np.full((len(c), 1), r)], 1)

    sph = np.array([[0.0, 0.0, 0.0, 0.5]])
    if kind == "cross":
        e = np.eye(3)
        cyl = np.concatenate([tube(_q(0.9 * e[k]) * np.ones((len(c), 1)), 0.25) for k in range(3)])
    elif kind == "pipe":
        e = _q(0.8 * d)
        cyl = np.concatenate([tube(e, 0.6), tube(e, 0.9)])
    elif kind == "sleeve":
        cyl = np.concatenate([tube(_q(1.2 * d), 0.2), tube(_q(0.5 * d), 0.45)])
    elif kind == "twice":
        cyl = np.concatenate([tube(_q(0.9 * d), 0.3), tube(_q(0.9 * d), 0.3)])
    else:
        cyl = tube(_q(1.1 * d), 0.45)
        sph = np.concatenate([c, np.full((len(c), 1), 0.5)], 1)
    return S.make_scene(sph, cyl)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("kind,eps,half", [("cross", 1e-3, 13.0), ("pipe", 1e-3, 13.0), ("sleeve", 1e-3, 13.0),
                                           ("twice", 1e-3, 13.0), ("sphere", 1e-4, 5.0)])
def test_objects_with_one_centre(G, kind, eps, half, fp64):
    import torch
    sc = _scene(kind)
    cam = S.Camera(eye=(0.0, 0.0, 30.0), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0), right=(1.0, 0.0, 0.0),
                   half_w=half, half_h=half)
    p = S.Params(ao_samples=16, seed=9, eps=eps, shadows=True,
                 precision=S.PRECISION_FP64 if fp64 else S.PRECISION_FP32)
    lights = S.default_lights()

    def outputs():
        return (torch.full((H, W, 3), -1.0, device="cuda", dtype=torch.float64 if fp64 else torch.float32),
                torch.full((H, W), -7, dtype=torch.int32, device="cuda"),
                torch.full((H, W), -7, dtype=torch.int32, device="cuda"))

    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=8.0)
        got, ref = outputs(), outputs()
        n0 = G.gbrt_launch_count(R.ctx)
        G.gbrt_render(R.ctx, scene, grid, cam, W, H, p.ao_samples, lights, p, *got)
        n1 = G.gbrt_launch_count(R.ctx)
        for k in range(BANDS):
            rows = (k * H // BANDS, (k + 1) * H // BANDS)
            G.gbrt_render_batch(R.ctx, [G.make_item(scene, grid, cam, W, H, p.ao_samples, lights, p, *ref, rows=rows)])
        n2 = G.gbrt_launch_count(R.ctx)
        G.gbrt_sync(R.ctx)
        assert n1 - n0 == 4 and n2 - n1 == 3 * BANDS
        for a, b in zip(got, ref):
            assert torch.equal(a, b), int((a != b).sum())


@pytest.mark.parametrize("fp64", [False, True])
def test_small_offsets(G, fp64):
    """Offsets eps from 1e-4 of a radius down to 0: an origin so close to its own
    atom must not send its rays through the whole walk after the near pass. Same
    bits as the bands, and no frame takes twice the time of the one at eps 1e-3
    (FP64 frames took seven times as long)."""
    import torch
    sc = S.globule(1500, 1425, 27.0, seed=3)
    cam, lights = S.ortho_camera(sc, W, H, angle_deg=20.0), S.default_lights()
    times = {}
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=8.0)
        for eps in (1e-3, 1e-4, 5e-5, 1e-5, 4e-6, 2e-6, 0.0):
            p = S.Params(ao_samples=16, seed=9, eps=eps, shadows=True,
                         precision=S.PRECISION_FP64 if fp64 else S.PRECISION_FP32)
            got, ref = [[torch.full((H, W, 3), -1.0, device="cuda", dtype=torch.float64 if fp64 else torch.float32)] +
                        [torch.full((H, W), -7, dtype=torch.int32, device="cuda") for _ in range(2)] for _ in range(2)]
            took = []
            for _ in range(5):
                a, b = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                a.record()
                G.gbrt_render(R.ctx, scene, grid, cam, W, H, p.ao_samples, lights, p, *got)
                b.record()
                b.synchronize()
                took.append(a.elapsed_time(b))
            times[eps] = min(took)
            for k in range(BANDS):
                rows = (k * H // BANDS, (k + 1) * H // BANDS)
                G.gbrt_render_batch(R.ctx, [G.make_item(scene, grid, cam, W, H, p.ao_samples, lights, p, *ref, rows=rows)])
            G.gbrt_sync(R.ctx)
            for a, b in zip(got, ref):
                assert torch.equal(a, b), (eps, int((a != b).sum()))
    assert all(times[e] < 2.0 * times[1e-3] for e in times if e >= 4e-6), times


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("far,eps", [(300.0, 3e-6), (9000.0, 1e-5), (20000.0, 1e-4)])
def test_origins_on_the_other_side(G, far, eps, fp64):
    """Far from the coordinates' zero an FP32 origin is rounded by more than eps:
    one on the inner wall of an open tube may come to lie outside, and its rays,
    which go inward, do meet that tube."""
    import torch
    rng = np.random.default_rng(4)
    off = np.array([far, -0.7 * far, 0.4 * far])
    m = rng.uniform(-6.0, 6.0, (150, 3)) + off
    d = rng.standard_normal((150, 3))
    d *= 0.6 / np.linalg.norm(d, axis=1, keepdims=True)
    sc = S.make_scene(np.concatenate([m[:40], np.full((40, 1), 0.2)], 1),
                      np.concatenate([m - d, m + d, rng.uniform(0.2, 0.5, (150, 1))], 1))
    cam = S.Camera(eye=tuple(off + [0.0, 0.0, 20.0]), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0), right=(1.0, 0.0, 0.0),
                   half_w=6.5, half_h=6.5)
    lights = S.default_lights()
    p = S.Params(ao_samples=16, seed=9, eps=eps, shadows=True,
                 precision=S.PRECISION_FP64 if fp64 else S.PRECISION_FP32)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=8.0)
        got, ref = [[torch.full((H, W, 3), -1.0, device="cuda", dtype=torch.float64 if fp64 else torch.float32)] +
                    [torch.full((H, W), -7, dtype=torch.int32, device="cuda") for _ in range(2)] for _ in range(2)]
        n0 = G.gbrt_launch_count(R.ctx)
        G.gbrt_render(R.ctx, scene, grid, cam, W, H, p.ao_samples, lights, p, *got)
        assert G.gbrt_launch_count(R.ctx) - n0 == 4
        for k in range(BANDS):
            rows = (k * H // BANDS, (k + 1) * H // BANDS)
            G.gbrt_render_batch(R.ctx, [G.make_item(scene, grid, cam, W, H, p.ao_samples, lights, p, *ref, rows=rows)])
        G.gbrt_sync(R.ctx)
        for a, b in zip(got, ref):
            assert torch.equal(a, b), int((a != b).sum())
