"""The AO rays' near pass against the plain walk: a frame large enough for the
pass, and the same frame rendered in row bands that are not. The pass settles
only rays whose outcome its error bounds decide, so ids, sample counts and
colours are the same bits. The launch counter shows which path ran.

Cases: jobs a hit around the pass's words of 16 (8, 16, 17, 36 with lights),
hits on a tube's outer and inner side, origins on the surface itself (eps 0:
every hit starts inside the pass's margin), more balls around a hit than its
lists hold, tubes that stick far out of their spheres, a pinhole camera inside
the molecule, supersampling, a grid rebuilt on the device, and a batch whose
frames differ in scene and in whether the pass suits them."""
import dataclasses

import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu

W, H = 1100, 1100
BANDS = 22


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt
    return gbrt


def _scene(kind):
    rng = np.random.default_rng(11)
    if kind == "crowded":  # ~400 balls within reach of a hit
        c = rng.uniform(-3.0, 3.0, (900, 3))
        far = rng.uniform(-40.0, 40.0, (600, 3))
        return S.make_scene(np.concatenate([np.concatenate([c, far]), np.full((1500, 1), 0.5)], 1))
    if kind == "tubes":
        p = rng.uniform(-14.0, 14.0, (700, 3))
        q = p + rng.normal(0.0, 2.0, p.shape)
        sph = np.concatenate([p[:300], np.full((300, 1), 0.6)], 1)
        return S.make_scene(sph, np.concatenate([p, q, np.full((700, 1), 0.45)], 1))
    return S.globule(1500, 1425, 27.0, seed=3)


def _camera(sc, kind, aa):
    if kind == "inside":
        return S.Camera(eye=(0.0, 0.0, 0.0), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0), right=(1.0, 0.0, 0.0),
                        half_w=1.0, half_h=1.0, kind=S.CAMERA_PINHOLE)
    return dataclasses.replace(S.ortho_camera(sc, W // aa, H // aa, angle_deg=20.0), aa=aa)


def _outputs(torch, w, h, aa):
    return (torch.full((h, w, 3), -1.0, device="cuda"),
            torch.full((aa * h, aa * w), -7, dtype=torch.int32, device="cuda"),
            torch.full((aa * h, aa * w), -7, dtype=torch.int32, device="cuda"))


def _in_bands(G, ctx, scene, grid, cam, w, h, lights, p, out, bands=BANDS):
    for k in range(bands):
        rows = (k * h // bands, (k + 1) * h // bands)
        G.gbrt_render_batch(ctx, [G.make_item(scene, grid, cam, w, h, p.ao_samples, lights, p, *out, rows=rows)])


@pytest.mark.parametrize("kind,spp,shadows,eps,aa", [
    ("globule", 8, False, 1e-3, 1), ("globule", 16, False, 1e-3, 1), ("globule", 17, False, 1e-3, 1),
    ("globule", 34, True, 1e-3, 1), ("globule", 16, True, 0.0, 1), ("globule", 12, False, 1e-3, 2),
    ("inside", 16, False, 1e-3, 1), ("crowded", 16, False, 1e-3, 1), ("tubes", 16, True, 1e-3, 1)])
def test_same_frame_with_and_without_the_near_pass(G, kind, spp, shadows, eps, aa):
    import torch
    sc = _scene(kind)
    w, h = W // aa, H // aa
    cam, lights = _camera(sc, kind, aa), S.default_lights()
    p = S.Params(ao_samples=spp, seed=5, eps=eps, shadows=shadows)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=8.0)
        got, ref = _outputs(torch, w, h, aa), _outputs(torch, w, h, aa)
        n0 = G.gbrt_launch_count(R.ctx)
        G.gbrt_render(R.ctx, scene, grid, cam, w, h, spp, lights, p, *got)
        n1 = G.gbrt_launch_count(R.ctx)
        _in_bands(G, R.ctx, scene, grid, cam, w, h, lights, p, ref)
        n2 = G.gbrt_launch_count(R.ctx)
        G.gbrt_sync(R.ctx)
        resolve = 1 if aa > 1 else 0
        assert n1 - n0 == 4 + resolve and n2 - n1 == BANDS * (3 + resolve)
        for a, b in zip(got, ref):
            assert torch.equal(a, b)


def test_rebuilt_grid_and_mixed_batch(G):
    import torch
    base = _scene("globule")
    lights = S.default_lights()
    with G.Renderer(0) as R:
        scene, grid = R.upload(base, lam=8.0)
        other, ogrid = R.upload(_scene("tubes"), lam=2.0)
        moved = S.MDTrajectory(base, amplitude=0.4, spin_deg=30.0, seed=1).frame(3)
        G.gbrt_scene_update(R.ctx, scene, moved.spheres, moved.cylinders)
        G.gbrt_grid_rebuild(R.ctx, grid, scene)
        frames = [(scene, grid, moved, W, H, S.Params(ao_samples=20, seed=1)),
                  (other, ogrid, _scene("tubes"), 300, 211, S.Params(ao_samples=40, seed=2, ao_maxdist=5.0)),
                  (other, ogrid, _scene("tubes"), 517, 400, S.Params(ao_samples=16, seed=3, shadows=True)),
                  (scene, grid, moved, 200, 200, S.Params(ao_samples=0, seed=4))]
        got, ref, items = [], [], []
        for sh, gh, sc, w, h, p in frames:
            cam = S.ortho_camera(sc, w, h)
            out = _outputs(torch, w, h, 1)
            items.append(G.make_item(sh, gh, cam, w, h, p.ao_samples, lights, p, *out))
            got += out
            out = _outputs(torch, w, h, 1)
            _in_bands(G, R.ctx, sh, gh, cam, w, h, lights, p, out, 22 if w > 400 else 1)
            ref += out
        n0 = G.gbrt_launch_count(R.ctx)
        G.gbrt_render_batch(R.ctx, items, G.BATCH_GRAPH)
        assert G.gbrt_launch_count(R.ctx) - n0 == 5  # one of them copies the rebuilt geometry
        G.gbrt_render_batch(R.ctx, items, G.BATCH_GRAPH)
        G.gbrt_sync(R.ctx)
        for a, b in zip(got, ref):
            assert torch.equal(a, b)


@pytest.mark.parametrize("kind,spp,shadows,eps,far", [
    ("globule", 16, False, 1e-3, 0.0), ("globule", 9, True, 1e-3, 0.0), ("globule", 17, False, 0.0, 0.0),
    ("globule", 16, False, 1e-3, 3000.0), ("inside", 8, False, 1e-3, 0.0), ("tubes", 16, True, 1e-3, 0.0),
    ("crowded", 16, False, 1e-3, 0.0)])
def test_fp64_frame_with_and_without_the_near_pass(G, kind, spp, shadows, eps, far):
    # far: the molecule stands away from the origin, where an FP32 coordinate
    # is 2e-4 wide
    import torch
    sc = _scene(kind)
    if far:
        shift = np.array([far, -far, 0.5 * far])
        sph, cyl = sc.spheres.copy(), sc.cylinders.copy()
        sph[:, :3] += shift
        cyl[:, :3] += shift
        cyl[:, 3:6] += shift
        sc = S.make_scene(sph, cyl)
    cam, lights = _camera(sc, kind, 1), S.default_lights()
    p = S.Params(ao_samples=spp, seed=5, eps=eps, shadows=shadows, precision=S.PRECISION_FP64)

    def outputs():
        return (torch.full((H, W, 3), -1.0, device="cuda", dtype=torch.float64),) + _outputs(torch, W, H, 1)[1:]

    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=8.0)
        got, ref = outputs(), outputs()
        n0 = G.gbrt_launch_count(R.ctx)
        G.gbrt_render(R.ctx, scene, grid, cam, W, H, spp, lights, p, *got)
        n1 = G.gbrt_launch_count(R.ctx)
        _in_bands(G, R.ctx, scene, grid, cam, W, H, lights, p, ref)
        n2 = G.gbrt_launch_count(R.ctx)
        G.gbrt_sync(R.ctx)
        assert n1 - n0 == 4 and n2 - n1 == BANDS * 3
        for a, b in zip(got, ref):
            assert torch.equal(a, b)
