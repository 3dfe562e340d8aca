"""A scene updated without a rebuild of its grid: the grid's lists stay those of
the old geometry, which still hold every object whose radius has only shrunk,
and every result is that of the new geometry. The same for a grid that serves a
second scene of as many objects."""
import dataclasses
import math

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


def _scenes():
    old = S.globule(1500, 1425, 27.0, seed=3)
    sph, cyl = old.spheres.copy(), old.cylinders.copy()
    sph[:, 3] *= 0.6
    cyl[:, 6] *= 0.6
    return old, dataclasses.replace(old, spheres=sph, cylinders=cyl)


def _frame(G, R, scene, grid, cam, w, h, p, bands=1):
    import torch
    rgb = torch.full((h, w, 3), -1.0, device="cuda",
                     dtype=torch.float64 if p.precision == S.PRECISION_FP64 else torch.float32)
    px = [torch.full((h, w), -7, dtype=torch.int32, device="cuda") for _ in range(2)]
    for k in range(bands):
        rows = (k * h // bands, (k + 1) * h // bands)
        G.gbrt_render_batch(R.ctx, [G.make_item(scene, grid, cam, w, h, p.ao_samples, S.default_lights(), p, rgb, *px,
                                                rows=rows)])
    return [rgb] + px


@pytest.mark.parametrize("how", ["built", "rebuilt", "other_scene"])
def test_results_are_those_of_the_new_geometry(G, how):
    import torch
    old, new = _scenes()
    cam = S.ortho_camera(old, W, H, angle_deg=20.0)
    rng = np.random.default_rng(2)
    k = rng.integers(0, len(new.spheres), 400)
    n = rng.standard_normal((400, 3))
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    pts = torch.from_numpy(new.spheres[k, :3].astype(np.float64) + new.spheres[k, 3:4].astype(np.float64) * n).cuda()
    nrm = torch.from_numpy(n).cuda()
    with G.Renderer(0) as R:
        scene, grid = R.upload(old, lam=8.0)
        fresh, fgrid = R.upload(new, lam=8.0)
        if how == "rebuilt":
            G.gbrt_grid_rebuild(R.ctx, grid, scene)
        if how == "other_scene":
            scene = fresh
        else:
            G.gbrt_scene_update(R.ctx, scene, new.spheres, new.cylinders)
        for prec in (S.PRECISION_FP32, S.PRECISION_FP64):
            p = S.Params(ao_samples=16, seed=5, shadows=True, precision=prec)
            got = _frame(G, R, scene, grid, cam, W, H, p)
            ref = _frame(G, R, scene, grid, cam, W, H, p, BANDS)
            for a, b in zip(got, ref):
                assert torch.equal(a, b), (prec, int((a != b).sum()))
            for dist in (math.inf, 9.0):
                p.ao_maxdist = dist
                a = _frame(G, R, scene, grid, cam, 300, 300, p)
                b = _frame(G, R, fresh, fgrid, cam, 300, 300, p)
                out = [torch.zeros(400, device="cuda") for _ in range(2)]
                G.gbrt_ao_probe(R.ctx, scene, grid, pts, nrm, 64, p, out[0])
                G.gbrt_ao_probe(R.ctx, fresh, fgrid, pts, nrm, 64, p, out[1])
                if prec == S.PRECISION_FP64:  # decided in FP64 whatever the grid
                    for x, y in zip(a, b):
                        assert torch.equal(x, y), (dist, int((x != y).sum()))
                    assert torch.equal(*out), dist
                else:  # the two grids' walks start at other points: the bits may differ, not the geometry
                    assert (a[0] - b[0]).abs().mean() < 1e-5 and (out[0] - out[1]).abs().mean() < 1e-4
        G.gbrt_sync(R.ctx)
        if how == "other_scene":
            return
        # and with the rebuild the near pass is back
        G.gbrt_grid_rebuild(R.ctx, grid, scene)
        G.gbrt_sync(R.ctx)
        n0 = G.gbrt_launch_count(R.ctx)
        p = S.Params(ao_samples=16, seed=5, shadows=True)
        got = _frame(G, R, scene, grid, cam, W, H, p)
        assert G.gbrt_launch_count(R.ctx) - n0 == 5  # one copies the rebuilt geometry
        for a, b in zip(got, _frame(G, R, scene, grid, cam, W, H, p, BANDS)):
            assert torch.equal(a, b)
