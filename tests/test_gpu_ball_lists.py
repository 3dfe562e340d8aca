"""The balls beside a grid's lists: counted, placed and cut right at the edges of
their kernels -- no spheres, no tubes, tubes that do not fill a warp's four
places, objects that do not fill a CTA -- by a host build and by a rebuild. The
near pass reads them, the same frame in row bands does not: same bits. Beside
that the bounding radius, which only objects far out evaluate in full."""
import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu

W, H, BANDS = 1100, 1100, 22


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n_s,n_c,far", [(0, 37, 0.0), (41, 0, 0.0), (33, 1, 0.0), (64, 30, 0.0), (255, 251, 0.0),
                                         (257, 515, 0.0), (300, 290, 2000.0)])
def test_near_pass_on_odd_counts(n_s, n_c, far, fp64):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
    rng = np.random.default_rng(n_s + 7 * n_c)
    p0 = rng.uniform(-6.0, 6.0, (max(n_s, n_c), 3)) + far
    p1 = p0 + rng.normal(0.0, 1.0, p0.shape)
    sph = np.concatenate([p0, rng.uniform(0.5, 1.0, (len(p0), 1))], 1)[:n_s]
    cyl = np.concatenate([p0, p1, np.full((len(p0), 1), 0.3)], 1)[:n_c]
    sc = S.make_scene(sph, cyl)
    cam, lights = S.ortho_camera(sc, W, H, angle_deg=35.0), S.default_lights()
    p = S.Params(ao_samples=16, seed=3, precision=S.PRECISION_FP64 if fp64 else S.PRECISION_FP32)

    def frame(bands):
        rgb = torch.full((H, W, 3), -1.0, device="cuda", dtype=torch.float64 if fp64 else torch.float32)
        px = [torch.full((H, W), -7, dtype=torch.int32, device="cuda") for _ in range(2)]
        n0 = G.gbrt_launch_count(R.ctx)
        for k in range(bands):
            rows = (k * H // bands, (k + 1) * H // bands)
            G.gbrt_render_batch(R.ctx, [G.make_item(scene, grid, cam, W, H, 16, lights, p, rgb, *px, rows=rows)])
        G.gbrt_sync(R.ctx)
        return [rgb] + px, G.gbrt_launch_count(R.ctx) - n0

    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=8.0)
        info = G.gbrt_grid_info(grid)
        for rebuilt in (0, 1):
            if rebuilt:
                G.gbrt_grid_rebuild(R.ctx, grid, scene)
                assert {k: v for k, v in G.gbrt_grid_info(grid).items() if k != "device_bytes"} == \
                    {k: v for k, v in info.items() if k != "device_bytes"}
            got, n = frame(1)
            ref, m = frame(BANDS)
            assert n == 4 + rebuilt and m == (3 + rebuilt) * BANDS
            for a, b in zip(got, ref):
                assert torch.equal(a, b), int((a != b).sum())
