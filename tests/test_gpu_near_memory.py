"""The near pass is an option: a frame whose pass finds no memory for its
records is rendered without it, with the same bits."""
import math

import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def test_a_frame_without_memory_for_the_pass():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
    W = H = 3000  # the pass wants some 70 MB
    sc = S.globule(1500, 1425, 27.0, seed=3)
    cam, lights = S.ortho_camera(sc, W, H), S.default_lights()
    rgb = [torch.zeros((H, W, 3), device="cuda") for _ in range(2)]
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=8.0)

        def render(out, dist):
            n0 = G.gbrt_launch_count(R.ctx)
            p = S.Params(ao_samples=8, seed=2, ao_maxdist=dist)
            G.gbrt_render(R.ctx, scene, grid, cam, W, H, 8, lights, p, out)
            G.gbrt_sync(R.ctx)
            return G.gbrt_launch_count(R.ctx) - n0

        assert render(rgb[0], 1e6) == 3  # what every frame needs is there now
        torch.cuda.empty_cache()
        fill, size = [], 1 << 38
        while size >= 1 << 21:
            if torch.cuda.mem_get_info()[0] >= size + (24 << 20):
                fill.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            else:
                size >>= 1
        assert torch.cuda.mem_get_info()[0] < 48 << 20
        assert render(rgb[0], math.inf) == 3
        fill.clear()
        torch.cuda.empty_cache()
        assert render(rgb[1], math.inf) == 4
        assert torch.equal(*rgb)
