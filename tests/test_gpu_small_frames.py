"""Frames whose work is dealt out in smaller pieces than a large one's: the rays
an AO warp claims at once shrink from 64 to 8 with the frame, and 1, 2, 4 or 8
lanes share a primary ray. A frame and the same frame in bands of a few rows
(other sizes, so other pieces) give the same bits; the sizes lie on both sides
of where the pieces change, with ragged tiles, and one camera stands among the
atoms."""
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


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("w,h,spp", [(3, 2, 1), (41, 30, 3), (140, 101, 3), (131, 97, 4), (258, 247, 4), (301, 290, 7),
                                     (517, 260, 20)])
def test_frame_and_its_bands(G, w, h, spp, precision):
    import torch
    sc = S.globule(1500, 1425, 27.0, seed=4)
    cam, lights = S.ortho_camera(sc, w, h, angle_deg=35.0), S.default_lights()
    if spp == 3:
        cam = S.Camera(eye=(0.0, 0.0, 0.0), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0), right=(1.0, 0.0, 0.0),
                       half_w=1.0, half_h=1.0, kind=S.CAMERA_PINHOLE)
    p = S.Params(ao_samples=spp, seed=9, shadows=spp == 7, precision=G.FP64 if precision == "fp64" else G.FP32)

    def outputs():
        dt = torch.float64 if precision == "fp64" else torch.float32
        return (torch.full((h, w, 3), -1.0, device="cuda", dtype=dt),
                torch.full((h, w), -7, dtype=torch.int32, device="cuda"),
                torch.full((h, w), -7, dtype=torch.int32, device="cuda"))

    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=8.0)
        got, ref = outputs(), outputs()
        G.gbrt_render(R.ctx, scene, grid, cam, w, h, spp, lights, p, *got)
        for r in range(0, h, 8):
            G.gbrt_render_batch(R.ctx, [G.make_item(scene, grid, cam, w, h, spp, lights, p, *ref,
                                                    rows=(r, min(r + 8, h)))])
        G.gbrt_sync(R.ctx)
        assert int((got[1] >= 0).sum()) > 0
        for a, b in zip(got, ref):
            assert torch.equal(a, b)
