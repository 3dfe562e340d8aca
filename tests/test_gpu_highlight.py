"""FP64 highlights with a whole Phong exponent are formed by squaring, others by
pow(). An exponent one unit in the last place away takes the other way and moves
x^p by at most max_x |x^p ln x| dp = dp / (e p) (dp: the step, p 2^-52 or less),
so the colours, sums of a few terms of at most 1, agree to a few 2^-53 (pow's
own error is 1 ulp): 1e-14."""
import math

import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1.0, 2.0, 3.0, 40.0, 63.0, 255.0, 1023.0, 1024.0])
def test_whole_exponents_match_pow(p):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
    sc = S.globule(60, 57, 6.0, seed=2)
    cam, lights = S.ortho_camera(sc, 160, 120, angle_deg=10.0), S.default_lights()
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=2.0)
        rgb = []
        for e in (p, math.nextafter(p, 1e9)):
            q = S.Params(ao_samples=2, seed=1, precision=S.PRECISION_FP64, k_s=0.7, phong_exp=e)
            rgb.append(R.render(scene, grid, cam, 160, 120, lights, q)[0])
        G.gbrt_sync(R.ctx)
        assert float((rgb[0] - rgb[1]).abs().max()) <= 1e-14
        assert float(rgb[0].max()) > 0.2
