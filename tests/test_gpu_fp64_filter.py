"""The FP64 path settles a (ray, object) pair in FP32 where the FP32 error
bounds allow it and in FP64 elsewhere; either way the decision is the FP64
one. Scenes that stress the bounds -- radii from 0.02 to 300, tubes much longer
than wide, coordinates far from the origin, a finite AO distance -- against the
oracle's brute force. Samples are random and the two FP64 evaluations differ by
at most ~1e-12 of a radius squared, so a sample that they decide differently is
a one-in-10^9 event: hit ids and AO counts must be equal."""
import math

import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _scene(kind):
    rng = np.random.default_rng(5)
    n = 300
    c = rng.uniform(-9.0, 9.0, (n, 3))
    r = rng.uniform(0.4, 1.3, n)
    p = rng.uniform(-9.0, 9.0, (120, 3))
    q = p + rng.normal(0.0, 2.0, p.shape)
    tr = np.full((120, 1), 0.3)
    off = 0.0
    if kind == "small_radii":
        r = np.exp(rng.uniform(math.log(0.02), math.log(2.0), n))
        tr = np.exp(rng.uniform(math.log(0.01), math.log(0.5), (120, 1)))
    elif kind == "long_tubes":
        q = p + rng.normal(0.0, 30.0, p.shape)
        q[:20] = p[:20] + [0.0, 0.0, 25.0]      # along the view
    elif kind == "large_balls":
        c[0], r[0] = (0.0, 0.0, -310.0), 300.0  # a floor
        c[1], r[1] = (0.0, 0.0, 0.0), 12.0      # atoms inside another
    elif kind == "far_off":
        off = 2700.0
    sph = np.concatenate([c + off, r[:, None]], 1)
    cyl = np.concatenate([p + off, q + off, tr], 1)
    return S.make_scene(sph, cyl)


@pytest.mark.parametrize("kind,maxdist", [("small_radii", math.inf), ("long_tubes", math.inf), ("large_balls", math.inf),
                                          ("far_off", math.inf), ("small_radii", 2.5), ("long_tubes", 6.0)])
def test_fp64_decisions_equal_the_oracle(oracle, kind, maxdist):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
    sc = _scene(kind)
    W, H = 61, 47
    ctr = sc.spheres[2:, :3].mean(0).astype(np.float64)
    eye = ctr + [0.0, 0.0, 40.0]
    cam = S.Camera(eye=tuple(eye), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0), right=(1.0, 0.0, 0.0), half_w=11.0,
                   half_h=9.0)
    p = S.Params(ao_samples=12, seed=77, precision=S.PRECISION_FP64, ao_maxdist=maxdist, shadows=True)
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=4.0)
        rgb, ids, vis = R.render(scene, grid, cam, W, H, S.default_lights(), p, ids=True, vis=True)
        G.gbrt_sync(R.ctx)
    ref = oracle.render(sc, cam, W, H, S.default_lights(), p, mode="brute")
    assert np.array_equal(ids.cpu().numpy().view(np.uint32).ravel(), ref["id"])
    assert np.array_equal(vis.cpu().numpy().view(np.uint32).ravel(), ref["vis"].astype(np.uint32))
    assert np.abs(rgb.cpu().numpy().reshape(-1, 3) - ref["rgb"]).max() < 1e-9
