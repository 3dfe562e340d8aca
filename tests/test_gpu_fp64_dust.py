"""FP64 frames of objects a hundred million and more times smaller than the
scene, seen from close by: FP32 coordinates of the scene are coarser than the
object, its hits are FP64's all the same. Against the oracle's brute force."""
import numpy as np
import pytest

from paper_0801_1500_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1e-1, 1e-3, 1e-4, 1e-5, 1e-6])
def test_tiny_objects_in_a_large_scene(oracle, r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0801_1500_gb300 import gbrt as G
    rng = np.random.default_rng(8)
    sph = [[-4999.0, -4999.0, -4999.0, 1.0], [4999.0, 4999.0, 4999.0, 1.0]]
    cyl = []
    at = rng.uniform(-3000.0, 3000.0, (12, 3)).astype(np.float32).astype(np.float64)
    for k, c in enumerate(at):
        if k % 3 == 2:
            p1 = (c + [0.0, 40.0 * max(r, 1e-4), 0.0]).astype(np.float32)
            cyl.append([*c, *p1, r])
        else:
            sph.append([*c, r])
    sc = S.make_scene(np.array(sph), np.array(cyl))
    p = S.Params(ao_samples=3, seed=2, eps=0.01 * r, precision=S.PRECISION_FP64)
    lights = S.default_lights()
    with G.Renderer(0) as R:
        scene, grid = R.upload(sc, lam=50.0)
        for c in at:
            for depth in (6000.0, 10.0):
                cam = S.Camera(eye=(c[0], c[1], c[2] + depth), dir=(0.0, 0.0, -1.0), up=(0.0, 1.0, 0.0),
                               right=(1.0, 0.0, 0.0), half_w=1.3 * r, half_h=1.3 * r)
                _, ids, _ = R.render(scene, grid, cam, 40, 40, lights, p, ids=True, vis=True)
                G.gbrt_sync(R.ctx)
                ids = ids.cpu().numpy().view(np.uint32).ravel()
                ref = oracle.render(sc, cam, 40, 40, lights, p, mode="brute")
                assert (ref["id"] != 0xffffffff).sum() > 300
                assert np.array_equal(ids, ref["id"]), (tuple(c), depth, int((ids != ref["id"]).sum()))
