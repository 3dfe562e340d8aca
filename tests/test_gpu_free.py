"""Freeing scenes and grids beside other work: a stream capture of another
thread goes on, and work of other streams that reads the freed memory is waited
for."""
import threading

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


def test_free_leaves_another_threads_capture_alone(G):
    import torch
    sc = S.globule(200, 190, 12.0, seed=1)
    x = torch.zeros(1000, device="cuda")
    failed = []

    def other():
        try:
            with G.Renderer(0, stream=torch.cuda.Stream()) as R:
                scene, grid = G.gbrt_scene_upload(R.ctx, sc.spheres, sc.cylinders, sc.color_idx, sc.palette), None
                grid = G.gbrt_grid_build(R.ctx, scene, 4.0)
                G.gbrt_grid_free(R.ctx, grid)
                G.gbrt_scene_free(R.ctx, scene)
        except Exception as e:  # reported by the test's thread
            failed.append(e)

    other()  # (module loading and first allocations, outside the capture)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        x += 1.0
        t = threading.Thread(target=other)
        t.start()
        t.join()
        x += 1.0
    graph.replay()
    torch.cuda.synchronize()
    assert not failed, failed
    assert bool((x == 2.0).all())


@pytest.mark.parametrize("how", ["render", "noalloc", "probe", "update", "freed_by_another"])
def test_free_waits_for_other_streams(G, how):
    import torch
    sc = S.globule(200, 190, 12.0, seed=1)
    cam, p = S.ortho_camera(sc, 64, 64), S.Params(ao_samples=4)
    lights = S.default_lights()
    with G.Renderer(0) as A, G.Renderer(0, stream=torch.cuda.Stream()) as B:
        rgb = torch.zeros((64, 64, 3), device="cuda")
        owner = B if how == "freed_by_another" else A
        scene = G.gbrt_scene_upload(owner.ctx, sc.spheres, sc.cylinders, sc.color_idx, sc.palette)
        grid = G.gbrt_grid_build(owner.ctx, scene, 4.0)
        pts = torch.zeros((1, 3), dtype=torch.float64, device="cuda")
        nrm = torch.tensor([[0.0, 0.0, 1.0]], dtype=torch.float64, device="cuda")
        new = [torch.from_numpy(a).cuda() for a in (sc.spheres, sc.cylinders)]
        out = torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
        done = torch.cuda.Event()
        with torch.cuda.stream(B.stream):
            torch.cuda._sleep(60_000_000)
        if how == "noalloc":
            G.gbrt_render_noalloc(scene, grid, cam, 64, 64, 4, lights, p, rgb, stream=B.stream)
        elif how == "probe":
            G.gbrt_ao_probe(B.ctx, scene, grid, pts, nrm, 4, p, out)
        elif how == "update":
            G.gbrt_scene_update(B.ctx, scene, new[0], new[1], G.DEVICE_PTRS)
        else:
            G.gbrt_render(B.ctx, scene, grid, cam, 64, 64, 4, lights, p, rgb)
        done.record(B.stream)
        if how == "update":  # the grid has not been read there
            G.gbrt_scene_free(A.ctx, scene)
            assert done.query()
            G.gbrt_grid_free(A.ctx, grid)
        else:
            G.gbrt_grid_free(A.ctx, grid)
            assert done.query()
            G.gbrt_scene_free(A.ctx, scene)
        torch.cuda.synchronize()
