"""What a user of the ray tracer has it do, as cases that can be timed.

A case is one call (or the few calls that belong together) through the C ABI's
binding, on seeded molecular globules of the sizes this repository renders:
1,014 to 249,990 objects, frames from a thumbnail to 3860 x 4548 pixels, 4 to
64 ambient-occlusion samples, both precisions, both cameras. The kinds:

  render    one frame into device memory (gbrt_render)
  noalloc   a small frame without any allocation (gbrt_render_noalloc)
  orbit     frames around one scene as one graph-replayed batch
  wave      row bands of requests on several resident scenes as one batch
  md        new geometry from page-locked host memory, grid rebuild, render,
            image copied back to the host
  load      scene upload and grid build from host arrays, a preview, free
  probe     ambient occlusion at given surface points (gbrt_ao_probe)

`exact` is a brute-force FP64 tracer over all objects, written from the
formulas the library documents, for the cases small enough for it.
"""
import math

import numpy as np
import torch

from paper_0801_1500_gb300 import gbrt as G
from paper_0801_1500_gb300 import scenes as S

CHAIN = 20       # atoms per chain
DENSITY = 13500 / 60.0 ** 3  # atoms per cubed globule radius of the paper-sized scene
LIGHTS = ((-0.1, 0.1, 1.0), (1.0, 2.0, 0.5))
K_AO, K_D, K_S, PHONG, EPS, SCALE, SKY = 0.6, 0.65, 0.4, 40.0, 1e-3, 0.3, 1.0
MISS = 0xFFFFFFFF


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, spheres=13500, cylinders=12818, width=965, height=1137, spp=16, fp64=False,
             pinhole=False, aa=1, shadows=False, maxdist=0.0, lam=8.0, ids=False)
    c.update(kw)
    return c


def listed():
    return [
        # a molecule viewer's thumbnail in a loop that must not allocate
        _case("thumbnail_noalloc", "noalloc", spheres=520, cylinders=494, width=128, height=96, spp=4, ids=True),
        # the smallest request the server takes (smallest resident scene, 256 x 256, 4 samples)
        _case("preview_256", "render", spheres=520, cylinders=494, width=256, height=256, spp=4),
        # the small all-double frame: 2,000 atoms, 1,900 bonds, hit ids and sample counts wanted
        _case("small_fp64", "render", spheres=2000, cylinders=1900, width=256, height=256, spp=8, fp64=True, ids=True),
        # the paper's frame: 26,318 objects at 965 x 1137
        _case("paper_1mp", "render"),
        # the same frame in all-double arithmetic, as the paper computed it
        _case("paper_1mp_fp64", "render", fp64=True),
        # the paper's largest frame
        _case("paper_17mp", "render", width=3860, height=4548),
        # a figure for print: perspective, 2 x 2 sub-pixel rays, shadowed lights
        _case("figure_aa2_shadows", "render", pinhole=True, aa=2, shadows=True),
        # the largest resident scene on a video frame with many samples
        _case("large_1080p_spp64", "render", spheres=128200, cylinders=121790, width=1920, height=1080, spp=64),
        # a turntable: 16 frames around the molecule, uneven sizes and sample counts
        _case("orbit_16", "orbit", frames=16),
        # one wave of the serving loop: bands of mixed requests on four resident scenes
        _case("serve_wave", "wave", frames=10, spheres=0, cylinders=0),
        # one frame of a simulation's trajectory, from host coordinates to host image
        _case("md_frame", "md"),
        # occlusion baked at 8,192 surface points, 64 samples each
        _case("probe_bake", "probe", frames=8192, spp=64, maxdist=20.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "noalloc", "orbit", "wave", "md", "load", "probe"])
    n_chains = _log(rng, 26, 6410)
    s = n_chains * CHAIN + rng.randrange(0, CHAIN)
    fp64 = rng.random() < 0.3
    c = _case("", kind, spheres=s, cylinders=s - n_chains, fp64=fp64, spp=_log(rng, 4, 64),
              pinhole=rng.random() < 0.35, shadows=rng.random() < 0.25,
              maxdist=rng.choice([0.0, 0.0, 0.0, 12.0]), lam=rng.choice([8.0, 8.0, 8.0, 2.0]), ids=rng.random() < 0.3)
    del c["name"]
    w, h = _log(rng, 96, 2600), _log(rng, 96, 2600)
    if kind == "noalloc":
        w, h = min(w, 256), min(h, 256)
    if kind == "render":
        c["aa"] = rng.choice([1, 1, 1, 2, 3])
    if kind in ("orbit", "wave"):
        c["frames"] = rng.randrange(2, 13)
        c["fp64"] = False
    if kind == "probe":
        c["frames"] = _log(rng, 16, 20000)
        c["maxdist"] = rng.choice([0.0, 8.0, 30.0])
    c["width"], c["height"] = w, h
    # no dearer than the largest listed frame
    rays = (c["frames"] if kind == "probe" else w * h * c["aa"] ** 2) * (c["spp"] + 1)
    most = 8e6 if c["fp64"] else 6e7
    if kind not in ("orbit", "wave") and rays > most:
        f = math.sqrt(most / rays)
        c["width"], c["height"] = max(33, int(w * f)), max(33, int(h * f))
        c["spp"] = max(2, min(c["spp"], int(most / (c["width"] * c["height"] * c["aa"] ** 2))))
        if kind == "probe":
            c["frames"] = max(16, int(c["frames"] * f * f))
    return c


# ---------------------------------------------------------------- inputs

def _globule(n_s, n_c, rng):
    """Chains of atoms as random walks of 3.8 A steps inside a ball, bonds
    between neighbours (the recipe of scenes.globule, all chains at once)."""
    radius = (n_s / DENSITY) ** (1.0 / 3.0)
    n_ch = n_s - n_c
    lengths = np.full(n_ch, n_s // n_ch)
    lengths[:n_s % n_ch] += 1

    def unit(n):
        v = rng.standard_normal((n, 3))
        return v / np.linalg.norm(v, axis=1, keepdims=True)

    p = unit(n_ch) * (0.9 * radius * rng.random((n_ch, 1)) ** (1.0 / 3.0))
    steps = [p]
    for _ in range(int(lengths.max()) - 1):
        q = p + 3.8 * unit(n_ch)
        for _ in range(100):
            out = np.flatnonzero((q * q).sum(1) > radius * radius)
            if not len(out):
                break
            q[out] = p[out] + 3.8 * unit(len(out))
        else:
            q[out] = p[out] * (1.0 - 3.8 / np.maximum(np.linalg.norm(p[out], axis=1, keepdims=True), 3.8))
        steps.append(q)
        p = q
    walk = np.stack(steps, 1)                                    # [chain, step, 3]
    used = np.arange(walk.shape[1])[None, :] < lengths[:, None]
    centres = walk[used]
    chain = np.repeat(np.arange(n_ch), lengths)
    spheres = np.concatenate([centres, rng.uniform(1.2, 2.0, (n_s, 1))], 1).astype(np.float32)
    bond = np.flatnonzero(chain[1:] == chain[:-1])
    cyl = np.concatenate([spheres[bond, :3], spheres[bond + 1, :3], np.full((len(bond), 1), 0.3)], 1).astype(np.float32)
    colour = np.concatenate([chain, chain[bond]]).astype(np.uint32) % 16
    return S.Scene(spheres=spheres, cylinders=cyl, color_idx=colour,
                   palette=rng.uniform(0.35, 1.0, (16, 3)).astype(np.float32), radius=radius)


def _moved(sc, rng):
    """The same molecule a little later: every atom displaced, bonds following."""
    sp = sc.spheres.copy()
    sp[:, :3] += rng.normal(0.0, 0.2, (len(sp), 3)).astype(np.float32)
    n_ch = len(sp) - len(sc.cylinders)
    lengths = np.full(n_ch, len(sp) // n_ch)
    lengths[:len(sp) % n_ch] += 1
    chain = np.repeat(np.arange(n_ch), lengths)
    bond = np.flatnonzero(chain[1:] == chain[:-1])
    cy = np.concatenate([sp[bond, :3], sp[bond + 1, :3], sc.cylinders[:, 6:7]], 1).astype(np.float32)
    return S.Scene(spheres=sp, cylinders=cy, color_idx=sc.color_idx, palette=sc.palette, radius=sc.radius)


def _camera(sc, w, h, angle, pinhole, aa=1):
    """A view of the whole ball from `angle` degrees about +y."""
    r = 1.05 * (sc.radius + 2.0)
    th = math.radians(angle)
    back, right = (math.sin(th), 0.0, math.cos(th)), (math.cos(th), 0.0, -math.sin(th))
    if pinhole:
        hh = math.tan(math.radians(15.0)) * max(1.0, h / w)
        hw, dist = hh * w / h, r / math.sin(math.radians(15.0))
    else:
        hh = r * max(1.0, h / w)
        hw, dist = hh * w / h, 1.8 * r + 1.0
    return S.Camera(eye=tuple(dist * b for b in back), dir=tuple(-b for b in back), up=(0.0, 1.0, 0.0), right=right,
                    half_w=hw, half_h=hh, kind=S.CAMERA_PINHOLE if pinhole else S.CAMERA_ORTHO, aa=aa)


def _lights():
    n = [np.asarray(v) / np.linalg.norm(v) for v in LIGHTS]
    return S.Lights(dirs=[tuple(float(x) for x in v) for v in n], intensity=[1.0, 1.0], scale=SCALE, skylight=SKY)


def _params(c, seed, frame=0, spp=None):
    return S.Params(ao_samples=c["spp"] if spp is None else spp, seed=seed, frame=frame,
                    precision=S.PRECISION_FP64 if c["fp64"] else S.PRECISION_FP32, eps=EPS,
                    ao_maxdist=c["maxdist"] or math.inf, k_ao=K_AO, k_d=K_D, k_s=K_S, phong_exp=PHONG,
                    shadows=c["shadows"])


def _inputs(c, seed):
    """Everything the seed decides, on the host: scene, camera, parameters."""
    rng = np.random.Generator(np.random.PCG64(seed))
    sc = _globule(c["spheres"], c["cylinders"], rng) if c["spheres"] else None
    angle = float(rng.uniform(0.0, 360.0))
    cam = _camera(sc, c["width"], c["height"], angle, c["pinhole"], c["aa"]) if sc is not None else None
    return rng, sc, cam, _params(c, int(rng.integers(1 << 40)))


def _probe_points(c, sc, rng):
    """Points on atoms, and the atoms' normals there."""
    k = rng.integers(0, len(sc.spheres), c["frames"])
    n = rng.standard_normal((c["frames"], 3))
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    return sc.spheres[k, :3].astype(np.float64) + sc.spheres[k, 3:4].astype(np.float64) * n, n


class _State:
    """Resident context, scenes, grids and outputs of one case."""

    def __init__(self):
        self.r = G.Renderer(0)

    def __del__(self):
        self.r.close()


def _out(c, h, w, m=1, dev="cuda"):
    rgb = torch.zeros((h, w, 3), dtype=torch.float64 if c["fp64"] else torch.float32, device=dev)
    px = [torch.zeros((m * h, m * w), dtype=torch.int32, device=dev) for _ in range(2)] if c["ids"] else [None, None]
    return rgb, px[0], px[1]


def prepare(case, seed):
    c = case
    rng, sc, cam, pa = _inputs(c, seed)
    s = _State()
    s.case, s.lights = c, G.make_lights(_lights())
    kind, w, h = c["kind"], c["width"], c["height"]
    mix = np.random.Generator(np.random.PCG64(c.get("frames", 0)))  # sizes belong to the case, not to the seed
    if kind in ("render", "noalloc"):
        s.scene, s.grid = s.r.upload(sc, lam=c["lam"])
        s.cam, s.pa = G.make_camera(cam), G.make_params(pa)
        s.out = _out(c, h, w, c["aa"])
    elif kind == "orbit":
        s.scene, s.grid = s.r.upload(sc, lam=c["lam"])
        s.items, s.out = [], []
        for k in range(c["frames"]):
            fw, fh = S.ORBIT_RESOLUTIONS[int(mix.integers(3))]
            spp = int(mix.integers(8, 33))
            rgb = torch.zeros((fh, fw, 3), device="cuda")
            cam = _camera(sc, fw, fh, 360.0 * k / c["frames"], False)
            s.items.append(G.make_item(s.scene, s.grid, cam, fw, fh, spp, s.lights, _params(c, k, k, spp), rgb))
            s.out.append(rgb)
    elif kind == "wave":
        res = []
        for n in np.geomspace(26, 6410, 4):
            n = int(round(n))
            sc = _globule(n * CHAIN, n * (CHAIN - 1), rng)
            res.append((sc,) + tuple(s.r.upload(sc, lam=c["lam"])))
        s.items, s.out = [], []
        for k in range(c["frames"]):
            sc, scene, grid = res[int(mix.integers(4))]
            fw, fh = S.SERVE_RESOLUTIONS[int(mix.integers(3))]
            spp = S.SERVE_SPP[int(mix.integers(3))]
            rgb = torch.zeros((fh, fw, 3), device="cuda")
            cam = _camera(sc, fw, fh, float(rng.uniform(0.0, 360.0)), False)
            p = _params(c, k, 0, spp)
            # about 4 million rays of each request, as the wave's ray budget leaves it
            rows = min(fh, max(64, int(4e6 / (fw * (1 + 0.6 * spp))) // 64 * 64))
            first = int(mix.integers(0, (fh - rows) // 64 + 1)) * 64
            for r0 in range(first, first + rows, 64):
                s.items.append(G.make_item(scene, grid, cam, fw, fh, spp, s.lights, p, rgb,
                                           rows=(r0, min(r0 + 64, fh))))
            s.out.append(rgb)
    elif kind == "md":
        s.scene, s.grid = s.r.upload(sc, lam=c["lam"])
        late = _moved(sc, rng)
        s.new = [torch.from_numpy(a).pin_memory().numpy() for a in (late.spheres, late.cylinders)]
        s.cam, s.pa = G.make_camera(cam), G.make_params(pa, out_flags=G.HOST_PTRS | G.HOST_ASYNC)
        s.out = torch.zeros((h, w, 3), dtype=torch.float64 if c["fp64"] else torch.float32).pin_memory()
    elif kind == "load":
        s.sc = sc
        s.cam, s.pa = G.make_camera(cam), G.make_params(pa)
        s.out = _out(c, h, w)
    elif kind == "probe":
        s.scene, s.grid = s.r.upload(sc, lam=c["lam"])
        p, n = _probe_points(c, sc, rng)
        s.pts, s.nrm = torch.from_numpy(p).cuda(), torch.from_numpy(n).cuda()
        s.pa = G.make_params(pa)
        s.out = torch.zeros(c["frames"], device="cuda")
    torch.cuda.synchronize()
    return s


def run(state):
    s, c, r = state, state.case, state.r
    kind, w, h, spp = c["kind"], c["width"], c["height"], c["spp"]
    if kind == "render":
        G.gbrt_render(r.ctx, s.scene, s.grid, s.cam, w, h, spp, s.lights, s.pa, *s.out)
    elif kind == "noalloc":
        G.gbrt_render_noalloc(s.scene, s.grid, s.cam, w, h, spp, s.lights, s.pa, *s.out, stream=r.stream)
    elif kind in ("orbit", "wave"):
        G.gbrt_render_batch(r.ctx, s.items, G.BATCH_GRAPH if kind == "orbit" else 0)
    elif kind == "md":
        G.gbrt_scene_update(r.ctx, s.scene, *s.new)
        G.gbrt_grid_rebuild(r.ctx, s.grid, s.scene)
        G.gbrt_render(r.ctx, s.scene, s.grid, s.cam, w, h, spp, s.lights, s.pa, s.out)
    elif kind == "load":
        scene = G.gbrt_scene_upload(r.ctx, s.sc.spheres, s.sc.cylinders, s.sc.color_idx, s.sc.palette)
        grid = G.gbrt_grid_build(r.ctx, scene, c["lam"])
        info = G.gbrt_grid_info(grid)
        G.gbrt_render(r.ctx, scene, grid, s.cam, w, h, spp, s.lights, s.pa, *s.out)
        G.gbrt_grid_free(r.ctx, grid)
        G.gbrt_scene_free(r.ctx, scene)
        return list(s.out) + [np.array(info["dims"]), np.array(info["lo"] + info["hi"])]
    elif kind == "probe":
        G.gbrt_ao_probe(r.ctx, s.scene, s.grid, s.pts, s.nrm, spp, s.pa, s.out)
    return s.out


def work(case):
    """Scene and results moved once; per primary ray 80 flops (ray, the one
    hit that counts, shading), per AO ray 100 (its sample's direction and the
    few objects that decide it). Six tenths of a frame's pixels hit the ball."""
    c = case
    objects = c["spheres"] + c["cylinders"]
    real = 8 if c["fp64"] else 4
    if c["kind"] == "probe":
        return {"bytes": 36.0 * objects + 52.0 * c["frames"], "flops": 100.0 * c["frames"] * c["spp"]}
    if c["kind"] == "orbit":
        px, spp = 1.15e6 * c["frames"], 20
    elif c["kind"] == "wave":
        objects, px, spp = 163000, 4e5 * c["frames"], 16
    else:
        px, spp = float(c["width"] * c["height"]), c["spp"]
    rays = px * c["aa"] ** 2
    return {"bytes": 36.0 * objects + 3 * real * px + (8.0 * rays if c["ids"] else 0.0),
            "flops": rays * (80.0 + 0.6 * 100.0 * (spp + (2 if c["shadows"] else 0)))}


# ---------------------------------------------------------------- the same in 64 bits

def _tables(sc, dev):
    """p0, axis, length, radius of every object; a sphere has no axis."""
    sp, cy = sc.spheres.astype(np.float64), sc.cylinders.astype(np.float64)
    ax = cy[:, 3:6] - cy[:, 0:3]
    ln = np.linalg.norm(ax, axis=1)
    p0 = np.concatenate([sp[:, :3], cy[:, :3]])
    a = np.concatenate([np.zeros((len(sp), 3)), ax / np.maximum(ln, 1e-300)[:, None]])
    return [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in
            (p0, a, np.concatenate([np.zeros(len(sp)), ln]), np.concatenate([sp[:, 3], cy[:, 6]]))]


def _roots(obj, o, d):
    """Both roots of every ray with every object, NaN where there is none."""
    p0, a, ln, r = obj
    wd = (o * d).sum(1)[:, None] - d @ p0.T
    ww = (o * o).sum(1)[:, None] - 2.0 * (o @ p0.T) + (p0 * p0).sum(1)[None, :]
    wa, da = o @ a.T - (p0 * a).sum(1)[None, :], d @ a.T
    A = 1.0 - da * da
    B = wd - wa * da
    q = torch.sqrt(B * B - A * (ww - wa * wa - (r * r)[None, :]))
    out = []
    for sign in (-1.0, 1.0):
        t = (sign * q - B) / A
        axial = wa + t * da
        out.append(torch.where((axial >= 0.0) & (axial <= ln[None, :]), t, torch.full_like(t, math.nan)))
    return out


def _chunks(n_rays, n_obj):
    step = max(1, int(3e7 / max(1, n_obj)))
    for k in range(0, n_rays, step):
        yield slice(k, min(n_rays, k + step))


def _nearest(obj, o, d):
    t, i = o.new_full((len(o),), math.inf), torch.zeros(len(o), dtype=torch.int64, device=o.device)
    for s in _chunks(len(o), len(obj[3])):
        t0, t1 = _roots(obj, o[s], d[s])
        best = torch.where(t0 > 0.0, t0, torch.where(t1 > 0.0, t1, torch.full_like(t1, math.inf)))
        t[s], i[s] = best.min(1)
    return t, i


def _blocked(obj, o, d, tmax):
    hit = torch.zeros(len(o), dtype=torch.bool, device=o.device)
    for s in _chunks(len(o), len(obj[3])):
        for t in _roots(obj, o[s], d[s]):
            hit[s] |= ((t > 0.0) & (t <= tmax)).any(1)
    return hit


def _philox(q, s, frame, seed):
    """The two sample uniforms of Philox4x32-10, counter (q, s, frame, 0xA0)."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [q.astype(np.uint64), s.astype(np.uint64), np.full(q.shape, frame, np.uint64), np.full(q.shape, 0xA0, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [(c[j] >> np.uint64(8)).astype(np.float64) / 16777216.0 for j in (0, 1)]


def _directions(n, u1, u2):
    """Cosine-weighted directions about n in the basis of Duff et al. 2017."""
    nx, ny, nz = n.unbind(1)
    sign = torch.where(nz.signbit(), -1.0, 1.0).to(n.dtype)
    a = -1.0 / (sign + nz)
    b = nx * ny * a
    e1 = torch.stack([1.0 + sign * nx * nx * a, sign * b, -sign * nx], 1)
    e2 = torch.stack([b, sign + ny * ny * a, -ny], 1)
    rr, phi = torch.sqrt(u1), 2.0 * math.pi * u2
    return (rr * torch.cos(phi))[:, None] * e1 + (rr * torch.sin(phi))[:, None] * e2 + torch.sqrt(1.0 - u1)[:, None] * n


def _visibility(obj, o, n, q, spp, frame, seed, tmax):
    """Share of the samples of each point that escape."""
    if spp == 0:
        return o.new_ones(len(o))
    dev = o.device
    k = torch.arange(len(o), device=dev).repeat_interleave(spp)
    smp = np.tile(np.arange(spp), len(o))
    u1, u2 = (torch.from_numpy(u).to(dev) for u in _philox(q.cpu().numpy().repeat(spp), smp, frame, seed))
    hit = _blocked(obj, o[k], _directions(n[k], u1, u2), tmax)
    return 1.0 - hit.double().reshape(-1, spp).mean(1)


def exact(case, seed):
    c = case
    objects = c["spheres"] + c["cylinders"]
    if c["kind"] == "probe":
        if float(c["frames"]) * c["spp"] * objects > 3e10:
            return None
        rng, sc, _, pa = _inputs(c, seed)
        p, n = (torch.from_numpy(x).cuda() for x in _probe_points(c, sc, rng))
        obj = _tables(sc, "cuda")
        return _visibility(obj, p + EPS * n, n, torch.arange(len(p)), c["spp"], 0, pa.seed, pa.ao_maxdist)
    if c["kind"] in ("orbit", "wave", "md") or c["aa"] > 1 or \
            float(c["width"] * c["height"]) * (1.0 + 0.6 * (c["spp"] + 2)) * objects > 3e10:
        return None
    _, sc, cam, pa = _inputs(c, seed)
    dev, w, h = "cuda", c["width"], c["height"]
    obj = _tables(sc, dev)
    vec = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
    q = torch.arange(w * h, device=dev)
    u = cam.half_w * (2.0 * ((q % w).double() + 0.5) / w - 1.0)
    v = cam.half_h * (1.0 - 2.0 * ((q // w).double() + 0.5) / h)
    off = u[:, None] * vec(cam.right) + v[:, None] * vec(cam.up)
    if c["pinhole"]:
        o, d = vec(cam.eye).expand(w * h, 3).contiguous(), off + vec(cam.dir)
        d = d / d.norm(dim=1, keepdim=True)
    else:
        o, d = vec(cam.eye) + off, vec(cam.dir).expand(w * h, 3).contiguous()
    t, i = _nearest(obj, o, d)
    rgb = torch.zeros((w * h, 3), dtype=torch.float64, device=dev)
    hit = torch.isfinite(t)
    o, d, t, i, q = o[hit], d[hit], t[hit], i[hit], q[hit]
    p0, a, _, r = (x[i] for x in obj)
    p = o + t[:, None] * d
    foot = p0 + ((p - p0) * a).sum(1, keepdim=True) * a
    n = (p - foot) / (p - foot).norm(dim=1, keepdim=True)
    p = foot + r[:, None] * n
    n = torch.where(((n * d).sum(1) > 0.0)[:, None], -n, n)
    o = p + EPS * n
    amb = SKY * K_AO * _visibility(obj, o, n, q, c["spp"], 0, pa.seed, pa.ao_maxdist)
    spec = torch.zeros_like(amb)
    for x in LIGHTS:
        light = vec(x) / vec(x).norm()
        ndl = (n * light).sum(1)
        lit = ndl > 0.0
        if c["shadows"]:
            lit &= ~_blocked(obj, o, light.expand_as(o).contiguous(), math.inf)
        rv = (-(2.0 * ndl[:, None] * n - light) * d).sum(1).clamp(min=0.0)
        amb = amb + torch.where(lit, SCALE * K_D * ndl, 0.0)
        spec = spec + torch.where(lit, SCALE * K_S * rv ** PHONG, 0.0)
    col = torch.from_numpy(sc.palette.astype(np.float64)[sc.color_idx]).to(dev)[i]
    rgb[hit] = (col * amb[:, None] + spec[:, None]).clamp(0.0, 1.0)
    rgb = rgb.reshape(h, w, 3)
    return [rgb, None, None, None, None] if c["kind"] == "load" else [rgb, None, None]
