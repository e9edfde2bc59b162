"""The work that users of the rasterizer have it do, as measurable cases.

A case is one call sequence of a user's program through the public entry
points of paper_2003_10558_gb300.vsr, at one size:

  frame   a new lens, new triangles or camera, the picture:
          Map.update, Scene.update, raster
  camera  a moved camera under a cached map: Scene.update, raster
  map     a new lens alone: Map.update (the direction map is the result)
  pstep   the per-fragment pixel step under a cached map with derivatives:
          Scene.update, raster_pstep
  host    a frame from and to pinned host memory: Map.update, render_host
  batch   many views of one scene in one call: Batch.render
  serve   a burst of requests to the rendering server: submit, wait
  grad    a shaded picture and its adjoint for a given upstream gradient:
          Map.update, Scene.update, raster_shaded, raster_backward
  train   the same behind autograd: render_shaded, an L2 loss, its gradients
          with respect to vertices, colours and lens

Scenes are the seeded ones of paper_2003_10558_gb300.scenes; lenses, sizes
and triangle counts are those of the tests and the benchmark, or spread over
the same ranges (draw).  exact() gives the results in 64-bit arithmetic from
the formulas of the method, in plain torch.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2003_10558_gb300 import scenes, vsr

DEV = "cuda"
TILE = 16


def listed():
    return [
        # the smallest picture in use (64 triangles, the tests' tiny scene):
        # launches and latency are everything
        dict(name="frame_tiny", kind="frame", W=256, H=256, k=0.0, l=1.0, s=1.0, omega=180.0, aov=0, T=64, sphere=0,
             rho=10.0, jitter=0.25),
        # the ordinary frame: full HD, a closed environment and 200k small
        # triangles around the eye
        dict(name="frame_1080p", kind="frame", W=1920, H=1080, k=0.32, l=0.62, s=0.86, omega=270.0, aov=0, T=200_000,
             sphere=5, rho=40.0, jitter=0.0192),
        # the largest frame: a wall or dome picture of a million triangles
        dict(name="frame_4096", kind="frame", W=4096, H=2176, k=0.32, l=0.62, s=0.86, omega=270.0, aov=0, T=1_000_000,
             sphere=5, rho=60.0, jitter=0.0096),
        # an odd window size, diagonal angle of view and a lens whose rim is
        # undefined (k < 0)
        dict(name="frame_ragged", kind="frame", W=1013, H=757, k=-0.51, l=0.8, s=0.9, omega=300.0, aov=1, T=60_000,
             sphere=0, rho=40.0, jitter=0.03),
        # a camera inside a cloud of a million triangles: many layers per
        # pixel, many triangles per tile
        dict(name="camera_cloud", kind="camera", W=1024, H=1024, k=0.4, l=0.8, s=0.9, omega=200.0, aov=0, T=1_000_000,
             sphere=0, rho=60.0, jitter=0.0096, eye=5.0),
        # a new lens for a large panorama picture, the map itself wanted
        dict(name="map_8192", kind="map", W=8192, H=4096, k=0.5, l=0.7, s=0.9, omega=240.0, aov=0),
        # the quality setting: every edge with its own pixel step
        dict(name="pstep_720p", kind="pstep", W=1280, H=720, k=0.32, l=0.62, s=0.86, omega=270.0, aov=0, T=100_000,
             sphere=0, rho=40.0, jitter=0.0192),
        # a program without GPU data: triangles in, pictures out
        dict(name="host_1080p", kind="host", W=1920, H=1080, k=0.32, l=0.62, s=0.86, omega=270.0, aov=0, T=200_000,
             sphere=5, rho=40.0, jitter=0.0192),
        # many views of uneven size of one large scene in one call
        dict(name="batch_12_views", kind="batch", views=12, T=1_000_000, rho=60.0, jitter=0.0096),
        # a burst of requests of mixed sizes, lenses and scenes
        dict(name="serve_32", kind="serve", requests=32, T=100_000, T2=300_000, rho=60.0, jitter=0.0096),
        # forward and backward of the differentiable path, full size, in a
        # program with an optimiser of its own
        dict(name="grad_1024", kind="grad", W=1024, H=1024, k=0.6, l=1.0, s=1.0, omega=180.0, T=10_000, jitter=0.05),
        # one step of fitting a lens and a scene to a small picture, as the
        # coarse stages of a fit take it
        dict(name="train_256", kind="train", W=256, H=256, k=0.4, l=0.85, s=0.95, omega=180.0, T=600, jitter=0.12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lens(rng):
    return dict(k=rng.uniform(-1.0, 1.0), l=rng.uniform(0.5, 1.0), s=rng.uniform(0.5, 1.0), omega=rng.uniform(90.0, 360.0),
                aov=rng.choice((0, 0, 1, 2, 3)))


def _size(rng, lo, hi):
    """A width, log-uniform, and a height of a common aspect ratio; every
    other one rounded to whole tiles."""
    W = _log(rng, lo, hi)
    H = max(16, int(W * rng.choice((0.5, 0.53, 0.5625, 0.625, 0.75, 1.0))))
    if rng.random() < 0.5:
        W, H = max(16, W // 16 * 16), max(16, H // 16 * 16)
    return dict(W=W, H=min(H, 2176))


def _triangles(rng, lo, hi, layers=(1.0, 14.0)):
    """T triangles of a size that gives the drawn number of caps per pixel."""
    T = _log(rng, lo, hi)
    j = math.sqrt(4.0 * rng.uniform(*layers) / T) / 0.82
    return dict(T=T, jitter=min(0.25, max(0.0096, j)), rho=rng.uniform(10.0, 60.0))


def draw(rng):
    kind = rng.choice(("frame", "frame", "frame", "camera", "camera", "map", "pstep", "host", "batch", "serve", "grad",
                       "train"))
    if kind == "frame":
        return dict(kind=kind, sphere=rng.choice((0, 3, 5)), **_size(rng, 128, 4096), **_lens(rng),
                    **_triangles(rng, 64, 1_000_000))
    if kind == "camera":
        return dict(kind=kind, sphere=0, eye=rng.uniform(0.0, 5.0), **_size(rng, 256, 2048), **_lens(rng),
                    **_triangles(rng, 1000, 1_000_000))
    if kind == "map":
        c = dict(kind=kind, **_size(rng, 256, 8192), **_lens(rng))
        return c
    if kind == "pstep":
        return dict(kind=kind, sphere=rng.choice((0, 3)), **_size(rng, 256, 1920), **_lens(rng),
                    **_triangles(rng, 500, 200_000))
    if kind == "host":
        return dict(kind=kind, sphere=rng.choice((0, 5)), **_size(rng, 320, 1920), **_lens(rng),
                    **_triangles(rng, 500, 200_000))
    if kind == "batch":
        return dict(kind=kind, views=rng.randint(2, 12), rho=60.0, jitter=0.0096, T=_log(rng, 20_000, 1_000_000))
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(4, 32), rho=60.0, jitter=0.0096, T=_log(rng, 10_000, 100_000),
                    T2=_log(rng, 100_000, 300_000))
    W = _log(rng, 128, 1024)
    T = _log(rng, 100, 10_000)
    return dict(kind=kind, W=W, H=W, k=rng.choice((-1.0, 1.0)) * rng.uniform(0.15, 0.9), l=rng.uniform(0.55, 0.95),
                s=rng.uniform(0.55, 0.95), omega=rng.uniform(120.0, 180.0), T=T,
                jitter=min(0.25, max(0.02, math.sqrt(4.0 * rng.uniform(2.0, 8.0) / T) / 0.82)))


# ---------------------------------------------------------------------------
# Inputs, from the seed alone (host arrays; exact() starts from the same).

def _rotation(rng):
    q, r = np.linalg.qr(rng.normal(size=(3, 3)))
    q = q * np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


def _scene(case, seed, n=None):
    """float32 [T, 3, 3] triangles and a camera of 12 floats."""
    rng = np.random.default_rng([int(seed), 1])
    tris = scenes.random_triangles(case["T"] if n is None else n, 1.0, case["rho"] if "rho" in case else 10.0,
                                   case["jitter"], int(rng.integers(1 << 30)))
    if case.get("sphere"):
        tris = np.concatenate([scenes.icosphere(case["sphere"], case["rho"] + 10.0), tris])
    if case["kind"] == "camera":
        d = rng.normal(size=3)
        eye = d / np.linalg.norm(d) * case["eye"] * rng.uniform(0.5, 1.0)
        return tris, scenes.camera(eye, _rotation(rng))
    # an eye next to the origin: the frames of one program differ in it
    return tris, scenes.camera(rng.uniform(-0.02, 0.02, 3))


def _lens_args(case, seed):
    """(W, H, k, l, s, omega, aov): the case's lens; omega moves with the seed
    by up to one degree."""
    om = case["omega"] - float(np.random.default_rng([int(seed), 2]).uniform(0.0, 1.0))
    return case["W"], case["H"], case["k"], case["l"], case["s"], om, case.get("aov", 0)


def _train_inputs(case, seed):
    rng = np.random.default_rng([int(seed), 3])
    tris = _scene(case, seed)[0]
    colors = rng.uniform(0.2, 1.0, case["T"]).astype(np.float32)
    # the observed picture (or the upstream gradient): a smooth one
    c = rng.uniform(0.0, 1.0, (8, 8))
    y, x = (np.linspace(0.0, 7.0, n) for n in (case["H"], case["W"]))

    def bands(t):
        i = np.minimum(t.astype(int), 6)
        b = np.zeros((len(t), 8))
        b[np.arange(len(t)), i] = 1.0 - (t - i)
        b[np.arange(len(t)), i + 1] = t - i
        return b

    target = (bands(y) @ c @ bands(x).T).astype(np.float32)
    return tris, colors, target


def _views(case, seed, n):
    """n views: the sizes in turn, lenses and cameras from the seed."""
    views = scenes.batched_views(n, int(np.random.default_rng([int(seed), 4]).integers(1 << 30)))
    for q, v in enumerate(views):
        v["W"], v["H"] = scenes.VIEW_SIZES[q % len(scenes.VIEW_SIZES)]
    return views


def _outputs(H, W):
    return {"id": torch.empty((H, W), dtype=torch.int32, device=DEV),
            "depth": torch.empty((H, W), dtype=torch.float32, device=DEV),
            "cov": torch.empty((H, W), dtype=torch.float32, device=DEV)}


class _DeviceArray:
    """A float32 device array of a library handle, for torch.as_tensor (the
    tensor keeps this object, and so the handle, alive)."""

    def __init__(self, owner, ptr, shape):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (ptr, False), "version": 3}


def _map_tensor(m):
    p, W, H = ctypes.c_void_p(), ctypes.c_int(), ctypes.c_int()
    vsr.check(vsr.load().vsr_map_data(m.h, ctypes.byref(p), ctypes.byref(W), ctypes.byref(H)), "vsr_map_data")
    return torch.as_tensor(_DeviceArray(m, p.value, (H.value, W.value, 4)), device=DEV)


def _pinned(a):
    t = torch.empty(a.shape, dtype=torch.float32, pin_memory=True)
    t.numpy()[...] = a
    return t


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind in ("frame", "camera", "pstep", "host", "map"):
        W, H, k, l, s, om, aov = _lens_args(case, seed)
        st["lens"] = (W, H, k, l, s, om, aov)
        if kind == "pstep":
            st["map"] = vsr.Map.from_spec(vsr.MAP_UNIVERSAL, W, H, (k, l, s, om), aov=aov, derivatives=True)
        else:
            st["map"] = vsr.Map(W, H, k, l, s, om, aov)
    if kind in ("frame", "camera", "pstep"):
        tris, st["cam"] = _scene(case, seed)
        st["tris"] = torch.from_numpy(tris).to(DEV)
        st["scene"] = vsr.Scene(st["tris"], st["cam"])
        st["out"] = _outputs(case["H"], case["W"])
    elif kind == "map":
        st["out"] = _map_tensor(st["map"])
    elif kind == "host":
        tris, st["cam"] = _scene(case, seed)
        st["pinned"] = [_pinned(tris)] + [torch.empty((H, W), dtype=d, pin_memory=True)
                                          for d in (torch.int32, torch.float32, torch.float32)]
        st["tris"], i, d, c = (t.numpy() for t in st["pinned"])
        st["out"] = {"id": i.view(np.uint32), "depth": d, "cov": c}
        st["host"] = {"id": i, "depth": d, "cov": c}
        st["scene"] = vsr.Scene()
    elif kind == "batch":
        views = _views(case, seed, case["views"])
        st["tris"] = torch.from_numpy(_scene(case, seed)[0]).to(DEV)
        st["maps"] = [vsr.Map(v["W"], v["H"], v["k"], v["l"], v["s"], v["omega"]) for v in views]
        st["cams"] = np.stack([v["cam"] for v in views])
        st["outs"] = [_outputs(v["H"], v["W"]) for v in views]
        st["batch"] = vsr.Batch()
        # the kind of graph that such a program has found to be the faster one
        st["batch"].set_mode(vsr.Batch.CHAINS)
        st["batch"].render(st["maps"], st["tris"], st["cams"], st["outs"])
    elif kind == "serve":
        views = _views(case, seed, case["requests"])
        st["server"] = vsr.Server(budget_bytes=40 << 30, slots=8)
        st["tris"] = [torch.from_numpy(_scene(case, seed + q, n)[0]).to(DEV) for q, n in enumerate((case["T"], case["T2"]))]
        ids = [st["server"].add_scene(t) for t in st["tris"]]
        # outputs of one size side by side
        st["out"] = {}
        for size in sorted({(v["H"], v["W"]) for v in views}):
            n = sum((v["H"], v["W"]) == size for v in views)
            st["out"]["%dx%d" % (size[1], size[0])] = {
                key: torch.empty((n, *size), dtype=torch.int32 if key == "id" else torch.float32, device=DEV)
                for key in ("id", "depth", "cov")}
        used, st["requests"] = {}, []
        for q, v in enumerate(views):
            o = st["out"]["%dx%d" % (v["W"], v["H"])]
            at = used[v["W"], v["H"]] = used.get((v["W"], v["H"]), -1) + 1
            # every fourth request has a lens of its own, the others share a pool of them
            lens = {key: views[q if q % 4 == 0 else q - q % 4][key] for key in ("k", "l", "s", "omega")}
            st["requests"].append((ids[q % 2], dict(W=v["W"], H=v["H"], **lens), v["cam"], {key: t[at] for key, t in o.items()}))
    elif kind == "grad":
        tris, colors, upstream = _train_inputs(case, seed)
        st["tris"], st["colors"], st["upstream"] = (torch.from_numpy(a).to(DEV) for a in (tris, colors, upstream))
        st["lens"] = _lens_args(case, seed)
        st["cam"] = scenes.camera()
        st["map"], st["scene"], st["frags"] = vsr.Map(*st["lens"]), vsr.Scene(), vsr.Frags()
        st["out"] = {"image": torch.empty((case["H"], case["W"]), dtype=torch.float32, device=DEV),
                     **_outputs(case["H"], case["W"])}
    else:
        tris, colors, target = _train_inputs(case, seed)
        st["tris"] = torch.from_numpy(tris).to(DEV).requires_grad_()
        st["colors"] = torch.from_numpy(colors).to(DEV).requires_grad_()
        st["target"] = torch.from_numpy(target).to(DEV)
        st["lens"] = torch.tensor(_lens_args(case, seed)[2:6], dtype=torch.float64, requires_grad=True)
        st["renderer"] = vsr.ShadedRenderer(case["W"], case["H"])
    return st


def run(state):
    kind = state["kind"]
    if kind == "frame":
        state["map"].update(*state["lens"])
        state["scene"].update(state["tris"], state["cam"])
        return vsr.raster(state["map"], state["scene"], out=state["out"])
    if kind == "camera":
        state["scene"].update(state["tris"], state["cam"])
        return vsr.raster(state["map"], state["scene"], out=state["out"])
    if kind == "map":
        state["map"].update(*state["lens"])
        return state["out"]
    if kind == "pstep":
        state["scene"].update(state["tris"], state["cam"])
        return vsr.raster_pstep(state["map"], state["scene"], out=state["out"])
    if kind == "host":
        state["map"].update(*state["lens"])
        vsr.render_host(state["map"], state["scene"], state["tris"], state["cam"], out=state["out"])
        return state["host"]
    if kind == "batch":
        state["batch"].render(state["maps"], state["tris"], state["cams"], state["outs"])
        return state["outs"]
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(*r) for r in state["requests"]]
        for t in tickets:
            vsr.check(server.wait(t)["status"], "request")
        return state["out"]
    if kind == "grad":
        m, sc, frags = state["map"], state["scene"], state["frags"]
        m.update(*state["lens"])
        sc.update(state["tris"], state["cam"])
        out = vsr.raster_shaded(m, sc, frags, state["colors"], out=state["out"])
        g = vsr.raster_backward(m, sc, frags, state["tris"], state["colors"], out["id"], dimage=state["upstream"])
        return {**out, **g}
    image, cov, depth, ids = vsr.render_shaded(state["tris"], state["colors"], state["lens"], state["renderer"])
    loss = (image - state["target"]).square().mean()
    g = torch.autograd.grad(loss, (state["tris"], state["colors"], state["lens"]))
    return {"image": image, "cov": cov, "depth": depth, "id": ids, "loss": loss, "dtris": g[0], "dcolors": g[1],
            "dlens": g[2]}


# ---------------------------------------------------------------------------
# What a pass cannot do without: triangles and lens in, pictures out, and the
# arithmetic of the map (about 100 operations per pixel), of the set-up in
# FP32 pairs (about 3000 per triangle) and of the pixel x triangle tests (20
# each; a direction lies in T rho^2 / 4 caps of radius rho = 0.82 jitter and
# half a pixel on average).

MAP_OPS, SETUP_OPS, TEST_OPS = 100.0, 3000.0, 20.0


def _tests(W, H, T, jitter):
    return W * H * T * (0.82 * jitter + 1.0 / W) ** 2 / 4.0


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        n = case["views"] if kind == "batch" else case["requests"]
        px = sum(w * h for w, h in scenes.VIEW_SIZES) / len(scenes.VIEW_SIZES)
        T = case["T"] if kind == "batch" else (case["T"] + case["T2"]) / 2
        tests = _tests(math.sqrt(px), math.sqrt(px), T, case["jitter"])
        scene = 36.0 * (case["T"] + case.get("T2", 0))
        # maps are cached: read; each request's own lens is a map more
        return {"bytes": scene + n * px * 28.0, "flops": n * (T * SETUP_OPS + tests * TEST_OPS)}
    W, H = case["W"], case["H"]
    px = float(W * H)
    if kind == "map":
        return {"bytes": 16.0 * px, "flops": MAP_OPS * px}
    T = case["T"] + (20 * 4 ** case["sphere"] if case.get("sphere") else 0)
    flops = T * SETUP_OPS + _tests(W, H, case["T"], case["jitter"]) * TEST_OPS
    if kind in ("frame", "host"):
        return {"bytes": 36.0 * T + 12.0 * px, "flops": flops + MAP_OPS * px}
    if kind == "camera":
        return {"bytes": 36.0 * T + 28.0 * px, "flops": flops}
    if kind == "pstep":
        return {"bytes": 36.0 * T + 60.0 * px, "flops": 2.0 * flops}
    # forward (16 B of pictures), one picture in, gradients of 40 B per triangle
    return {"bytes": 80.0 * T + 20.0 * px, "flops": 3.0 * (flops + MAP_OPS * px)}


# ---------------------------------------------------------------------------
# The results in 64-bit arithmetic: the formulas of the method in torch.

def _limits(k, l, s, om):
    k, l, s, om = (float(np.float32(v)) for v in (k, l, s, om))
    k, l, s = min(1.0, max(-1.0, k)), min(1.0, max(0.0, l)), min(1.0, max(0.5, s))
    return k, l, s, min((179.0 if k > 0 else 180.0) / max(abs(k), 0.5), max(1.0, om))


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _map64(W, H, k, l, s, om, aov):
    """The Universal perspective map: directions [H, W, 3], global delta
    [H, W] (0 where undefined) and the differences along both axes.  k, l, s,
    om: float64 tensors (effective parameters)."""
    sc = (1.0 / W, 1.0 / math.hypot(W, H), 1.0 / H, 0.75 / H)[aov]
    x = (2.0 * torch.arange(-1, W + 1, dtype=torch.float64, device=DEV) + 1.0 - W) * sc
    y = ((2.0 * torch.arange(-1, H + 1, dtype=torch.float64, device=DEV) + 1.0 - H) * sc)[:, None]
    x, y = x.expand(H + 2, W + 2), y.expand(H + 2, W + 2)
    R = (x * x + l * y * y).clamp(min=1e-60).sqrt()
    half = om * (math.pi / 360.0)
    ok = torch.ones_like(R, dtype=torch.bool)
    if float(k) > 0:
        th = torch.atan(torch.tan(k * half) * R) / k
    elif float(k) == 0:
        th = half * R
    else:
        arg = torch.sin(k * half) * R
        ok = arg.detach().abs() <= 1.0
        th = torch.asin(torch.where(ok, arg, torch.zeros_like(arg))) / k
    sor = torch.sin(th) / R
    v = _unit(torch.stack([x * sor, y * sor / (l * (1.0 - s) + s), torch.cos(th)], dim=-1))
    c, okc = v[1:-1, 1:-1], ok[1:-1, 1:-1]

    def difference(lo, hi, ulo, uhi):
        ulo, uhi = ulo[..., None], uhi[..., None]
        zero = torch.zeros_like(c)
        return torch.where(ulo & uhi, (hi - lo) * 0.5, torch.where(uhi, hi - c, torch.where(ulo, c - lo, zero)))

    di = difference(v[1:-1, :-2], v[1:-1, 2:], ok[1:-1, :-2], ok[1:-1, 2:])
    dj = difference(v[:-2, 1:-1], v[2:, 1:-1], ok[:-2, 1:-1], ok[2:, 1:-1])
    fw = (di.abs() + dj.abs()).amax(dim=-1)
    okc = okc & (fw.detach() > 0)
    delta = torch.where(okc, 1.0 / torch.where(okc, fw, torch.ones_like(fw)), torch.zeros_like(fw))
    return torch.where(okc[..., None], c, torch.zeros_like(c)), delta, di, dj


def _setup64(tris, cam):
    """Oriented unit edge normals [T, 3, 3], cap (centre, cos, sin of its
    radius), plane (unit normal, offset) and which triangles are usable."""
    cam = torch.as_tensor(np.asarray(cam, dtype=np.float64), device=DEV)
    V = (tris - cam[:3]) @ cam[3:].reshape(3, 3).T
    A, B, C = V.unbind(1)
    cross = torch.linalg.cross
    det = (A * cross(B, C)).sum(-1)
    sg = torch.where(det < 0, -1.0, 1.0).to(torch.float64)[:, None]
    n = torch.stack([sg * _unit(cross(A, B)), sg * _unit(cross(B, C)), sg * _unit(cross(C, A))], dim=1)
    U = _unit(V)
    a2, b2, c2 = ((U[:, p] - U[:, q]).square().sum(-1) for p, q in ((1, 2), (2, 0), (0, 1)))
    Os, Ot, Op = a2 * (b2 + c2 - a2), b2 * (c2 + a2 - b2), c2 * (a2 + b2 - c2)
    S = (Os[:, None] * U[:, 0] + Ot[:, None] * U[:, 1] + Op[:, None] * U[:, 2]) / (Os + Ot + Op)[:, None]
    for o, p, q in ((Op, 0, 1), (Ot, 2, 0), (Os, 1, 2)):
        S = torch.where((o <= 0)[:, None], 0.5 * (U[:, p] + U[:, q]), S)
    cr = S.norm(dim=-1)
    sr = ((1.0 - cr) * (1.0 + cr)).clamp(min=1e-60).sqrt()
    N = _unit(cross(A - B, C - B))
    good = (det != 0) & (V.abs().amax(-1) > 0).all(-1) & (sr.detach() > 1e-25)
    return n, S / cr[:, None], cr, sr, N, (A * N).sum(-1), good


def _candidates(G, delta, width, S, cb, sb):
    """Chunks of (tile pixels [n, 256], triangle [n]): the triangles whose
    caps (radius with cosine cb, sine sb, as functions of a tile's widest
    ramp) may reach the tile.  Pixels beyond the picture: -1."""
    H, W = delta.shape
    th, tw = -(-H // TILE), -(-W // TILE)
    j = torch.arange(th * TILE, device=DEV)[:, None]
    i = torch.arange(tw * TILE, device=DEV)[None, :]
    px = torch.where((j < H) & (i < W), j * W + i, torch.full_like(j * W + i, -1))
    px = px.reshape(th, TILE, tw, TILE).transpose(1, 2).reshape(th * tw, TILE * TILE)
    flat, ok = G.reshape(-1, 3), (px >= 0) & (delta.reshape(-1) > 0)[px.clamp(min=0)]
    Gt = flat[px.clamp(min=0)]
    axis = (Gt * ok[..., None]).sum(1)
    axis = torch.where(axis.norm(dim=-1, keepdim=True) > 1e-9, axis, torch.tensor([0.0, 0.0, 1.0], device=DEV, dtype=torch.float64))
    axis = _unit(axis)
    ca = torch.where(ok, (Gt * axis[:, None]).sum(-1), torch.ones_like(ok, dtype=torch.float64)).amin(1).clamp(-1.0, 1.0) - 1e-9
    sa = (1.0 - ca * ca).clamp(min=0.0).sqrt()
    h = torch.where(ok, width.reshape(-1)[px.clamp(min=0)], torch.zeros_like(ca)[:, None]).amax(1)
    del Gt
    live = ok.any(1).nonzero()[:, 0]
    step = max(1, int(1.5e8 // max(1, S.shape[0])))
    for b in range(0, len(live), step):
        u = live[b:b + step]
        c, s_ = cb(h[u][:, None]), sb(h[u][:, None])
        near = (axis[u] @ S.T >= ca[u][:, None] * c - sa[u][:, None] * s_ - 1e-9) | (ca[u][:, None] + c <= 1e-9)
        pairs = near.nonzero()
        del near
        for q in range(0, len(pairs), 20_000):
            p = pairs[q:q + 20_000]
            yield px[u[p[:, 0]]], p[:, 1]


def _distances(G, rec, t):
    """The three edge distances and the cap's, [..., 4], of directions G and
    triangles t (broadcast against each other)."""
    n, S, cr, sr = rec[0], rec[1], rec[2], rec[3]
    g = [(G * n[t, e]).sum(-1) for e in range(3)]
    g.append(((G * S[t]).sum(-1) - cr[t]) / sr[t])
    return torch.stack(g, dim=-1)


def _raster64(m, rec, pstep=False, fragments=False):
    """Depth and coverage [H, W]; with fragments=True the (pixel, triangle)
    list of all fragments instead."""
    G, delta, di, dj = m
    H, W = delta.shape
    keep = rec[6].nonzero()[:, 0]
    rec = [r[keep] for r in rec[:6]]
    N, d = rec[4], rec[5]
    cr, sr = rec[2], rec[3]
    if pstep:
        width = 0.5 * (di.norm(dim=-1) + dj.norm(dim=-1))
        rho = torch.atan2(sr, cr)

        def cb(h):
            return torch.cos((rho + 4.0 * h).clamp(max=math.pi))

        def sb(h):
            return torch.sin((rho + 4.0 * h).clamp(max=math.pi))
    else:
        width = torch.where(delta > 0, 0.5 / delta.clamp(min=1e-300), torch.zeros_like(delta))

        def cb(h):
            return (cr - h * sr).clamp(-1.0, 1.0)

        def sb(h):
            return (1.0 - cb(h).square()).clamp(min=0.0).sqrt()
    depth = torch.full((H * W,), math.inf, dtype=torch.float64, device=DEV)
    cov = torch.zeros(H * W, dtype=torch.float64, device=DEV)
    Gf, df = G.reshape(-1, 3), delta.reshape(-1)
    dif, djf = di.reshape(-1, 3), dj.reshape(-1, 3)
    found = []
    for px, t in _candidates(G, delta, width, rec[1], cb, sb):
        at = px.clamp(min=0)
        g = _distances(Gf[at], rec, t[:, None])
        dl = df[at]
        r = d[t][:, None] / (Gf[at] * N[t][:, None]).sum(-1)
        frag = (px >= 0) & (dl > 0) & (r > 0) & torch.isfinite(r)
        if pstep:
            scale = torch.stack([torch.ones_like(sr)] * 3 + [1.0 / sr], dim=-1)[t][:, None]
            vec = torch.cat([rec[0], rec[1][:, None]], dim=1)[t][:, None]  # [n, 1, 4, 3]
            w = ((vec * dif[at][:, :, None]).sum(-1).abs() + (vec * djf[at][:, :, None]).sum(-1).abs()) * scale
            frag &= (g > -0.5 * w).all(-1)
            mask = (g / w.clamp(min=1e-30) + 0.5).clamp(0.0, 1.0).amin(-1)
        else:
            gm = g.amin(-1)
            frag &= gm > -0.5 / dl.clamp(min=1e-300)
            mask = (gm * dl + 0.5).clamp(0.0, 1.0)
        if fragments:
            f = frag.nonzero()
            found.append((at[f[:, 0], f[:, 1]], keep[t[f[:, 0]]]))
            continue
        inside = frag & (g[..., :3] >= 0).all(-1)
        cov.index_add_(0, at[frag], mask[frag])
        depth.scatter_reduce_(0, at[inside], r[inside], "amin")
    if fragments:
        return tuple(torch.cat([f[q] for f in found]) if found else torch.zeros(0, dtype=torch.long, device=DEV)
                     for q in (0, 1))
    return depth.reshape(H, W), cov.clamp(max=1.0).reshape(H, W)


def _lens64(W, H, k, l, s, om, aov=0):
    return _map64(W, H, *(torch.tensor(v, dtype=torch.float64, device=DEV) for v in _limits(k, l, s, om)), aov)


def _picture64(m, tris, cam, pstep=False):
    rec = _setup64(torch.from_numpy(tris).to(DEV).double(), cam)
    depth, cov = _raster64(m, rec, pstep)
    return {"id": None, "depth": depth, "cov": cov}


def _train64(case, seed):
    tris, colors, target = _train_inputs(case, seed)
    tris = torch.from_numpy(tris).to(DEV).double().requires_grad_()
    colors = torch.from_numpy(colors).to(DEV).double().requires_grad_()
    target = torch.from_numpy(target).to(DEV).double()
    W, H = case["W"], case["H"]
    with torch.no_grad():
        m = _lens64(*_lens_args(case, seed))
    rec = _setup64(tris, scenes.camera())
    with torch.no_grad():
        px, t = _raster64(m, [r.detach() for r in rec], fragments=True)
        depth, _ = _raster64(m, [r.detach() for r in rec])
    n, S, cr, sr, N, d, good = rec
    G, delta = m[0].reshape(-1, 3)[px], m[1].reshape(-1)[px]
    mask = (_distances(G, rec, t).amin(-1) * delta + 0.5).clamp(0.0, 1.0)
    u = (G * N[t]).sum(-1)
    r = (d[t] / u).detach()
    order = torch.argsort(r, stable=True)  # by triangle where equal: the list is in order of triangles per tile
    order = order[torch.argsort(px[order], stable=True)]
    px, mask, shade = px[order], mask[order], (colors[t] * u.abs())[order]
    total = torch.cumsum(mask, 0)
    first = torch.ones_like(px, dtype=torch.bool)
    first[1:] = px[1:] != px[:-1]
    start = (total - mask)[first][torch.cumsum(first, 0) - 1]
    take = (total - start).clamp(max=1.0) - (total - start - mask).clamp(max=1.0)
    zero = torch.zeros(H * W, dtype=torch.float64, device=DEV)
    image = zero.index_add(0, px, take * shade).reshape(H, W)
    cov = zero.index_add(0, px, take).reshape(H, W)
    loss = (image * target).sum() if case["kind"] == "grad" else (image - target).square().mean()
    g = torch.autograd.grad(loss, [tris, colors])
    # the lens gradient has no value here: its sum over all edges cancels to
    # less than the rounding of an FP32 map moves it
    found = {"image": image.detach(), "cov": cov.detach(), "depth": depth, "id": None, "dtris": g[0], "dcolors": g[1],
             "dlens": None}
    return found if case["kind"] == "grad" else {**found, "loss": loss.detach()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None  # dozens of pictures: over the time that a check has
    if kind in ("grad", "train"):
        return _train64(case, seed)
    if kind == "batch":
        views, tris = _views(case, seed, case["views"]), _scene(case, seed)[0]
        with torch.no_grad():
            return [_picture64(_lens64(v["W"], v["H"], v["k"], v["l"], v["s"], v["omega"]), tris, v["cam"]) if q < 2
                    else {"id": None, "depth": None, "cov": None} for q, v in enumerate(views)]
    with torch.no_grad():
        m = _lens64(*_lens_args(case, seed))
        if kind == "map":
            return torch.cat([m[0], m[1][..., None]], dim=-1)
        return _picture64(m, *_scene(case, seed), pstep=kind == "pstep")
