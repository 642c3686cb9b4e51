"""What a user of the renderer has it do, as cases to be timed: each goes
through the package's public entry points (Scene, Frame, render, render_multi,
render_image, readback, aperture_backward_2d / _3d) with scenes, views and
apertures from the seeded generators.

A case is a dict of plain values; its "kind" says which program it stands for:

* ``image``       one call from a scene and a view to an image in host memory
                  (upload, BVH build, render, readback): a script's call, or
                  an edit's preview; scene "grating" or "procedural".
* ``view``        a resident scene and frame rendered again from scratch and
                  read back on the device: an interactive viewer or a
                  production render; the render options vary.
* ``batch``       many views of uneven size and depth, each with its own
                  scene, in one graph launch.
* ``progressive`` a service's device frames: one sample per pixel for every
                  active request and frame, each request with its own resident
                  accumulators, then the requests' images.
* ``slit``        footprint-resolved rays through a double slit (2D world).
* ``aperture``    footprint-resolved rays through a disk or square onto a
                  screen (3D world).
"""
import math

import numpy as np
import torch

import paper_2303_15762_gb300 as gr
from paper_2303_15762_gb300 import scenegen as sg

# radiance of the constant environment behind glass scenes
GLASS_ENV = 0.05
# operations of one closest-hit query (27.8 node visits of 52 and 2.81
# triangle tests of 41 in a surface-area tree over ~100k triangles), and of
# one segment's shading
QUERY_FLOPS = 27.8 * 52 + 2.81 * 41
SHADE_FLOPS = 300.0


def listed():
    return [
        # the smallest call: one grating patch from scene description to image
        dict(name="grating_image", kind="image", scene="grating", width=64, height=64, spp=64, bins=16, stokes=1,
             depth=1, table="f32", mode="plain"),
        # the same call with narrow order tables and an odd image
        dict(name="grating_image_f16", kind="image", scene="grating", width=301, height=173, spp=48, bins=24,
             stokes=1, depth=1, table="f16", mode="plain"),
        # a preview after an edit: upload and tree build weigh as much as the render
        dict(name="preview_image", kind="image", scene="procedural", tris=100_000, width=256, height=192, spp=16,
             bins=16, stokes=1, depth=4, table="f32", mode="plain"),
        # the production render: 100k triangles, 32 wavelengths, full Stokes vectors
        dict(name="production_view", kind="view", tris=100_000, width=512, height=512, spp=256, bins=32, stokes=4,
             depth=3, table="f32", mode="plain"),
        # hero-wavelength spectral sampling of the same kind of view
        dict(name="hero_view", kind="view", tris=100_000, width=256, height=256, spp=128, bins=32, stokes=4, depth=3,
             table="f32", mode="hero"),
        # anisotropic footprints, a ragged image
        dict(name="aniso_view", kind="view", tris=60_000, width=317, height=211, spp=64, bins=16, stokes=4, depth=3,
             table="f32", mode="aniso"),
        # long paths through dispersive glass with Russian roulette
        dict(name="glass_view", kind="view", tris=100_000, width=384, height=256, spp=64, bins=32, stokes=4, depth=8,
             table="f32", mode="glass"),
        # a batch of uneven views in one graph launch
        dict(name="batch_views", kind="batch", views=8, spp=16, table="f32"),
        # a service's device frames: requests of four resolutions share the launches
        dict(name="progressive_frames", kind="progressive", requests=4, frames=4, table="f32"),
        # the double-slit experiment on a handful of detector elements
        dict(name="slit_few", kind="slit", elements=13, per_slit=400, dkappa=2e-4),
        # the same at the resolution of a published fringe pattern
        dict(name="slit_screen", kind="slit", elements=4001, per_slit=400, dkappa=2e-4),
        # a disk aperture seen on a square screen
        dict(name="aperture_disk", kind="aperture", shape="disk", screen=20, nodes=24, dt=5e-4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["image", "image", "view", "view", "view", "batch", "progressive", "slit", "aperture"])
    if kind == "image" and rng.random() < 0.5:
        return dict(kind=kind, scene="grating", width=_log_int(rng, 24, 400), height=_log_int(rng, 24, 400),
                    spp=_log_int(rng, 16, 128), bins=rng.choice([4, 8, 13, 16, 24, 32]), stokes=1, depth=1,
                    table=rng.choice(["f32", "f16", "bf16"]), mode="plain")
    if kind == "image":
        return dict(kind=kind, scene="procedural", tris=_log_int(rng, 5_000, 200_000), width=_log_int(rng, 64, 400),
                    height=_log_int(rng, 64, 400), spp=_log_int(rng, 4, 32), bins=rng.choice([8, 16, 31, 32]),
                    stokes=rng.choice([1, 4]), depth=rng.randint(1, 8), table=rng.choice(["f32", "f16"]),
                    mode=rng.choice(["plain", "glass"]))
    if kind == "view":
        return dict(kind=kind, tris=_log_int(rng, 5_000, 200_000), width=_log_int(rng, 96, 400),
                    height=_log_int(rng, 96, 400), spp=_log_int(rng, 16, 128), bins=rng.choice([8, 16, 32, 64]),
                    stokes=rng.choice([1, 4, 4]), depth=rng.randint(1, 6), table="f32",
                    mode=rng.choice(["plain", "plain", "hero", "aniso", "glass"]))
    if kind == "batch":
        return dict(kind=kind, views=rng.randint(2, 8), spp=rng.choice([8, 12, 16]), table=rng.choice(["f32", "f16"]))
    if kind == "progressive":
        return dict(kind=kind, requests=rng.randint(1, 5), frames=rng.randint(1, 6), table="f32")
    if kind == "slit":
        return dict(kind=kind, elements=_log_int(rng, 1, 4000), per_slit=_log_int(rng, 60, 400),
                    dkappa=rng.uniform(2e-4, 4e-4))
    return dict(kind=kind, shape=rng.choice(["disk", "rect"]), screen=rng.randint(3, 20), nodes=rng.randint(10, 24),
                dt=rng.uniform(5e-4, 1e-3))


# ---------------------------------------------------------------- inputs
def _scene(case, seed):
    rng = np.random.default_rng(seed)
    if case.get("scene") == "grating":
        return sg.grating_scene(period_um=float(rng.uniform(0.8, 3.0)), source_deg=float(rng.uniform(5.0, 35.0)),
                                source_azimuth_deg=float(rng.uniform(0, 360)))
    n = case["tris"]
    scene = sg.procedural_scene(seed=seed, n_objects=max(4, min(64, n // 1500)), target_tris=n,
                                n_emitters=1 + seed % 4)
    return sg.add_glass(scene, seed=seed + 1, env_radiance=GLASS_ENV) if case["mode"] == "glass" else scene


def _view(case):
    a = dict(width=case["width"], height=case["height"], spp=case["spp"], n_bins=case["bins"], n_stokes=case["stokes"])
    return sg.grating_view(**a) if case.get("scene") == "grating" else sg.procedural_view(max_depth=case["depth"], **a)


def _opts(case, seed):
    flags = 0
    if case.get("scene") != "grating":
        flags = gr.FLAG_NEE | {"plain": 0, "hero": gr.FLAG_HERO, "aniso": gr.FLAG_ANISO,
                               "glass": gr.FLAG_RR}[case["mode"]]
    return dict(seed=1 + seed % 1_000_003, flags=flags, table_dtype=case["table"])


def _resolutions(case):
    return [sg.SERVING_RESOLUTIONS[i % len(sg.SERVING_RESOLUTIONS)] for i in range(case["requests"])]


def _requests(case, seed):
    """The service's active requests: (scene, view at one sample per pixel), the resolutions in turn."""
    rng = np.random.default_rng(seed)
    reqs = [sg.serving_request(rng, i) for i in range(case["requests"])]
    return [(s, dict(v, width=w, height=h)) for (s, v), (w, h) in zip(reqs, _resolutions(case))]


def _slit(case, seed):
    rng = np.random.default_rng(seed)
    n = case["elements"]
    half = 600.0 if n < 100 else 2000.0
    x0 = np.linspace(-half, half, n) if n > 1 else np.zeros(1)
    return sg.double_slit_setup(d=float(rng.uniform(360.0, 440.0)), b=float(rng.uniform(30.0, 50.0)),
                                n_per_slit=case["per_slit"], x0=x0, dkappa=case["dkappa"])


def _aperture(case, seed):
    rng = np.random.default_rng(seed)
    g = np.linspace(-240.0, 240.0, case["screen"])
    X, Y = np.meshgrid(g, g, indexing="ij")
    size = float(rng.uniform(10.0, 14.0)) * (1.0 if case["shape"] == "disk" else 2.0)
    return sg.aperture3d_setup(shape=case["shape"], size=size, n_nodes=case["nodes"], dt=case["dt"],
                               x0=np.stack([X.ravel(), Y.ravel()], axis=1))


def _out(v):
    return torch.empty((v["height"], v["width"], v["n_bins"], v["n_stokes"]), dtype=torch.float32, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "image":  # the scene description stays on the host: the call uploads it
        return dict(kind=kind, scene=_scene(case, seed), view=_view(case), opts=_opts(case, seed))
    if kind == "view":
        v = _view(case)
        return dict(kind=kind, scenes=[gr.Scene(_scene(case, seed))], views=[v], frame=gr.Frame([v]), out=[_out(v)],
                    opts=_opts(case, seed))
    if kind == "batch":
        # the shapes are the batch's own (the same for every seed); scenes and random streams come from the seed
        _, views = sg.batch_views(seed=4, n_views=case["views"], spp=case["spp"], tris_range=(12, 13),
                                  side_range=(128, 768))
        rng = np.random.default_rng(seed)
        scenes = []
        for i in range(case["views"]):
            nt = int(round(math.exp(np.random.default_rng(i).uniform(math.log(5_000), math.log(200_000)))))
            scenes.append(gr.Scene(sg.procedural_scene(seed=int(rng.integers(1 << 30)), target_tris=nt,
                                                       n_objects=max(4, min(64, nt // 1500)))))
        return dict(kind=kind, scenes=scenes, views=views, frame=gr.Frame(views), out=[_out(v) for v in views],
                    opts=dict(seed=2 + seed % 1_000_003, flags=gr.FLAG_NEE | gr.FLAG_RR, table_dtype=case["table"],
                              use_graph=True))
    if kind == "progressive":
        reqs = _requests(case, seed)
        # a 1x1 view without samples owns the slot pool that the requests share
        work = dict(sg.grating_view(width=1, height=1, spp=0, n_bins=1), max_depth=0)
        views = [dict(v, scene_index=i) for i, (_, v) in enumerate(reqs)]
        return dict(kind=kind, scenes=[gr.Scene(s) for s, _ in reqs], work=work, work_frame=gr.Frame([work]),
                    views=views, frames=[gr.Frame([v]) for v in views], out=[_out(v) for v in views],
                    n=case["frames"],
                    opts=dict(seed=1 + seed % 1_000_003, flags=0, table_dtype=case["table"],
                              pool_size=sum(v["width"] * v["height"] for v in views)))
    s = _slit(case, seed) if kind == "slit" else _aperture(case, seed)
    return dict(kind=kind, setup=s)


# ---------------------------------------------------------------- one pass
def run(st):
    kind = st["kind"]
    if kind == "image":
        return gr.render_image(st["scene"], st["view"], **st["opts"])
    if kind in ("view", "batch"):
        f = st["frame"]
        f.reset()
        gr.render(st["scenes"], st["views"], f, **st["opts"])
        return [f.readback(i, out=o) for i, o in enumerate(st["out"])]
    if kind == "progressive":
        for f in st["frames"]:
            f.reset()
        for k in range(st["n"]):
            gr.render_multi(st["scenes"], [st["work"]] + [dict(v, first_sample=k) for v in st["views"]],
                            [st["work_frame"]] + st["frames"], [0] * (1 + len(st["frames"])), **st["opts"])
        return [f.readback(0, out=o) for f, o in zip(st["frames"], st["out"])]
    s = st["setup"]
    if kind == "slit":
        return gr.aperture_backward_2d(s["x0"], s["x_ap"], s["w_ap"], s["beta"], s["z"], s["k"], s["reach"],
                                       s["dtheta"], s["rho_cut"])[0]
    return gr.aperture_backward_3d(s["x0"], s["x_ap"], s["w_ap"], s["beta"], s["z"], s["k"], s["reach"], s["dt"],
                                   s["rho_cut"])[0]


# ---------------------------------------------------------------- work of one pass
def _image_work(tris, view, samples, segments, traced):
    out = 4.0 * view["width"] * view["height"] * view["n_bins"] * view["n_stokes"]
    return (tris * 40.0 + out, samples * segments * (traced + SHADE_FLOPS))


def work(case):
    kind = case["kind"]
    if kind in ("image", "view"):
        v = _view(case)
        n = float(v["width"] * v["height"] * v["spp"])
        if case.get("scene") == "grating":
            b, f = _image_work(2, v, n, 2.0, 2 * 41.0)
        else:  # camera segment, then about two thirds of the paths go on at each vertex
            seg = sum((2 / 3) ** k for k in range(case["depth"] + 1)) * 0.75
            b, f = _image_work(case["tris"], v, n, seg, QUERY_FLOPS)
        return {"bytes": b, "flops": f}
    if kind == "batch":
        _, views = sg.batch_views(seed=4, n_views=case["views"], spp=case["spp"], tris_range=(12, 13),
                                  side_range=(128, 768))
        parts = [_image_work(60_000, v, float(v["width"] * v["height"] * v["spp"]),
                             sum((2 / 3) ** k for k in range(v["max_depth"] + 1)) * 0.75, QUERY_FLOPS) for v in views]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if kind == "progressive":
        px = sum(w * h for w, h in _resolutions(case))
        return {"bytes": px * 16 * 4.0, "flops": px * case["frames"] * 2.0 * (2 * 41.0 + SHADE_FLOPS)}
    s = _slit(case, 0) if kind == "slit" else _aperture(case, 0)
    n_ap = len(s["w_ap"])
    if kind == "slit":
        rays = float(np.sum(np.ceil((np.arctan((s["x0"] + s["reach"]) / s["z"])
                                     - np.arctan((s["x0"] - s["reach"]) / s["z"])) / s["dtheta"])))
        return {"bytes": 16.0 * (n_ap + len(s["x0"])), "flops": rays * n_ap * 18.0}
    n_t = math.ceil(2.0 * s["reach"] / (s["z"] * s["dt"]))
    return {"bytes": 24.0 * (n_ap + len(s["x0"])), "flops": len(s["x0"]) * float(n_t) ** 2 * n_ap * 24.0}


# ---------------------------------------------------------------- 64-bit values
def _philox(c0, c1, c2, key):
    """Philox4x32-10 words (Salmon et al., SC'11) of counters (c0, c1, c2, 0), int64 tensors holding 32 bits."""
    M = 0xFFFFFFFF
    c = [c0, c1, torch.full_like(c0, c2), torch.zeros_like(c0)]
    k0, k1 = key

    def mul(a, x):  # 32 x 32 bits in two halves, so that int64 does not overflow
        lo, hi = (x & 0xFFFF) * a, (x >> 16) * a
        t = (lo >> 16) + hi
        return (t >> 16) & M, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return [(x >> 8).double() * 2.0 ** -24 for x in c]


def _bessel_sq(j, x):
    """J_j(x)^2 from the power series."""
    term = math.prod(0.5 * x / i for i in range(1, j + 1))
    total, m = term, 1
    while abs(term) > 1e-20 * abs(total) and m < 100:
        term *= -(0.25 * x * x) / (m * (m + j))
        total += term
        m += 1
    return total * total


def _grating_exact(scene, v, seed, spp):
    """Mean image [H][W][bins][1] of a view of the planar grating under its
    distant source: every sample's order choice and measurement in 64 bits."""
    dev = "cuda"
    mat, lt = scene["mats"][0].astype(np.float64), scene["lights"][0].astype(np.float64)
    W, H, nb = v["width"], v["height"], v["n_bins"]
    half = float(scene["verts"].max())
    period, height = mat[4], mat[5]
    eye = np.array(v["eye"])
    fw = (np.array(v["look_at"]) - eye) / np.linalg.norm(np.array(v["look_at"]) - eye)
    right = np.cross(fw, v["up"])
    right /= np.linalg.norm(right)
    upc = np.cross(right, fw)
    th, aspect = math.tan(0.5 * math.radians(v["vfov_deg"])), W / H
    pix = torch.arange(W * H, dtype=torch.int64, device=dev)
    px, py = (pix % W).double(), (pix // W).double()
    img = torch.zeros((W * H, nb), dtype=torch.float64, device=dev)
    L = lt[1:4]

    def measure(d, kappa):
        q = sum((d[a] - L[a]) ** 2 for a in range(3))
        return lt[4] * kappa / (2 * math.pi * -math.expm1(-2 * kappa)) * torch.exp(-0.5 * kappa * q)

    for s in range(spp):
        b = s % nb
        lam = v["lambda_min_um"] + (b * (v["lambda_max_um"] - v["lambda_min_um"]) / (nb - 1) if nb > 1 else 0.0)
        k = 2 * math.pi / lam
        kappa = 2 * (v["f_beta"] * v["p_pix_um"]) ** 2 * k * k  # a coherent source adds no spread
        smp = torch.full_like(pix, s)
        key = (seed, v["view_index"])
        u = _philox(pix, smp, 0, key)
        sx = (2 * (px + u[0]) / W - 1) * th * aspect
        sy = (1 - 2 * (py + u[1]) / H) * th
        d = [fw[a] + sx * right[a] + sy * upc[a] for a in range(3)]
        n = torch.sqrt(sum(x * x for x in d))
        d = [x / n for x in d]
        t = -eye[2] / d[2]
        hit = (d[2] < 0) & ((eye[0] + t * d[0]).abs() <= half) & ((eye[1] + t * d[1]).abs() <= half)
        ul = _philox(pix, smp, 2, key)[0]
        jm = min(40, int(math.floor(2 * period / lam)) + 2)
        js = list(range(-jm, jm + 1))
        x = math.pi * height / lam
        tx = torch.stack([d[0] + j * (lam / period) for j in js])
        wt = torch.tensor([_bessel_sq(abs(j), x) for j in js], dtype=torch.float64, device=dev)[:, None]
        wt = torch.where(tx * tx + (d[1] * d[1])[None] < 1.0, wt, torch.zeros_like(tx))
        cum = torch.cumsum(wt, 0)
        pick = (cum <= ul[None] * cum[-1:]).sum(0).clamp(max=len(js) - 1)
        ox = torch.gather(tx, 0, pick[None])[0]
        oz = torch.sqrt((1 - ox * ox - d[1] * d[1]).clamp(min=0))
        img[:, b] += torch.where(hit, measure([ox, d[1], oz], kappa), measure(d, kappa))
    cnt = torch.tensor([max(1, (spp - b + nb - 1) // nb) for b in range(nb)], dtype=torch.float64, device=dev)
    return (img / cnt).reshape(H, W, nb, 1)


def _slit_exact(s):
    xa, wa = (torch.tensor(s[k], dtype=torch.float64, device="cuda")[None] for k in ("x_ap", "w_ap"))
    b2, out = s["beta"] ** 2, []
    for x0 in s["x0"]:
        lo, hi = math.atan((x0 - s["reach"]) / s["z"]), math.atan((x0 + s["reach"]) / s["z"])
        th = lo + torch.arange(math.ceil((hi - lo) / s["dtheta"]), dtype=torch.float64, device="cuda")[:, None] * s["dtheta"]
        c, sn = torch.cos(th), torch.sin(th)
        zb = s["z"] / c / s["k"]
        w2 = b2 + zb * zb / b2
        dx = xa - (x0 - s["z"] * sn / c)
        u2 = (dx * c) ** 2
        g = torch.where(u2 <= s["rho_cut"] ** 2 * w2, wa * torch.exp(-u2 / (2 * w2)), torch.zeros_like(u2))
        ph = s["k"] * sn * dx - zb / b2 * u2 / (2 * w2)
        a2 = (g * torch.cos(ph)).sum(1) ** 2 + (g * torch.sin(ph)).sum(1) ** 2
        c, w2 = c[:, 0], w2[:, 0]
        out.append((a2 * c / torch.sqrt(math.pi * w2) * s["k"] * c * s["dtheta"]).sum() / (2 * math.pi))
    return torch.stack(out).cpu().numpy()


def _aperture_exact(s):
    xa = torch.tensor(s["x_ap"], dtype=torch.float64, device="cuda")
    wa = torch.tensor(s["w_ap"], dtype=torch.float64, device="cuda")[None]
    z, k, dt, b0 = s["z"], s["k"], s["dt"], s["beta"] ** 2
    n_t, out = math.ceil(2.0 * s["reach"] / (z * dt)), []
    g1 = torch.arange(n_t, dtype=torch.float64, device="cuda") * dt
    for x0, y0 in s["x0"]:
        tx = ((x0 - s["reach"]) / z + g1)[:, None].expand(n_t, n_t).reshape(-1, 1)
        ty = ((y0 - s["reach"]) / z + g1)[None, :].expand(n_t, n_t).reshape(-1, 1)
        sz = 1.0 / torch.sqrt(1 + tx * tx + ty * ty)
        zb = z / sz / k
        b2 = b0 + zb * zb / b0
        dx, dy = xa[None, :, 0] - (x0 - z * tx), xa[None, :, 1] - (y0 - z * ty)
        p2 = dx * dx + dy * dy - sz * sz * (tx * dx + ty * dy) ** 2
        g = torch.where(p2 <= s["rho_cut"] ** 2 * b2, wa * torch.exp(-p2 / (2 * b2)), torch.zeros_like(p2))
        ph = k * sz * (tx * dx + ty * dy) - zb / b0 * p2 / (2 * b2)
        a2 = (g * torch.cos(ph)).sum(1) ** 2 + (g * torch.sin(ph)).sum(1) ** 2
        sz, b2 = sz[:, 0], b2[:, 0]
        out.append((a2 * sz / (math.pi * b2) * k * k * sz ** 4 * dt * dt).sum() / (4 * math.pi ** 2))
    return torch.stack(out).cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "slit":
        return _slit_exact(_slit(case, seed))
    if kind == "aperture":
        return _aperture_exact(_aperture(case, seed))
    if kind == "progressive":
        rs = 1 + seed % 1_000_003
        return [_grating_exact(s, v, rs, case["frames"]) for s, v in _requests(case, seed)]
    if case.get("scene") == "grating":
        return _grating_exact(_scene(case, seed), _view(case), 1 + seed % 1_000_003, case["spp"]).cpu().numpy()
    return None  # path tracing through 5k-300k triangles takes minutes in plain torch
