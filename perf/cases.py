"""The renders that this library is used for, as measurable cases.

Every case is a dict of plain values (``listed`` and ``draw``); ``prepare``
builds what a program has in hand before it renders (fields packed into a
resident volume, cameras, output buffers), ``run`` makes the calls, ``work``
says what such a pass cannot do without, and ``exact`` computes the same images
in float64 with plain torch.

Fields: a blob moving along a steady jet (``field`` "blob"), or a turbulent jet
whose lognormal density and tilted velocities come from Kolmogorov random
fields ("turbulent").  The seed sets the random phases, the blob's path and
the azimuth of the cameras.
"""
from __future__ import annotations

import math
from dataclasses import dataclass

import numpy as np
import torch

from paper_2609_09322_gb300 import Context

DEVICE = "cuda"


# ------------------------------------------------------------------ the cases
_BASE = dict(kind="batch", nx=64, ny=64, nz=64, dx=1.0, dy=1.0, dz=1.0, epochs=1, cdt=4.0, field="turbulent",
             store="f32", layout="", launch="", width=64, height=64, dirs=1, times=1, beaming=True, lookback=True,
             samples=False, channels=0, inputs="f32")


def _case(name=None, n=None, **kw):
    c = dict(_BASE)
    if n is not None:
        c.update(nx=n, ny=n, nz=n)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest render: one 64^2 image of one 32^3 snapshot without light-travel delay, where the call's own
        # latency is all there is (interactive previews, unit-sized scenes)
        _case("tiny_image", n=32, kind="image", width=64, height=64, lookback=False),
        # one large image per call with the default layout and launch: a program that renders frame by frame
        _case("image_f32", n=512, kind="image", epochs=8, cdt=128.0, width=1024, height=1024),
        # the same from half-size records in the layout and launch that the autotuner settled on for it
        _case("image_bf16", n=512, kind="image", epochs=8, cdt=128.0, width=1024, height=1024, store="bf16",
              layout="8,4,1", launch="4,8,4,4,1,0,2"),
        # a light curve: two directions at nine observer times each, everything at its default
        _case("series_f32", n=256, epochs=16, cdt=4.0, field="blob", width=512, height=512, dirs=2, times=9),
        # the same from half-size records, as tuned
        _case("series_bf16", n=256, epochs=16, cdt=4.0, field="blob", width=512, height=512, dirs=2, times=9,
              store="bf16", layout="4,2,1", launch="8,4,8,4,1,0,4"),
        # an orbit around the source: every view another direction, each ray marched whole, default launch
        _case("orbit_f32", n=256, epochs=16, cdt=16.0, width=384, height=384, dirs=24),
        # the largest: 256 orientations of a 384^3 x 32 series, marched region by region as tuned
        _case("sphere_f32", n=384, epochs=32, cdt=24.0, width=256, height=256, dirs=256, launch="4,8,4,2,1,64",
              layout="8,4,0"),
        # the same use from half-size records at a smaller size
        _case("sphere_bf16", n=256, epochs=16, cdt=16.0, width=192, height=192, dirs=96, store="bf16",
              launch="4,8,4,2,1,64", layout="4,4,1"),
        # vector integration: j' and three more channels along every ray
        _case("vector_f32", n=192, epochs=8, cdt=24.0, kind="vector", channels=3, width=384, height=384, dirs=6),
        # a render service: requests of mixed sizes and directions against two resident volumes
        _case("serve_mixed", n=192, epochs=8, cdt=12.0, kind="serve", width=512, height=512, dirs=40),
        # odd and ragged: unequal axes, cells that are not cubes, odd image, no beaming, with sample counts
        _case("ragged_counts", nx=97, ny=131, nz=203, dx=1.25, dy=0.8, dz=1.0, epochs=7, cdt=20.0, width=211,
              height=173, dirs=5, beaming=False, samples=True),
        # a new series arrives: load it (device arrays), look at one image, drop it
        _case("load_f32", n=256, epochs=8, cdt=16.0, kind="load", width=256, height=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["image", "image", "series", "series", "orbit", "sphere", "vector", "serve", "ragged", "load"])
    store = rng.choice(["f32", "f32", "bf16"])
    layout = rng.choice(["", "", "8,4,0", "8,4,1", "4,4,0", "4,2,1"])
    if kind == "image":
        n = [_log_int(rng, 32, 512) for _ in range(3)]
        return _case(nx=n[0], ny=n[1], nz=n[2], kind="image", epochs=rng.randint(1, 12),
                     cdt=max(n) / rng.choice([4.0, 16.0]), width=_log_int(rng, 48, 1024), height=_log_int(rng, 48, 1024),
                     store=store, layout=layout, lookback=rng.random() < 0.8)
    if kind == "series":
        n = _log_int(rng, 64, 256)
        return _case(n=n, epochs=rng.randint(6, 20), cdt=n / 64.0, field="blob", width=_log_int(rng, 64, 512),
                     height=_log_int(rng, 64, 512), dirs=rng.randint(1, 3), times=rng.randint(2, 12), store=store,
                     layout=layout, launch=rng.choice(["", "", "8,4,8,4,1,0,4", "4,8,4,2,1,0,8", "4,8,4,2,1,0,2"]))
    if kind == "orbit":
        n = _log_int(rng, 64, 256)
        return _case(n=n, epochs=rng.randint(1, 16), cdt=n / 16.0, width=_log_int(rng, 48, 384),
                     height=_log_int(rng, 48, 384), dirs=rng.randint(2, 24), store=store, layout=layout,
                     launch=rng.choice(["", "", "4,8,4,2,1,0,1", "16,2,2,1,0,0,1", "8,4,8,4,1,0,1"]))
    if kind == "sphere":
        n = _log_int(rng, 96, 320)
        return _case(n=n, epochs=rng.randint(4, 24), cdt=n / 16.0, width=_log_int(rng, 64, 224),
                     height=_log_int(rng, 64, 224), dirs=rng.randint(16, 160), store=store, layout=layout,
                     launch=rng.choice(["4,8,4,2,1,64", "4,8,4,2,1,64", "4,8,4,2,1,32", "4,8,8,1,1,64"]))
    if kind == "vector":
        n = _log_int(rng, 48, 192)
        return _case(n=n, epochs=rng.randint(2, 10), cdt=n / 8.0, kind="vector", channels=rng.choice([1, 3]),
                     width=_log_int(rng, 48, 384), height=_log_int(rng, 48, 384), dirs=rng.randint(1, 8), store=store,
                     layout=layout)
    if kind == "serve":
        n = _log_int(rng, 48, 192)
        return _case(n=n, epochs=rng.randint(2, 12), cdt=n / 16.0, kind="serve", width=_log_int(rng, 64, 512),
                     height=_log_int(rng, 64, 512), dirs=rng.randint(4, 48))
    if kind == "ragged":
        n = [_log_int(rng, 17, 260) for _ in range(3)]
        return _case(nx=n[0], ny=n[1], nz=n[2], dx=rng.uniform(0.5, 2.0), dy=rng.uniform(0.5, 2.0),
                     dz=rng.uniform(0.5, 2.0), epochs=rng.randint(1, 12), cdt=max(n) / 10.0, width=_log_int(rng, 33, 400),
                     height=_log_int(rng, 33, 400), dirs=rng.randint(1, 8), store=store, layout=layout,
                     beaming=rng.random() < 0.5, lookback=rng.random() < 0.7, samples=rng.random() < 0.5)
    n = _log_int(rng, 64, 288)
    return _case(n=n, epochs=rng.randint(1, 8), cdt=n / 16.0, kind="load", width=_log_int(rng, 64, 512),
                 height=_log_int(rng, 64, 512), store=store, layout=layout, inputs=rng.choice(["f32", "f32", "f64"]))


# ------------------------------------------------------------------ grids, cameras and fields
@dataclass
class Grid:
    n: tuple
    origin: tuple
    dx: tuple
    n_epochs: int
    t0: float
    dt: float


@dataclass
class View:
    dir: tuple
    up: tuple
    center: tuple
    t_obs: float
    c: float
    alpha: float
    nu_ratio: float
    beaming: bool
    lookback: bool
    width: int
    height: int
    fov_u: float
    fov_v: float


def _grid(case):
    return Grid(n=(case["nx"], case["ny"], case["nz"]), origin=(0.0, 0.0, 0.0),
                dx=(case["dx"], case["dy"], case["dz"]), n_epochs=case["epochs"], t0=0.0, dt=case["cdt"])


def _view(case, grid, n_hat, t_obs, width, height):
    ext = [grid.n[i] * grid.dx[i] for i in range(3)]
    fov = math.sqrt(3.0) * max(ext)
    return View(dir=tuple(-float(x) for x in n_hat), up=(0.0, 0.0, 1.0), center=tuple(0.5 * e for e in ext),
                t_obs=float(t_obs), c=1.0, alpha=-0.6, nu_ratio=1.0, beaming=case["beaming"],
                lookback=case["lookback"], width=width, height=height, fov_u=fov, fov_v=fov * height / width)


def _polar(theta_deg, phi_deg):
    th, ph = math.radians(theta_deg), math.radians(phi_deg)
    return (math.sin(th) * math.cos(ph), math.sin(th) * math.sin(ph), math.cos(th))


def _sphere(n, turn):
    """n directions spread evenly over the sphere, turned about z."""
    k = np.arange(n)
    z = 1.0 - (2.0 * k + 1.0) / n
    r = np.sqrt(1.0 - z * z)
    ph = math.pi * (3.0 - math.sqrt(5.0)) * k + turn
    return np.stack([r * np.cos(ph), r * np.sin(ph), z], axis=1)


def _blob_start(case, seed):
    rng = np.random.default_rng([seed, 7])
    n = np.array([case["nx"] * case["dx"], case["ny"] * case["dy"], case["nz"] * case["dz"]])
    return n * np.array([0.5, 0.5, 0.25]) + rng.uniform(-0.02, 0.02, 3) * n


BLOB_BETA = 0.95


def _views(case, seed):
    """The cameras of a case: a time series per direction (blob), single images, or an orbit."""
    grid = _grid(case)
    w, h = case["width"], case["height"]
    rng = np.random.default_rng([seed, 11])
    turn = float(rng.uniform(0.0, 360.0))
    ext = np.array([grid.n[i] * grid.dx[i] for i in range(3)])
    mid = 0.5 * (grid.n_epochs - 1) * grid.dt
    if case["field"] == "blob":
        # observer times at which the blob centre is seen at snapshots from a fifth to four fifths of the series
        start, out = _blob_start(case, seed), []
        lo, hi = 0.2 * (grid.n_epochs - 1), 0.8 * (grid.n_epochs - 1)
        for d in range(case["dirs"]):
            n_hat = _polar(10.0 + 35.0 * d, turn + 50.0 * d)
            for t in range(case["times"]):
                m = lo + (hi - lo) * t / max(case["times"] - 1, 1)
                pos = start + np.array([0.0, 0.0, BLOB_BETA * grid.dt * m])
                depth = -float(np.dot(pos - 0.5 * ext, n_hat))
                out.append(_view(case, grid, n_hat, m * grid.dt + depth, w, h))
        return out
    if case["kind"] == "serve":
        out = []
        for k, n_hat in enumerate(_sphere(case["dirs"], math.radians(turn))):
            s = 2 ** (k % 3)  # full, half and quarter size images
            t = float(rng.uniform(0.0, 2.0 * mid))
            out.append(_view(case, grid, n_hat, t, max(8, w // s), max(8, h // s)))
        return out
    if case["dirs"] == 1:
        return [_view(case, grid, _polar(30.0, turn), mid, w, h)]
    return [_view(case, grid, n_hat, mid, w, h) for n_hat in _sphere(case["dirs"], math.radians(turn))]


def _kolmogorov(shape, gen):
    """A random field of power spectrum k^(-11/3), zero mean and unit rms."""
    nz, ny, nx = shape
    k = torch.sqrt(torch.fft.rfftfreq(nx, device=DEVICE)[None, None, :] ** 2
                   + torch.fft.fftfreq(ny, device=DEVICE)[None, :, None] ** 2
                   + torch.fft.fftfreq(nz, device=DEVICE)[:, None, None] ** 2)
    amp = torch.where(k > 0, k.clamp_min(1e-12) ** (-11.0 / 6.0), torch.zeros_like(k))
    phase = torch.rand(k.shape, generator=gen, device=DEVICE) * (2.0 * math.pi)
    f = torch.fft.irfftn(torch.polar(amp, phase), s=(nz, ny, nx))
    f -= f.mean()
    return f / f.std().clamp_min(1e-20)


def _fields(case, seed):
    """j[M][nz][ny][nx] and beta[M][nz][ny][nx][3], float32 on the device."""
    grid = _grid(case)
    nx, ny, nz = grid.n
    m_all, shape = grid.n_epochs, (nz, ny, nx)
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed) * 1000003 + 17)
    axis = [torch.arange(grid.n[i], device=DEVICE, dtype=torch.float32) * grid.dx[i] + 0.5 * grid.dx[i] for i in range(3)]
    x, y, z = axis[0][None, None, :], axis[1][None, :, None], axis[2][:, None, None]
    ext = [grid.n[i] * grid.dx[i] for i in range(3)]
    r = z - ext[2] / 16.0
    rr = r.clamp_min(1.0)
    rho2 = (x - 0.5 * ext[0]) ** 2 + (y - 0.5 * ext[1]) ** 2
    core = torch.exp(-rho2 / (2.0 * (rr * math.tan(math.radians(5.0))) ** 2))
    jet = torch.where(r >= 0, core / (rr * rr), torch.zeros_like(core))
    j = torch.empty((m_all, *shape), dtype=torch.float32, device=DEVICE)
    beta = torch.zeros((m_all, *shape, 3), dtype=torch.float32, device=DEVICE)
    if case["field"] == "blob":
        start, sigma = _blob_start(case, seed), max(ext) / 32.0
        jet = 0.1 * jet * torch.exp(0.01 * torch.randn(shape, generator=gen, device=DEVICE))
        for m in range(m_all):
            d2 = ((x - float(start[0])) ** 2 + (y - float(start[1])) ** 2
                  + (z - float(start[2] + BLOB_BETA * grid.dt * m)) ** 2)
            j[m] = jet + torch.exp(-d2 / (2.0 * sigma * sigma))
        beta[..., 2] = BLOB_BETA
        return j, beta
    # each random field turns slowly between two draws of it
    pairs = [(_kolmogorov(shape, gen), _kolmogorov(shape, gen)) for _ in range(4)]
    for m in range(m_all):
        a = 0.15 * m
        dens, dmag, tx, ty = (math.cos(a) * p + math.sin(a) * q for p, q in pairs)
        j[m] = jet * torch.exp(0.3 * dens) + 1e-3
        mag = (0.5 + 0.49 * core + 0.05 * dmag).clamp(0.5, 0.99)
        sx, sy = torch.sin(0.1 * tx), torch.sin(0.1 * ty)
        beta[m, ..., 0] = mag * sx
        beta[m, ..., 1] = mag * sy
        beta[m, ..., 2] = mag * torch.sqrt((1.0 - sx * sx - sy * sy).clamp_min(0.0))
    return j, beta


def _channels(case, seed, j):
    """Signed extra emissivities: the field j' times slow waves along the axes."""
    rng = np.random.default_rng([seed, 13])
    out = torch.empty((case["channels"], *j.shape), dtype=torch.float32, device=DEVICE)
    for c in range(case["channels"]):
        n = j.shape[1 + c % 3]
        ph = torch.arange(n, device=DEVICE, dtype=torch.float32) * (2.0 * math.pi * (2 + c) / n) + float(rng.uniform(0, 6.28))
        out[c] = j * torch.sin(ph).reshape([n if 1 + c % 3 == d else 1 for d in range(4)])
    return out


def _layout(case):
    if not case["layout"]:
        return {}
    b, s, p = (int(v) for v in case["layout"].split(","))
    return dict(brick=b, super_brick=s, paired=bool(p))


def _launch(case):
    if not case["launch"]:
        return None
    v = ([int(x) for x in case["launch"].split(",")] + [0, 0])[:7]
    return {"packet": (v[0], v[1]), "cta_warps": v[2], "depth": v[3], "regcap": v[4], "region": v[5], "group": v[6],
            "persistent": 0 if v[5] else 1}


# ------------------------------------------------------------------ one pass
def prepare(case, seed):
    grid, views = _grid(case), _views(case, seed)
    j, beta = _fields(case, seed)
    st = dict(case=case, grid=grid, views=views, launch=_launch(case), ctx=Context(torch.cuda.current_device()))
    ctx = st["ctx"]
    if case["kind"] == "load":
        st["fields"] = (j.double(), beta.double()) if case["inputs"] == "f64" else (j, beta)
        return st
    torch.cuda.synchronize()
    st["vol"] = ctx.load_snapshots(grid, j, beta, store=case["store"], **_layout(case))
    if case["kind"] == "serve":
        # the first volume in float32 records, the second in half-size ones
        st["vol2"] = ctx.load_snapshots(grid, j, beta, store="bf16", paired=True)
        st["out"] = [torch.empty((v.height, v.width), dtype=torch.float32, device=DEVICE) for v in views]
        ctx.serve_start()
    elif case["kind"] == "vector":
        ctx.load_channels(st["vol"], _channels(case, seed, j))
        st["out"] = torch.empty((len(views), 1 + case["channels"], case["height"], case["width"]),
                                dtype=torch.float32, device=DEVICE)
    elif case["kind"] == "batch":
        st["out"] = torch.empty((len(views), case["height"], case["width"]), dtype=torch.float32, device=DEVICE)
    del j, beta
    torch.cuda.empty_cache()
    return st


def run(st):
    case, ctx, views = st["case"], st["ctx"], st["views"]
    if case["kind"] == "image":
        return ctx.render(st["vol"], views[0], launch=st["launch"])
    if case["kind"] == "batch":
        r = ctx.render_batch(st["vol"], views, out=st["out"], samples=case["samples"], launch=st["launch"])
        return list(r) if case["samples"] else r
    if case["kind"] == "vector":
        return ctx.render_vector(st["vol"], views, out=st["out"], launch=st["launch"])
    if case["kind"] == "serve":
        tickets = [ctx.submit(st["vol"] if k % 2 == 0 else st["vol2"], v, st["out"][k]) for k, v in enumerate(views)]
        for t in tickets:
            ctx.wait(t)
        return st["out"]
    vol = ctx.load_snapshots(st["grid"], *st["fields"], store=case["store"], **_layout(case))
    img = ctx.render(vol, views[0], launch=st["launch"])
    ctx.unload(vol)
    return img


# ------------------------------------------------------------------ what a pass cannot do without
def _ray_frame(view, grid, p, q):
    """Positions on the image plane (cells) and the direction (cells per unit length) of rays (p, q), float64."""
    sh = np.asarray(view.dir, dtype=np.float64)
    sh = sh / np.linalg.norm(sh)
    up = np.asarray(view.up, dtype=np.float64)
    ev = up - np.dot(up, sh) * sh
    ev /= np.linalg.norm(ev)
    eu = np.cross(sh, ev)
    a = (p + 0.5 - 0.5 * view.width) * (view.fov_u / view.width)
    b = (q + 0.5 - 0.5 * view.height) * (view.fov_v / view.height)
    g = [(view.center[i] + a * eu[i] + b * ev[i] - grid.origin[i]) / grid.dx[i] for i in range(3)]
    return g, [sh[i] / grid.dx[i] for i in range(3)], sh


def _samples(case):
    """Cell-samples of all images, from the chords of a subset of the rays."""
    grid, total = _grid(case), 0.0
    for v in _views(case, 1):
        q, p = np.meshgrid(np.linspace(0, v.height - 1, 24), np.linspace(0, v.width - 1, 24), indexing="ij")
        g, a, _ = _ray_frame(v, grid, p, q)
        lo, hi = np.full(p.shape, -1e30), np.full(p.shape, 1e30)
        if v.lookback:
            lo[:] = v.c * (v.t_obs - grid.t0 - grid.n_epochs * grid.dt)
            hi[:] = v.c * (v.t_obs - grid.t0 + grid.dt)
        for i in range(3):
            s0, s1 = -g[i] / (a[i] or 1e-30), (grid.n[i] - g[i]) / (a[i] or 1e-30)
            lo, hi = np.maximum(lo, np.minimum(s0, s1)), np.minimum(hi, np.maximum(s0, s1))
        cells = np.where(hi > lo, (hi - lo) * sum(abs(x) for x in a) + 1.0, 0.0)
        total += float(cells.mean()) * v.width * v.height
    return total


def work(case):
    cells = float(case["nx"]) * case["ny"] * case["nz"] * case["epochs"]
    pixels = float(sum(v.width * v.height for v in _views(case, 1)))
    samples, per = _samples(case), 2 if case["epochs"] > 1 else 1
    record = 12.0 if case["kind"] == "serve" else 16.0 if case["store"] == "f32" else 8.0
    held = cells * (2 if case["kind"] == "serve" else 1)
    read = min(samples * per, held) * (record + 4.0 * case["channels"])
    out = pixels * 4.0 * (1 + case["channels"]) * (2 if case["samples"] else 1)
    if case["kind"] == "load":
        read += cells * ((16.0 if case["inputs"] == "f32" else 32.0) + record)
    flops = samples * (per * (24.0 if case["beaming"] else 2.0) + 16.0 + 6.0 * case["channels"])
    return {"bytes": read + out, "flops": flops}


# ------------------------------------------------------------------ the same in float64
def _exact_image(grid, view, fields, beta):
    """Eq. 19 for every pixel in float64: cell by cell along each ray, all rays of a block in step.  ``fields`` holds
    the emissivities (j' and any channels); returns one image each."""
    nx, ny, nz = grid.n
    m_all, dev = grid.n_epochs, beta.device
    js, vel = [f.reshape(-1) for f in fields], beta.reshape(-1, 3)
    kk = 1.0 / (view.c * grid.dt) if view.lookback else 0.0
    u_obs = (view.t_obs - grid.t0) / grid.dt
    win = (-1e30, 1e30)
    if view.lookback:
        win = ((u_obs - m_all) / kk, (u_obs + 1.0) / kk)
    else:
        u_obs = min(max(u_obs, 0.0), m_all - 1.0)
    out = [torch.zeros(view.height * view.width, dtype=torch.float64, device=dev) for _ in js]
    for first in range(0, view.height * view.width, 1 << 20):
        pix = torch.arange(first, min(first + (1 << 20), view.height * view.width), device=dev)
        g, a, sh = _ray_frame(view, grid, (pix % view.width).double(), (pix // view.width).double())
        lo, hi = torch.full_like(g[0], win[0]), torch.full_like(g[0], win[1])
        for i in range(3):
            if abs(a[i]) > 1e-12:
                s0, s1 = -g[i] / a[i], (grid.n[i] - g[i]) / a[i]
                lo, hi = torch.maximum(lo, torch.minimum(s0, s1)), torch.minimum(hi, torch.maximum(s0, s1))
            else:
                hi = torch.where((g[i] >= 0) & (g[i] < grid.n[i]), hi, lo - 1.0)
        keep = (hi > lo).nonzero().reshape(-1)
        if not keep.numel():
            continue
        pix, lo, g = pix[keep], lo[keep], [v[keep] for v in g]
        k, t, s_cur = [], [], torch.full_like(lo, -1e30)
        up = [1 if a[i] > 0 else 0 for i in range(3)]
        for i in range(3):
            ki = torch.floor(g[i] + lo * a[i]).clamp(0, grid.n[i] - 1)
            k.append(ki)
            if abs(a[i]) > 1e-12:
                t.append((ki + up[i] - g[i]) / a[i])
                s_cur = torch.maximum(s_cur, (ki + 1 - up[i] - g[i]) / a[i])
            else:
                t.append(torch.full_like(lo, 1e30))
        acc = [torch.zeros_like(lo) for _ in js]
        alive = torch.ones_like(lo, dtype=torch.bool)
        for step in range(nx + ny + nz + 6):
            s_exit = torch.minimum(torch.minimum(t[0], t[1]), t[2])
            ds = s_exit - s_cur
            u = u_obs - kk * 0.5 * (s_cur + s_exit)
            fl = torch.floor(u)
            w = u - fl
            m = fl.long()
            cell = ((k[2] * ny + k[1]) * nx + k[0]).long()
            good = alive & (ds > 0)
            for side in (0, 1):
                ok = good & (m + side >= 0) & (m + side < m_all)
                at = torch.where(ok, (m + side) * (nx * ny * nz) + cell, 0)
                wd = torch.where(ok, (w if side else 1.0 - w) * ds, 0.0)
                if view.beaming:
                    b = vel[at].double()
                    d = torch.sqrt(1.0 - (b * b).sum(1)) / (1.0 + b[:, 0] * sh[0] + b[:, 1] * sh[1] + b[:, 2] * sh[2])
                    wd = wd * d ** (2.0 - view.alpha)
                for c, f in enumerate(js):
                    acc[c] += wd * f[at].double()
            s_cur = torch.maximum(s_cur, s_exit)
            x0 = (t[0] <= t[1]) & (t[0] <= t[2])
            x1 = ~x0 & (t[1] <= t[2])
            for i, x in enumerate((x0, x1, ~x0 & ~x1)):
                if abs(a[i]) > 1e-12:
                    k[i] = torch.where(alive & x, k[i] + (1 if up[i] else -1), k[i])
                    t[i] = (k[i] + up[i] - g[i]) / a[i]
                    alive = alive & (k[i] >= 0) & (k[i] < grid.n[i])
            alive = alive & (s_cur < win[1])
            if step % 32 == 31 and not bool(alive.any()):
                break
        for c in range(len(js)):
            out[c][pix] = acc[c] * view.nu_ratio ** view.alpha
    return [o.reshape(view.height, view.width) for o in out]


def exact(case, seed):
    grid, views = _grid(case), _views(case, seed)
    j, beta = _fields(case, seed)
    fields = [j]
    if case["kind"] == "vector":
        fields += list(_channels(case, seed, j))
    images = [_exact_image(grid, v, fields, beta) for v in views]
    if case["kind"] in ("image", "load"):
        return images[0][0]
    if case["kind"] == "serve":
        return [im[0] for im in images]
    if case["kind"] == "vector":
        return torch.stack([torch.stack(im) for im in images])
    stack = torch.stack([im[0] for im in images])
    return [stack, None] if case["samples"] else stack
