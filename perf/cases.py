"""What a user of the raycaster has it do, as measurable cases.

Each case is one call chain through the package's public entry points (``Volume.render``,
``RaycastFn``, ``Volume.upload_level`` + ``build_lod``, a batch provider):

frame   one or more views of a resident volume (the render loop of a viewer)
train   forward + adjoint of the differentiable renderer (density and transfer function)
update  a new time step: upload a dense level, rebuild the LOD pyramid, render a frame
stream  a frame of a volume larger than its brick cache, bricks served by a batch provider

Sizes are those of the repository's workloads (synth/workloads.py, bench.py) and tests, with odd
and ragged ones between them.  Inputs are made on the GPU from the seed: fractal value noise with
embedded spheres, or Gaussian blobs with noise, as in synth/.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2509_26213_gb300 import _capi
from paper_2509_26213_gb300.volume import RaycastFn, Volume

DEV = "cuda"


def _case(kind, dims, dtype, brick, levels, w, h, views=1, **kw):
    c = {"kind": kind, "dx": dims[0], "dy": dims[1], "dz": dims[2], "dtype": dtype, "brick": brick, "levels": levels,
         "w": w, "h": h, "views": views, "layout": "quad", "data": "noise", "lod": True, "composite": "dvr",
         "skip": False, "step": 0.5}
    c.update(kw)
    return c


def listed():
    return [
        # a thumbnail of a small volume (the smoke test's size): launches and host work count
        _case("frame", (48, 40, 36), "u8", 16, 2, 40, 32, data="blobs", name="thumbnail"),
        # the plain single view: a preview pane
        _case("frame", (128, 128, 128), "u8", 32, 2, 256, 256, data="blobs", lod=False, name="frame_256"),
        # the headline: a full-HD frame of a 1024^3 scan with footprint LOD
        _case("frame", (1024, 1024, 1024), "u16", 64, 5, 1920, 1080, name="frame_1080p"),
        # a ragged float volume and an odd window, no LOD bias, 32^3 bricks
        _case("frame", (701, 333, 520), "f32", 32, 4, 1283, 717, name="frame_ragged"),
        # reduced-precision storage in the compact layout (the one a brick cache uses)
        _case("frame", (612, 612, 499), "f16", 64, 4, 1024, 768, layout="compact", name="frame_compact"),
        # the projections a microscopist looks at first
        _case("frame", (1024, 1024, 1024), "u16", 64, 5, 1920, 1080, composite="mip", name="mip_1080p"),
        _case("frame", (768, 640, 512), "u8", 32, 4, 1280, 720, composite="mop", data="blobs", skip=True,
              name="mop_skip"),
        # many views of one volume in one call (novel-view sets, 360-degree capture)
        _case("frame", (2048, 2048, 2048), "u8", 32, 6, 0, 0, views=64, data="blobs", name="batch_64"),
        # one optimisation step of the differentiable workload
        _case("train", (256, 256, 256), "f32", 32, 1, 512, 512, views=16, data="blobs", lod=False, name="train"),
        # the same through the LOD pyramid, small and ragged
        _case("train", (101, 90, 77), "f32", 16, 3, 203, 151, views=3, data="blobs", name="train_lod"),
        # the next time step of a simulation or a live acquisition
        _case("update", (512, 512, 512), "u16", 32, 4, 1280, 720, skip=True, name="update"),
        # the first frame from a new place in a volume that does not fit its cache
        _case("stream", (384, 384, 384), "u8", 64, 3, 960, 540, layout="compact", name="stream"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "train", "update", "stream"])
    hi = {"frame": 1024, "train": 256, "update": 600, "stream": 400}[kind]
    lo = {"frame": 36, "train": 48, "update": 64, "stream": 200}[kind]
    dims = tuple(_log(rng, lo, hi) for _ in range(3))
    brick = 64 if kind == "stream" else rng.choice([16, 32, 32, 64])
    levels = max(1, min(6, int(math.log2(max(dims) / brick)) + 2 if max(dims) > brick else 1))
    w = _log(rng, 40, {"frame": 1920, "train": 512, "update": 1280, "stream": 960}[kind])
    h = max(16, int(w * rng.uniform(0.5, 1.2)))
    c = _case(kind, dims, "u8", brick, levels, w, h)
    c["data"] = rng.choice(["noise", "blobs"])
    c["lod"] = rng.random() < 0.7
    c["step"] = rng.choice([0.5, 0.5, 0.5, 1.0, 0.37])
    if kind == "train":
        c.update(dtype="f32", views=rng.randint(1, 16))
        return c
    c["dtype"] = "u8" if kind == "stream" else rng.choice(["u8", "u16", "f16", "f32"])
    if kind == "frame":
        c.update(views=rng.choice([1, 1, 1, 2, 5, 12]), layout=rng.choice(["quad", "quad", "compact"]))
    if kind == "stream":
        c["layout"] = "compact"
    else:
        c.update(composite=rng.choice(["dvr", "dvr", "dvr", "mop", "mip"]), skip=rng.random() < 0.3)
    return c


# ---------------------------------------------------------------------- inputs

def _level_dims(case):
    d = (case["dx"], case["dy"], case["dz"])
    out = [d]
    for _ in range(case["levels"] - 1):
        d = tuple((x + 1) // 2 for x in d)
        out.append(d)
    return out


def _store(v, dtype):
    """Values in [0, 1] (float32) as stored voxels."""
    if dtype == "u8":
        return (v * 255.0).round_().to(torch.uint8)
    if dtype == "u16":
        return (v * 65535.0).round_().to(torch.int32).to(torch.uint16)
    return v.to(torch.float16 if dtype == "f16" else torch.float32)


def _noise(case, g):
    dx, dy, dz = case["dx"], case["dy"], case["dz"]
    v = torch.zeros((1, 1, dz, dy, dx), device=DEV)
    period, amp, tot = max(4.0, max(dx, dy, dz) / 8.0), 1.0, 0.0
    for _ in range(5):
        n = [max(2, int(math.ceil(d / period)) + 1) for d in (dz, dy, dx)]
        lat = torch.rand((1, 1, *n), generator=g, device=DEV)
        v += amp * torch.nn.functional.interpolate(lat, size=(dz, dy, dx), mode="trilinear", align_corners=True)
        tot += amp
        amp, period = amp * 0.5, max(2.0, period * 0.5)
    v = v[0, 0].div_(tot).clamp_(0.0, 1.0)
    m = max(dx, dy, dz)
    p = torch.rand((200, 5), generator=g, device=DEV).cpu().numpy()
    for cx, cy, cz, r, val in p:
        c = np.array([cz * dz, cy * dy, cx * dx])
        rad = m * (0.004 + 0.055 * float(r))
        lo = [max(0, int(c[a] - rad)) for a in range(3)]
        hi = [min((dz, dy, dx)[a], int(c[a] + rad) + 1) for a in range(3)]
        if any(lo[a] >= hi[a] for a in range(3)):
            continue
        d2 = sum((torch.arange(lo[a], hi[a], device=DEV, dtype=torch.float32) + 0.5 - float(c[a])).square()
                 .reshape([-1 if b == a else 1 for b in range(3)]) for a in range(3))
        box = v[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]]
        box.copy_(torch.where(d2 <= rad * rad, 0.3 + 0.7 * float(val), box))
    return _store(v, case["dtype"])


def _blobs(case, g):
    """Sum of Gaussian blobs (separable, so a matrix product per slab) plus uniform noise."""
    dx, dy, dz = case["dx"], case["dy"], case["dz"]
    m, n = max(dx, dy, dz), 32 if max(dx, dy, dz) > 1024 else 8
    p = torch.rand((n, 5), generator=g, device=DEV)
    sig = m * (0.04 + 0.10 * p[:, 3:4])

    def axis(d, c):
        return torch.exp(-0.5 * ((torch.arange(d, device=DEV) + 0.5)[None] - c[:, None] * d).square() / sig.square())

    gx, gy, gz = axis(dx, p[:, 0]), axis(dy, p[:, 1]), axis(dz, p[:, 2])
    gz = gz * (0.25 + 0.55 * p[:, 4:5])
    slab = max(1, min(dz, (1 << 27) // (dx * dy)))
    out = None
    for z in range(0, dz, slab):
        w = torch.einsum("bz,by->bzy", gz[:, z:z + slab], gy).reshape(n, -1).t() @ gx
        w = w.reshape(-1, dy, dx)
        w += torch.rand(w.shape, generator=g, device=DEV) * (0.06 if case["dtype"] == "u8" else 0.02)
        part = _store(w.clamp_(0.0, 1.0), case["dtype"])
        if out is None:
            out = torch.empty((dz, dy, dx), dtype=part.dtype, device=DEV)
        out[z:z + slab] = part
    return out


def _voxels(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return (_noise if case["data"] == "noise" else _blobs)(case, g)


def _camera(dims, w, h, theta, phi, inside=False):
    D = np.asarray(dims, np.float64)
    direction = np.array([math.cos(phi) * math.cos(theta), math.cos(phi) * math.sin(theta), math.sin(phi)])
    # outside: the bounding sphere fits the vertical field of view; inside: a fly-through's place
    dist = 0.3 * D.min() if inside else 0.5 * np.linalg.norm(D) / math.sin(math.radians(22.5)) * 1.1
    eye = D / 2 + dist * direction
    fwd = -direction
    right = np.cross(fwd, [0.0, 0.0, 1.0])
    right /= np.linalg.norm(right)
    f = np.float32
    return {"eye": f(eye), "right": f(right), "up": f(np.cross(right, fwd)), "fwd": f(fwd),
            "tan_half_fov": f(math.tan(math.radians(22.5))), "aspect": f(w / h), "w": int(w), "h": int(h)}


def _cameras(case, seed):
    rng = np.random.default_rng(seed)
    cams = []
    for i in range(case["views"]):
        w, h = case["w"], case["h"]
        if w == 0:  # the batched workload's sides
            w = h = (256, 512, 768, 1024)[i % 4]
        cams.append(_camera((case["dx"], case["dy"], case["dz"]), w, h, rng.uniform(0, 2 * math.pi),
                            math.radians(rng.uniform(-30, 30)), inside=case["kind"] == "stream"))
    return cams


def _tf(case, seed):
    """Opacity peaks for the noise volumes, a colour ramp for the blobs."""
    rng = np.random.default_rng(seed + 1)
    x = np.arange(256) / 255.0
    if case["data"] == "blobs":
        a = np.where(x < 0.1, 0.0, 0.08 * (x - 0.1) / 0.9)
        rgb = np.stack([np.clip(0.2 + 0.8 * x, 0, 1), x * x, 1.0 - x], 1)
    else:
        a, rgb = np.zeros(256), np.zeros((256, 3))
        for _ in range(3):
            c, hw, ht, col = rng.uniform(0.2, 0.9), rng.uniform(0.02, 0.1), rng.uniform(0.05, 0.5), rng.random(3)
            p = ht * np.clip(1.0 - np.abs(x - c) / hw, 0.0, None)
            rgb[p > a] = col
            a = np.maximum(a, p)
    return torch.from_numpy(np.concatenate([rgb, a[:, None]], 1).astype(np.float32)).to(DEV)


def _params(case):
    return {"step": case["step"], "et": 0.99, "bg": (0.1, 0.2, 0.3, 0.0), "lod_mode": int(case["lod"]),
            "composite": case["composite"], "flags": _capi.VOL_RENDER_SKIP_EMPTY if case["skip"] else 0}


def _pyramid(vox, case):
    """Every level's stored voxels: 2x2x2 box filter, an index past the edge being the last voxel."""
    out = [vox]
    for _ in range(case["levels"] - 1):
        v = out[-1]
        dt = case["dtype"]
        v = v.to(torch.int32) if dt in ("u8", "u16") else v.to(torch.float32)
        for a in range(3):
            if v.shape[a] & 1:
                v = torch.cat([v, v.narrow(a, v.shape[a] - 1, 1)], a)
        s = None
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    p = v[dz::2, dy::2, dx::2]
                    s = p.clone() if s is None else s + p
        if dt in ("u8", "u16"):
            out.append(((s + 4) >> 3).to(vox.dtype))
        else:
            out.append((s * 0.125).to(vox.dtype))
    return out


def _upstream(case, cams, seed):
    """The gradient that arrives from a loss on the images."""
    n = sum(c["w"] * c["h"] for c in cams)
    g = torch.Generator(device=DEV).manual_seed(seed + 2)
    return torch.randn((n, 4), generator=g, device=DEV) / n


class _Bricks:
    """Host-side brick store behind a batch provider: every brick with its apron, cut once."""

    def __init__(self, case, vox):
        B = case["brick"]
        self.at, cut = {}, []
        for l, v in enumerate(_pyramid(vox, case)):
            v = v.cpu().numpy()
            nb = [(s + B - 1) // B for s in v.shape]
            for bz in range(nb[0]):
                for by in range(nb[1]):
                    for bx in range(nb[2]):
                        ix = [np.minimum(np.arange(b * B, b * B + B + 1), s - 1)
                              for b, s in zip((bz, by, bx), v.shape)]
                        self.at[(l, bx, by, bz)] = len(cut)
                        cut.append(v[np.ix_(*ix)])
        self.store = np.ascontiguousarray(np.stack(cut))
        self.nbytes = self.store[0].nbytes

        def fill(_user, n, reqs, dst):
            for i in range(n):
                b = self.at[(reqs[4 * i], reqs[4 * i + 1], reqs[4 * i + 2], reqs[4 * i + 3])]
                ctypes.memmove(dst + i * self.nbytes, self.store.ctypes.data + b * self.nbytes, self.nbytes)
            return 0

        self.fn = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.POINTER(ctypes.c_int32),
                                   ctypes.c_void_p)(fill)
        self.address = ctypes.cast(self.fn, ctypes.c_void_p).value


def prepare(case, seed):
    dims = (case["dx"], case["dy"], case["dz"])
    vox = _voxels(case, seed)
    cams, tf, params = _cameras(case, seed), _tf(case, seed), _params(case)
    st = {"kind": case["kind"], "cams": cams, "tf": tf, "params": params, "levels": case["levels"]}
    if case["kind"] == "stream":
        st["bricks"] = _Bricks(case, vox)
        cache = int(0.6 * st["bricks"].store.nbytes)  # the cache holds about 60 % of the bricks
        st["vol"] = Volume(dims, case["dtype"], case["brick"], case["levels"], cache_bytes=cache, layout=case["layout"])
        st["vol"].set_provider_batch(st["bricks"].address, ctypes.c_int(0), case["dtype"])
        return st
    st["vol"] = Volume(dims, case["dtype"], case["brick"], case["levels"], layout=case["layout"])
    if case["kind"] == "frame":
        st["vol"].upload_level(0, vox, case["dtype"])
        if case["levels"] > 1:
            st["vol"].build_lod(0)
        torch.cuda.synchronize()
        st["vol"]._keep = None  # the source is not needed any more
    elif case["kind"] == "update":
        st["vox"], st["dtype"] = vox, case["dtype"]
    else:
        st["vox"] = vox.requires_grad_(True)
        st["tf"] = tf.requires_grad_(True)
        st["g"] = _upstream(case, cams, seed)
    return st


def run(st):
    vol = st["vol"]
    if st["kind"] == "train":
        out = RaycastFn.apply(st["vox"], st["tf"], vol, st["cams"], st["params"])
        return (out.detach(), *torch.autograd.grad(out, (st["vox"], st["tf"]), st["g"]))
    if st["kind"] == "update":
        vol.upload_level(0, st["vox"], st["dtype"])
        if st["levels"] > 1:
            vol.build_lod(0)
    elif st["kind"] == "stream":
        vol.evict_all()
    return vol.render(st["cams"], st["tf"], st["params"])


def _ray_samples(case):
    """Samples per level of the case's rays without early termination, from 48 x 48 rays of each of
    up to 8 views (a fixed seed's cameras)."""
    dims = np.array([case["dx"], case["dy"], case["dz"]], np.float64)
    cams = _cameras(case, 0)
    per = np.zeros(case["levels"])
    for c in cams[:8]:
        u, v = np.meshgrid((np.arange(48) + 0.5) / 24 - 1, 1 - (np.arange(48) + 0.5) / 24)
        t = float(c["tan_half_fov"])
        d = c["fwd"] + (u * t * float(c["aspect"]))[..., None] * c["right"] + (v * t)[..., None] * c["up"]
        d = d / np.linalg.norm(d, axis=-1, keepdims=True)
        a, b = (0 - c["eye"]) / d, (dims - c["eye"]) / d
        t0 = np.maximum(np.minimum(a, b).max(-1), 0)
        t1 = np.maximum(a, b).min(-1)
        px = c["w"] * c["h"] / 2304.0 * len(cams) / min(8, len(cams))
        for l in range(case["levels"]):
            lo, hi = (0.0, np.inf) if not case["lod"] else (2.0 ** l, 2.0 ** (l + 1))
            if case["lod"] and l == 0:
                lo = 0.0
            if case["lod"] and l == case["levels"] - 1:
                hi = np.inf
            s = 2 * t / c["h"]
            seg = np.clip(np.minimum(t1, hi / s) - np.maximum(t0, lo / s), 0, None)
            per[l] += px * seg.sum() / case["step"]
            if not case["lod"]:
                break
    return per


def work(case):
    """Voxels the rays can touch (each read once), images written, and about 70 operations per sample
    (position, voxel, 8-corner interpolation, transfer function, compositing; twice that again for the
    adjoint).  Early termination, which depends on the data, is counted as half of the samples."""
    bpv = {"u8": 1, "u16": 2, "f16": 2, "f32": 4}[case["dtype"]]
    dims = _level_dims(case)
    vox = [float(np.prod(d)) for d in dims]
    n = _ray_samples(case) * (0.5 if case["composite"] == "dvr" else 1.0)
    px = sum(c["w"] * c["h"] for c in _cameras(case, 0))
    b = 16.0 * px + 4096 + sum(min(v, k) for v, k in zip(vox, n)) * bpv
    f = 70.0 * n.sum()
    if case["kind"] == "train":
        b += 16.0 * px + 4.0 * vox[0] + 4096  # upstream gradient, dL/ddensity, dL/dtf
        f *= 3
    elif case["kind"] == "update":
        b += vox[0] * bpv + sum(vox[1:]) * bpv
        f += 8.0 * sum(vox[1:])
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------- exact values

def _rays(c, dims):
    """Ray set-up of a view in binary32, each operation rounded once."""
    f = lambda x: torch.tensor(x, dtype=torch.float32, device=DEV)
    px = torch.arange(c["w"], device=DEV, dtype=torch.float32) + 0.5
    py = torch.arange(c["h"], device=DEV, dtype=torch.float32) + 0.5
    tan, asp = f(c["tan_half_fov"]), f(c["aspect"])
    cx = (px / f(float(c["w"])) * 2.0 - 1.0) * (tan * asp)
    cy = (1.0 - py / f(float(c["h"])) * 2.0) * tan
    cx, cy = cx[None].expand(c["h"], -1).reshape(-1), cy[:, None].expand(-1, c["w"]).reshape(-1)
    dd = [(cx * f(c["right"][a]) + f(c["fwd"][a])) + cy * f(c["up"][a]) for a in range(3)]
    inv = torch.ones_like(cx) / torch.sqrt(dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2])
    t0, t1 = torch.zeros_like(cx), torch.full_like(cx, math.inf)
    hit = torch.ones_like(cx, dtype=torch.bool)
    o, d = [f(c["eye"][a]) for a in range(3)], []
    for a in range(3):
        da = dd[a] * inv
        d.append(da)
        ta, tb = (0.0 - o[a]) / da, (f(float(dims[a])) - o[a]) / da
        zero = da == 0
        hit &= ~zero | ((o[a] >= 0) & (o[a] < dims[a]))
        t0 = torch.where(zero, t0, torch.maximum(t0, torch.minimum(ta, tb)))
        t1 = torch.where(zero, t1, torch.minimum(t1, torch.maximum(ta, tb)))
    return o, d, t0, t1, hit & (t0 < t1)


class _Exact:
    """The renderer in float64 on plain tensors: binary32 sample positions, levels and voxels (they
    are part of the image's definition), values, compositing and gradients in float64."""

    K = 32  # samples per block

    def __init__(self, case, seed, pyramid):
        self.case = case
        self.p = _params(case)
        self.dims = _level_dims(case)
        self.tf = _tf(case, seed).double()
        n = len(pyramid) if case["lod"] else 1
        conv = torch.int32 if case["dtype"] == "u16" else pyramid[0].dtype
        self.flat = torch.cat([v.to(conv).reshape(-1) for v in pyramid[:n]])
        tab = lambda x, dt: torch.tensor(x, dtype=dt, device=DEV)
        self.off = tab(np.cumsum([0] + [int(np.prod(d)) for d in self.dims])[:n].tolist(), torch.int64)
        self.D = tab([list(d) for d in self.dims[:n]], torch.int64)
        self.r = tab([[float(d[a]) for a in range(3)] for d in self.dims[:n]], torch.float32) / \
            tab([float(x) for x in self.dims[0]], torch.float32)
        self.nlev = n
        self.scale = {"u8": 1.0, "u16": 255.0 / 65535.0, "f16": 255.0, "f32": 255.0}[case["dtype"]]

    def sample(self, R, k0):
        """Block of samples k0 .. k0 + K - 1 of rays R: valid, TF coordinate, cell base, strides, weights."""
        o, d, t0, t1, lodscale = R
        k = torch.arange(k0, k0 + self.K, device=DEV, dtype=torch.float32)
        t = t0[:, None] + (k * float(self.p["step"]))[None]
        ok = t < t1[:, None]
        if self.nlev > 1:
            e = ((t * lodscale).view(torch.int32) >> 23) - 127
            l = e.clamp(0, self.nlev - 1).long()
        else:
            l = torch.zeros_like(t, dtype=torch.int64)
        i0, w, D = [], [], []
        for a in range(3):
            Da = self.D[:, a][l]
            x = (t * d[a][:, None] + o[a]) * self.r[:, a][l] - 0.5
            x = torch.minimum(x.clamp(min=0.0), (Da - 1).float())
            fl = torch.floor(x)
            i0.append(fl.long())
            w.append((x - fl).double())
            D.append(Da)
        sy, sz = D[0], D[0] * D[1]
        base = self.off[l] + i0[0] + i0[1] * sy + i0[2] * sz
        step = [torch.where(i0[0] < D[0] - 1, 1, 0), torch.where(i0[1] < D[1] - 1, sy, 0),
                torch.where(i0[2] < D[2] - 1, sz, 0)]
        val = None
        for c in range(8):
            wc, at = None, base
            for a in range(3):
                f = w[a] if (c >> a) & 1 else 1.0 - w[a]
                wc = f if wc is None else wc * f
                if (c >> a) & 1:
                    at = at + step[a]
            v = self.flat[torch.where(ok, at, 0)].double() * wc
            val = v if val is None else val + v
        x = val * self.scale
        inside = (x >= 0) & (x <= 255.0)
        return ok, x.clamp(0.0, 255.0), base, step, w, inside

    def lookup(self, x):
        i = x.long().clamp(max=254)
        w = (x - i).unsqueeze(-1)
        a = self.tf[i]
        return a + w * (self.tf[i + 1] - a), i, w.squeeze(-1)

    def view_rays(self, c):
        o, d, t0, t1, hit = _rays(c, self.dims[0])
        scale = float(np.float32(np.float32(2.0) * np.float32(c["tan_half_fov"])) / np.float32(c["h"]))
        return o, d, t0, t1, hit, scale

    def march(self, c, rec=None):
        """One view's image [w * h, 4]; rec receives (ray indices, T at block start, samples kept) per block."""
        o, d, t0, t1, hit, scale = self.view_rays(c)
        bg = torch.tensor(self.p["bg"], dtype=torch.float32, device=DEV).double()
        mode = self.case["composite"]
        out = bg.expand(t0.numel(), 4).clone()
        for idx in torch.nonzero(hit).reshape(-1).split(1 << 18):
            n = idx.numel()
            C = torch.zeros((n, 3), dtype=torch.float64, device=DEV)
            T = torch.full((n,), {"dvr": 1.0, "mop": 0.0, "mip": -1.0}[mode], dtype=torch.float64, device=DEV)
            live, k0 = torch.arange(n, device=DEV), 0
            while live.numel():
                at = idx[live]
                R = (o, [x[at] for x in d], t0[at], t1[at], scale)
                ok, x, *_ = self.sample(R, k0)
                Tl = T[live]
                if mode == "mip":
                    Tl = torch.maximum(Tl, torch.where(ok, x, -1.0).amax(1))
                    T[live] = Tl
                    go = ok[:, -1] & (Tl < 255.0)
                else:
                    rgba = self.lookup(x)[0]
                    a = torch.where(ok, rgba[..., 3], -1.0 if mode == "mop" else 0.0)
                    if mode == "mop":
                        best, j = a.max(1)
                        take = best > Tl
                        col = rgba.gather(1, j[:, None, None].expand(-1, 1, 4))[:, 0, :3]
                        C[live] = torch.where(take[:, None], col, C[live])
                        T[live] = torch.maximum(Tl, best)
                        go = ok[:, -1]
                    else:
                        Tk = Tl[:, None] * torch.cumprod(torch.cat([torch.ones_like(a[:, :1]), 1.0 - a], 1), 1)
                        done = (1.0 - Tk) >= float(np.float32(self.p["et"]))
                        use = ok & ~done[:, :-1]
                        C[live] += (torch.where(use, Tk[:, :-1] * a, 0.0)[..., None] * rgba[..., :3]).sum(1)
                        cnt = use.sum(1)
                        if rec is not None:
                            rec.append((at, k0, Tl, cnt))
                        T[live] = Tk.gather(1, cnt[:, None])[:, 0]
                        go = (cnt == self.K) & ~done[:, -1]
                live, k0 = live[go], k0 + self.K
            if mode == "mip":
                rgba = self.lookup(T.clamp(min=0.0))[0]
                al, C = torch.where(T >= 0, rgba[:, 3], 0.0), rgba[:, :3]
            else:
                al = T
            if mode == "dvr":
                out[idx] = torch.cat([C + T[:, None] * bg[:3], (1.0 - T + T * bg[3])[:, None]], 1)
            else:
                out[idx] = torch.cat([al[:, None] * C + (1.0 - al)[:, None] * bg[:3],
                                      (al + (1.0 - al) * bg[3])[:, None]], 1)
        return out

    def grads(self, c, rec, g, dflat, dtf):
        """Adds a view's gradients to dflat (every level, flat) and dtf."""
        o, d, t0, t1, _, scale = self.view_rays(c)
        bg = torch.tensor(self.p["bg"], dtype=torch.float32, device=DEV).double()
        behind = bg.expand(t0.numel(), 4).clone()
        for at, k0, Tl, cnt in reversed(rec):
            R = (o, [x[at] for x in d], t0[at], t1[at], scale)
            _, x, base, step, w, inside = self.sample(R, k0)
            use = torch.arange(self.K, device=DEV)[None] < cnt[:, None]
            rgba, i, wt = self.lookup(x)
            a = torch.where(use, rgba[..., 3], 0.0)
            Tk = Tl[:, None] * torch.cumprod(torch.cat([torch.ones_like(a[:, :1]), 1.0 - a[:, :-1]], 1), 1)
            gv, B = g[at].double(), behind[at]
            dal = torch.empty_like(a)
            for j in range(self.K - 1, -1, -1):
                col = torch.cat([rgba[:, j, :3], torch.ones_like(a[:, :1])], 1)
                dal[:, j] = Tk[:, j] * (gv * (col - B)).sum(1)
                B = B + a[:, j:j + 1] * (col - B)
            behind[at] = B
            d4 = torch.cat([gv[:, None, :3] * (Tk * a)[..., None], dal[..., None]], 2)
            d4 = torch.where(use[..., None], d4, 0.0)
            # few entries receive everything: sum per entry on the sorted order of a histogram
            m = i.reshape(-1)
            for e, f in ((0, 1.0 - wt), (1, wt)):
                v = (d4 * f[..., None]).reshape(-1, 4)
                for ch in range(4):
                    dtf[:, ch] += torch.bincount(m + e, weights=v[:, ch], minlength=256)
            dv = 255.0 * (d4 * (self.tf[i + 1] - self.tf[i])).sum(-1)
            dv = torch.where(use & inside, dv, 0.0)
            for cnr in range(8):
                wc, p = dv, base
                for ax in range(3):
                    wc = wc * (w[ax] if (cnr >> ax) & 1 else 1.0 - w[ax])
                    if (cnr >> ax) & 1:
                        p = p + step[ax]
                dflat.index_add_(0, torch.where(use, p, 0).reshape(-1), wc.reshape(-1))

    def level0(self, dflat):
        """Carries coarser levels' gradients to level 0 through the box filter's adjoint."""
        parts = [dflat[int(self.off[l]):int(self.off[l]) + int(np.prod(self.dims[l]))].reshape(
            self.dims[l][2], self.dims[l][1], self.dims[l][0]) for l in range(self.nlev)]
        for l in range(self.nlev - 1, 0, -1):
            up, fine = parts[l] * 0.125, parts[l - 1]
            for a in range(3):
                up = up.repeat_interleave(2, a)
                if fine.shape[a] & 1:
                    n = fine.shape[a]
                    last = up.narrow(a, n - 1, 2).sum(a, keepdim=True)
                    up = torch.cat([up.narrow(a, 0, n - 1), last], a)
            parts[l - 1] = fine + up
        return parts[0]


def exact(case, seed):
    if case["views"] * case["dx"] > 40000:
        return None  # 64 views of 2048^3: 2e10 samples
    X = _Exact(case, seed, _pyramid(_voxels(case, seed), case))
    cams = _cameras(case, seed)
    if case["kind"] != "train":
        return torch.cat([X.march(c) for c in cams])
    g = _upstream(case, cams, seed)
    dflat = torch.zeros(X.flat.numel(), dtype=torch.float64, device=DEV)
    dtf = torch.zeros((256, 4), dtype=torch.float64, device=DEV)
    imgs, at = [], 0
    for c in cams:
        rec, n = [], c["w"] * c["h"]
        imgs.append(X.march(c, rec))
        X.grads(c, rec, g[at:at + n], dflat, dtf)
        at += n
    return torch.cat(imgs), X.level0(dflat), dtf
