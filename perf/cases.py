"""The work a user has this renderer do, as measurable cases.

A case is one pass through the public entry points on inputs that are drawn
from a seed: a frame of a resident particle set, the allocation-free frame, a
batch of views, a set streamed from host memory, the whole host-to-host frame
(upload, encode, render, download), and a training step of the tile-cost
network.  The particle sets follow the package's own scenes (uniform with
log-normal smoothing lengths; Plummer haloes over a diffuse background with
density-derived smoothing lengths, grouped by halo as a snapshot is; heavy-
tailed smoothing lengths), drawn on the GPU so that a new set costs
milliseconds.
"""
from __future__ import annotations

import ctypes as C
import functools
import math

import numpy as np
import torch

from paper_1309_1114_gb300 import scenes
from paper_1309_1114_gb300 import splotch as S

CHI = 3.0            # the library's default clip factor
R_POINT = 0.5        # its default point radius
H_LOG2_MIN = -14.0   # log2 of the smoothing length of code 0 (16-bit log codes)
ATTRS = {"f32": S.SPL_ATTR_F32, "f16": S.SPL_ATTR_F16, "f16_is": S.SPL_ATTR_F16_IS,
         "logh16": S.SPL_ATTR_LOGH16}
MODES = {"additive": S.SPL_MODE_ADDITIVE, "ea": S.SPL_MODE_EA, "absorb": S.SPL_MODE_ABSORB}
COST_LIMIT = 6.0e10  # covered (particle, pixel) pairs of the largest listed case
EXACT_PAIRS = 1.6e10  # box pixels up to which the 64-bit image is worked out
NFEAT, NHID, NPARAM = 32, 64, S.SPL_MLP_NPARAM


def _case(name, kind, scene, n, width, height, **over):
    c = {"name": name, "kind": kind, "scene": scene, "n": n, "width": width, "height": height,
         "attr": "f32", "mode": "additive", "support": False, "rgb": False, "tile": 32,
         "azimuth": 0.0, "views": 1, "chunk": 0}
    c.update(over)
    return c


def listed():
    return [
        # a thumbnail through the allocation-free call: launches and waits are all of it
        _case("noalloc_thumb_20k", "noalloc", "uniform", 20_000, 96, 80),
        # an interactive preview of a small set
        _case("preview_200k", "frame", "uniform", 200_000, 256, 256),
        # a movie frame of a medium set: ragged sides, a direct RGB quantity, the E = A map
        _case("movie_rgb_1.3M", "frame", "clustered", 1_300_000, 1366, 768, mode="ea", rgb=True,
              azimuth=30.0),
        # the ordinary frame
        _case("frame_10M", "frame", "clustered", 10_000_000, 1024, 1024),
        # h read as the support radius (sigma = h / chi), 18-byte layout, full-HD
        _case("support_logh16_30M", "frame", "clustered", 30_000_000, 1920, 1080, attr="logh16",
              support=True, mode="ea"),
        # the largest ordinary frame
        _case("frame_100M", "frame", "clustered", 100_000_000, 2048, 2048),
        # heavy-tailed radii: most particles are points, some cover the image
        _case("heavy_tail_100M", "frame", "pareto", 100_000_000, 4096, 4096),
        # general absorption: depth sort and front-to-back compositing
        _case("absorb_10M", "frame", "clustered", 10_000_000, 1024, 1024, mode="absorb"),
        # an orbit rendered as one batch, resolutions cycling 512, 1024, 2048
        _case("orbit_1M_6views", "batch", "clustered", 1_000_000, 2048, 2048, views=6),
        # a set that stays in page-locked host memory, eight chunks
        _case("stream_32M", "stream", "clustered", 32_000_000, 2048, 2048, chunk=4_000_000),
        # a new snapshot from host memory to a host image, stored in 18 bytes per particle
        _case("snapshot_logh16_4M", "host", "clustered", 4_000_000, 1024, 1024, attr="logh16"),
        # one full-batch training step of the tile-cost network: gradient and Adam
        _case("train_step_8k", "train", "features", 8_000, 0, 0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["noalloc", "frame", "frame", "frame", "frame", "absorb", "batch",
                           "stream", "host", "train"])
        if kind == "train":
            return _unnamed("train", "features", log_int(500, 100_000), 0, 0)
        over = {"azimuth": round(rng.uniform(0.0, 360.0), 3), "rgb": rng.random() < 0.2,
                "tile": rng.choice([32, 32, 32, 16, 64])}
        w, h = log_int(64, 2048), log_int(64, 2048)
        scene = rng.choice(["uniform", "clustered", "clustered", "pareto"])
        mode = rng.choice(["additive", "additive", "ea"])
        if kind == "noalloc":
            scene = rng.choice(["uniform", "clustered"])
            n, w, h = log_int(1_000, 60_000), log_int(48, 512), log_int(48, 512)
        elif kind == "frame":
            n = log_int(20_000, {"uniform": 3_000_000, "pareto": 60_000_000}.get(scene, 60_000_000))
            if scene == "pareto":
                w, h = log_int(256, 4096), log_int(256, 4096)
            over["attr"] = rng.choice(["f32", "f32", "f16", "f16_is", "logh16"])
            over["support"] = rng.random() < 0.25
        elif kind == "absorb":
            kind, mode = "frame", "absorb"
            n, w, h = log_int(20_000, 6_000_000), log_int(64, 1024), log_int(64, 1024)
            if scene == "uniform":
                n = min(n, 1_000_000)
        elif kind == "batch":
            n = log_int(50_000, 3_000_000)
            scene = "clustered"
            over["views"] = rng.randint(2, 16)
        elif kind == "stream":
            n = log_int(500_000, 30_000_000)
            scene = "clustered"
            over["chunk"] = max(1, n // rng.randint(2, 9))
        else:
            n = log_int(20_000, 5_000_000)
            scene = "clustered"
            over["attr"] = rng.choice(["f32", "f16", "logh16"])
        case = _unnamed(kind, scene, n, w, h, mode=mode, **over)
        if _pairs(case) * (1.6 if mode == "absorb" else 1.0) <= COST_LIMIT / 4:
            return case


def _unnamed(*a, **over):
    c = _case("", *a, **over)
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs
def _halo_table(seed):
    """500 haloes: masses, Plummer scale radii, centres."""
    rng = np.random.default_rng(seed)
    u = rng.random(500)
    m = (1.0 + u * (1e3 ** -0.9 - 1.0)) ** (1.0 / -0.9)
    a = 0.002 + 0.048 * (np.cbrt(m) - 1.0) / (np.cbrt(1e3) - 1.0)
    return m, a, 0.1 + 0.8 * rng.random((500, 3))


def _clustered(n, seed, dev, sample=None):
    """Positions and number densities of n particles, 70 % in haloes (grouped by
    halo) and 30 % uniform; sample: that many of them, with the densities of n."""
    m, a, ctr = _halo_table(seed)
    k = n if sample is None else min(sample, n)
    per_halo = np.floor(0.7 * n * m / m.sum())
    n_bg = n - per_halo.sum()
    counts = per_halo if k == n else np.floor(per_halo * (k / n))
    counts = torch.from_numpy(counts.astype(np.int64)).to(dev)
    in_halo = int(counts.sum())
    g = torch.Generator(dev).manual_seed(seed)
    xyz = torch.rand((3, k), generator=g, device=dev)
    dens = torch.full((k,), float(n_bg), device=dev)
    if in_halo:
        hid = torch.repeat_interleave(torch.arange(500, device=dev), counts, output_size=in_halo)
        ah = torch.from_numpy(a.astype(np.float32)).to(dev)[hid]
        nh = torch.from_numpy(per_halo.astype(np.float32)).to(dev)[hid]
        u = torch.rand((in_halo,), generator=g, device=dev).mul_(0.999).clamp_(min=1e-7)
        rad = ah / torch.sqrt(u.pow(-2.0 / 3.0) - 1.0)
        cth = 1.0 - 2.0 * torch.rand((in_halo,), generator=g, device=dev)
        phi = torch.rand((in_halo,), generator=g, device=dev).mul_(2.0 * math.pi)
        sth = torch.sqrt((1.0 - cth * cth).clamp_(min=0.0))
        for axis, d in enumerate((sth * torch.cos(phi), sth * torch.sin(phi), cth)):
            c = torch.from_numpy(ctr[:, axis].astype(np.float32)).to(dev)[hid]
            p = c + rad * d
            xyz[axis, :in_halo] = (p - torch.floor(p)).clamp_(max=1.0 - 6e-8)   # periodic box
        dens[:in_halo] += 3.0 * nh / (4.0 * math.pi * ah ** 3) * (1.0 + (rad / ah) ** 2).pow(-2.5)
    return xyz, dens, g


def _particles(case, seed, dev, sample=None):
    """x, y, z, h, I, s (and cr, cg, cb) as float32 tensors on dev."""
    n = case["n"]
    k = n if sample is None else min(sample, n)
    if case["scene"] == "uniform":
        g = torch.Generator(dev).manual_seed(seed)
        xyz = torch.rand((3, k), generator=g, device=dev)
        h = torch.exp(math.log(0.005) + 0.5 * torch.randn((k,), generator=g, device=dev))
    else:
        xyz, dens, g = _clustered(n, seed, dev, sample)
        if case["scene"] == "clustered":
            h = (scenes.ETA_SPH * dens.pow(-1.0 / 3.0)).clamp_(1e-4, 0.05)
        else:
            # r = 0.5 px at depth 2 for the commonest particle, Pareto tail (alpha 1.5),
            # capped where r at depth 2 is the image diagonal
            f = 0.5 * case["height"] / math.tan(math.radians(30.0))
            h_m = 0.5 * 2.0 / (CHI * f)
            cap = math.hypot(case["width"], case["height"]) * 2.0 / (CHI * f)
            u = 1.0 - torch.rand((k,), generator=g, device=dev)
            h = (h_m * u.clamp_(min=1e-7).pow(-1.0 / 1.5)).clamp_(max=cap)
    p = {"x": xyz[0], "y": xyz[1], "z": xyz[2], "h": h,
         "I": torch.rand((k,), generator=g, device=dev),
         "s": torch.rand((k,), generator=g, device=dev)}
    if case["rgb"]:
        p.update({c: torch.rand((k,), generator=g, device=dev) for c in ("cr", "cg", "cb")})
    return p


def _cameras(case):
    if case["kind"] != "batch":
        return [scenes.camera(case["width"], case["height"], azimuth_deg=case["azimuth"])]
    cams = scenes.orbit_cameras(case["views"], step_deg=360.0 / case["views"])
    w, h = case["width"], case["height"]
    return [dict(c, width=max(8, c["width"] * w // 2048), height=max(8, c["height"] * h // 2048))
            for c in cams]


def _features(case, seed, dev):
    """Item features and log cycles as recorded: log1p counts over radius bins,
    log1p covered areas, and a cost that grows with both; a network and Adam
    moments part-way through training."""
    n = case["n"]
    rng = np.random.default_rng(seed)
    theta = np.zeros(NPARAM, np.float32)
    theta[:NHID * NFEAT] = rng.normal(0.0, math.sqrt(2.0 / NFEAT), NHID * NFEAT)
    theta[NHID * NFEAT:NHID * NFEAT + NHID] = rng.normal(0.0, 0.1, NHID)
    theta[NHID * NFEAT + NHID:-1] = rng.normal(0.0, math.sqrt(1.0 / NHID), NHID)
    theta[-1] = 11.0
    m = rng.normal(0.0, 1e-2, NPARAM).astype(np.float32)
    v = (rng.normal(0.0, 1e-1, NPARAM) ** 2 + 1e-4).astype(np.float32)
    g = torch.Generator(dev).manual_seed(seed)
    cnt = torch.rand((n, 16), generator=g, device=dev).mul_(7.0)
    cnt[:, 9:] *= (torch.rand((n, 7), generator=g, device=dev) < 0.2)
    area = (cnt + torch.linspace(-4.0, 2.0, 16, device=dev)).clamp_(min=0.0)
    x = torch.cat([cnt, area], 1).contiguous()
    t = 9.0 + 0.25 * area.sum(1) / 4.0 + 0.2 * torch.randn((n,), generator=g, device=dev)
    d = lambda a: torch.from_numpy(a).to(dev)  # noqa: E731
    return {"x": x, "t": t.contiguous(), "theta": d(theta), "m": d(m), "v": d(v)}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        st = _features(case, seed, "cuda")
        st.update(case=case, step=1000, grad=torch.empty(NPARAM, device="cuda"),
                  loss=torch.empty(1, device="cuda"))
        return st
    parts = _particles(case, seed, "cuda")
    cams = _cameras(case)
    pal = scenes.ramp_palette()
    params = {"mode": MODES[case["mode"]], "tile_px": case["tile"]}
    if case["support"]:
        params["sigma_per_h"] = 1.0 / CHI
    image = lambda c: torch.empty((c["height"], c["width"], 3), device="cuda")  # noqa: E731
    if kind == "noalloc":
        p = S.spl_particles(case["n"], *[parts[k].data_ptr() for k in ("x", "y", "z", "h", "I", "s")],
                            S.SPL_ATTR_F32, S.SPL_MEM_DEVICE)
        if case["rgb"]:
            p.cr, p.cg, p.cb = (parts[k].data_ptr() for k in ("cr", "cg", "cb"))
        return {"case": case, "parts": parts, "p": p, "cam": S.make_camera(cams[0]),
                "q": S.default_params(**params), "pal": np.ascontiguousarray(pal),
                "image": image(cams[0])}
    r = S.Renderer(0)
    r.set_colormap(pal)
    r.set_params(**params)
    r.set_camera(cams[0])
    st = {"case": case, "r": r, "cams": cams}
    if kind in ("stream", "host"):
        st["parts"] = {k: v.cpu().pin_memory() for k, v in parts.items()}
    elif case["attr"] == "f32":
        r.load(parts)
    else:
        r.load(parts, store_as=ATTRS[case["attr"]], h_log2_min=H_LOG2_MIN)
    if kind == "host":
        st["out"] = torch.empty((case["height"], case["width"], 3)).pin_memory().numpy()
    else:
        st["images"] = [image(c) for c in cams]
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "frame":
        return state["r"].render(state["images"][0])
    if kind == "batch":
        return state["r"].render_batch(state["cams"], state["images"])
    if kind == "stream":
        return state["r"].render_stream(state["parts"], case["chunk"], state["images"][0])
    if kind == "host":
        r = state["r"]
        if case["attr"] == "f32":
            r.load(state["parts"])
        else:
            r.load(state["parts"], store_as=ATTRS[case["attr"]], h_log2_min=H_LOG2_MIN)
        return r.render_host(state["out"])
    if kind == "noalloc":
        S.check(S.spl_render_noalloc(C.byref(state["p"]), C.byref(state["cam"]), C.byref(state["q"]),
                                     state["pal"].ctypes.data, state["pal"].shape[0], 0.0, 1.0,
                                     state["image"].data_ptr(), 0, None), "spl_render_noalloc")
        return state["image"]
    # a training step: the gradient of the loss over all samples, then Adam in place
    ptr = {k: state[k].data_ptr() for k in ("theta", "x", "t", "grad", "loss", "m", "v")}
    S.check(S.spl_mlp_loss_grad(ptr["theta"], ptr["x"], ptr["t"], case["n"], ptr["grad"],
                                ptr["loss"], None), "spl_mlp_loss_grad")
    S.check(S.spl_mlp_adam(ptr["theta"], ptr["grad"], ptr["m"], ptr["v"], NPARAM, state["step"],
                           3e-3, 0.9, 0.999, 1e-8, None), "spl_mlp_adam")
    return {k: state[k] for k in ("grad", "loss", "theta", "m", "v")}


# ------------------------------------------------------------- work, 64 bits
def _project(case, cam, p):
    """Screen position, smoothing length, radius and depth in 64 bits, and which
    particles are active."""
    d = lambda v: np.asarray(v, np.float64)  # noqa: E731
    fwd = d(cam["target"]) - d(cam["eye"])
    fwd /= np.linalg.norm(fwd)
    right = np.cross(fwd, d(cam["up"]))
    right /= np.linalg.norm(right)
    up = np.cross(right, fwd)
    xyz = [p[k].double() for k in ("x", "y", "z")]
    xc, yc, zc = (sum(ax[i] * (xyz[i] - float(cam["eye"][i])) for i in range(3))
                  for ax in (right, up, fwd))
    w, h = cam["width"], cam["height"]
    f = 0.5 * h / math.tan(math.radians(0.5 * cam["fov_y_deg"]))
    safe = torch.where(zc > cam["z_near"], zc, torch.ones_like(zc))
    xs = 0.5 * w + f * xc / safe
    ys = 0.5 * h - f * yc / safe
    sig = p["h"].double() * (f / (CHI if case["support"] else 1.0)) / safe
    r = CHI * sig
    act = (zc > cam["z_near"]) & (xs + r >= 0) & (xs - r < w) & (ys + r >= 0) & (ys - r < h)
    return xs, ys, sig, r, zc, act


@functools.lru_cache(maxsize=256)
def _pairs_of(items):
    """Covered (particle, pixel) pairs and box pixels of one pass, from a sample
    of the particles."""
    case = dict(items)
    m = min(case["n"], 40_000)
    p = _particles(case, 12345, "cpu", m)
    pairs = box = 0.0
    for cam in _cameras(case):
        xs, ys, _, r, _, act = _project(case, cam, p)
        bw = ((xs + r).clamp(max=cam["width"]) - (xs - r).clamp(min=0)).clamp(min=0)
        bh = ((ys + r).clamp(max=cam["height"]) - (ys - r).clamp(min=0)).clamp(min=0)
        a = torch.where(r <= R_POINT, torch.ones_like(r), bw * bh)[act]
        k = case["n"] / m
        box += float(a.sum()) * k
        pairs += float(torch.where((r > R_POINT)[act], a * (math.pi / 4), a).sum()) * k
    return pairs, box


def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k != "name"))


def _pairs(case):
    return _pairs_of(_key(case))[0]


def work(case):
    if case["kind"] == "train":
        # forward, the weight gradient, and the update's state in and out
        n = case["n"]
        return {"bytes": 4.0 * (n * (NFEAT + 1) + 7 * NPARAM), "flops": 6.0 * n * NHID * (NFEAT + 1)}
    per = {"f32": 24, "f16": 18, "f16_is": 20, "logh16": 18}[case["attr"]]
    if case["kind"] == "host":
        per = 24
    if case["rgb"]:
        per += 12
    pixels = sum(c["width"] * c["height"] for c in _cameras(case))
    return {"bytes": float(case["n"] * per + 12 * pixels),
            "flops": (11.0 if case["mode"] == "absorb" else 7.0) * _pairs(case)}


def _stored(case, p):
    """The particles as the layout stores them."""
    p = dict(p)
    if case["attr"] == "f32":
        return p
    half = ("h", "I", "s") if case["attr"] == "f16" else ("I", "s")
    for k in half:
        p[k] = p[k].half().double()
    if case["attr"] == "logh16":
        k = torch.round((torch.log2(p["h"].double()) - H_LOG2_MIN) * 4096.0).clamp_(0, 65535)
        p["h"] = torch.exp2(H_LOG2_MIN + k / 4096.0)
    return p


def _emission(case, p):
    if case["rgb"]:
        col = torch.stack([p[k].double() for k in ("cr", "cg", "cb")], 1)
    else:
        pal = torch.from_numpy(scenes.ramp_palette()).to(p["s"].device).double()
        u = p["s"].double().clamp(0.0, 1.0) * (pal.shape[0] - 1)
        k = u.floor().long().clamp(max=pal.shape[0] - 2)
        col = pal[k] + (u - k).unsqueeze(1) * (pal[k + 1] - pal[k])
    return p["I"].double().unsqueeze(1) * col


def _boxes(r, w, h):
    """Groups of particle indices with a common box side, each small enough to
    expand: (indices, side)."""
    side = (2.0 * r).floor().long() + 2
    edges = [2]
    while edges[-1] < max(w, h) * 3:
        edges.append(max(edges[-1] + 1, int(edges[-1] * 1.15)))
    edge = torch.tensor(edges, device=r.device)
    which = torch.bucketize(side, edge)
    for b in torch.unique(which).tolist():
        idx = (which == b).nonzero().squeeze(1)
        k = edges[b] if b < len(edges) else int(side[idx].max())
        per = max(1, int(4e7) // (k * k))
        for a in range(0, idx.numel(), per):
            yield idx[a:a + per], k


def _expand(xs, ys, sig, r, k, w, h):
    """Weights of Eq. 2 over the k x k pixel boxes, flat pixel numbers, and which
    of them are covered pixels of the image."""
    o = torch.arange(k, device=xs.device)
    i = (xs - r - 0.5).ceil().long().unsqueeze(1) + o
    j = (ys - r - 0.5).ceil().long().unsqueeze(1) + o
    dx2 = (i.double() + 0.5 - xs.unsqueeze(1)) ** 2
    dy2 = (j.double() + 0.5 - ys.unsqueeze(1)) ** 2
    s2 = (sig * sig).unsqueeze(1)
    wt = torch.exp(-dy2 / s2).unsqueeze(2) * torch.exp(-dx2 / s2).unsqueeze(1)
    ok = (dx2.unsqueeze(1) + dy2.unsqueeze(2)) <= (r * r).view(-1, 1, 1)
    ok &= ((i >= 0) & (i < w)).unsqueeze(1) & ((j >= 0) & (j < h)).unsqueeze(2)
    pix = j.clamp(0, h - 1).unsqueeze(2) * w + i.clamp(0, w - 1).unsqueeze(1)
    return wt, pix, ok


def _exact_additive(case, cam, p):
    w, h = cam["width"], cam["height"]
    xs, ys, sig, r, _, act = _project(case, cam, p)
    e = _emission(case, p)
    img = [torch.zeros(w * h, dtype=torch.float64, device=xs.device) for _ in range(3)]
    pt = act & (r <= R_POINT)
    inside = pt & (xs >= 0) & (xs < w) & (ys >= 0) & (ys < h)
    pix = ys[inside].floor().long() * w + xs[inside].floor().long()
    for c in range(3):
        img[c].index_add_(0, pix, e[inside, c])
    rest = (act & ~pt).nonzero().squeeze(1)
    for idx, k in _boxes(r[rest], w, h):
        idx = rest[idx]
        wt, pix, ok = _expand(xs[idx], ys[idx], sig[idx], r[idx], k, w, h)
        wt = torch.where(ok, wt, torch.zeros_like(wt))
        for c in range(3):
            img[c].index_add_(0, pix.reshape(-1), (wt * e[idx, c].view(-1, 1, 1)).reshape(-1))
    out = torch.stack(img, 1).reshape(h, w, 3)
    return -torch.expm1(-out) if case["mode"] == "ea" else out


def _exact_absorb(case, cam, p):
    """Front-to-back compositing, a run of depth-ordered particles at a time."""
    w, h = cam["width"], cam["height"]
    xs, ys, sig, r, zc, act = _project(case, cam, p)
    absorb = p["I"].double()                    # A = absorption * brightness * I, both 1
    src = _emission(case, p) / absorb.clamp(min=1e-300).unsqueeze(1)
    ids = (act & (absorb > 0)).nonzero().squeeze(1)
    # the depth key is z_c rounded to FP32, equal keys by index
    ids = ids[torch.sort(zc[ids].float(), stable=True)[1]]
    cum = torch.cumsum(((2.0 * r[ids]).floor() + 2.0) ** 2, 0)
    img = torch.zeros((w * h, 3), dtype=torch.float64, device=xs.device)
    tr = torch.ones(w * h, dtype=torch.float64, device=xs.device)
    at = 0
    while at < ids.numel():
        base = float(cum[at - 1]) if at else 0.0
        end = max(at + 1, int(torch.searchsorted(cum, base + 2.0e8)))
        run_ids = ids[at:end]
        at = end
        pixs, order, taus = [], [], []
        rr = r[run_ids]
        pt = (rr <= R_POINT).nonzero().squeeze(1)
        if pt.numel():
            q = run_ids[pt]
            ok = (xs[q] >= 0) & (xs[q] < w) & (ys[q] >= 0) & (ys[q] < h)
            pixs.append((ys[q].floor().long() * w + xs[q].floor().long())[ok])
            order.append(pt[ok])
            taus.append(absorb[q][ok])
        rest = (rr > R_POINT).nonzero().squeeze(1)
        for sub, k in _boxes(rr[rest], w, h):
            pos = rest[sub]
            q = run_ids[pos]
            wt, pix, ok = _expand(xs[q], ys[q], sig[q], r[q], k, w, h)
            pixs.append(pix[ok])
            order.append(pos.view(-1, 1, 1).expand_as(ok)[ok])
            taus.append((wt * absorb[q].view(-1, 1, 1))[ok])
        pix, pos, tau = torch.cat(pixs), torch.cat(order), torch.cat(taus)
        key, perm = torch.sort(pix * run_ids.numel() + pos)
        pix = key // run_ids.numel()
        pos, tau = pos[perm], tau[perm]
        tot = torch.cumsum(tau, 0)
        first = torch.ones_like(pix, dtype=torch.bool)
        first[1:] = pix[1:] != pix[:-1]
        start = first.nonzero().squeeze(1)
        seg = torch.cumsum(first, 0) - 1
        before = tot - tau
        before -= before[start][seg]
        amount = tr[pix] * torch.exp(-before) * -torch.expm1(-tau)
        sid = run_ids[pos]
        for c in range(3):
            img[:, c].index_add_(0, pix, amount * src[sid, c])
        sums = torch.zeros_like(tr).index_add_(0, pix, tau)
        tr *= torch.exp(-sums)
    return img.reshape(h, w, 3)


def _exact_train(case, seed):
    f = {k: v.double() for k, v in _features(case, seed, "cuda").items()}
    n = case["n"]
    nw = NHID * NFEAT
    w1, b1 = f["theta"][:nw].view(NHID, NFEAT), f["theta"][nw:nw + NHID]
    w2, b2 = f["theta"][nw + NHID:-1], f["theta"][-1]
    z = f["x"] @ w1.T + b1
    hid = z.clamp(min=0.0)
    res = hid @ w2 + b2 - f["t"]
    dy = 2.0 * res / n
    dz = dy.unsqueeze(1) * w2 * (z > 0)
    grad = torch.cat([(dz.T @ f["x"]).reshape(-1), dz.sum(0), hid.T @ dy, dy.sum().view(1)])
    m = 0.9 * f["m"] + 0.1 * grad
    v = 0.999 * f["v"] + 0.001 * grad * grad
    step = lambda q, b: q / (1.0 - b ** 1000)  # noqa: E731
    theta = f["theta"] - 3e-3 * step(m, 0.9) / (torch.sqrt(step(v, 0.999)) + 1e-8)
    return {"grad": grad, "loss": (res * res).mean().view(1), "theta": theta, "m": m, "v": v}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    box = _pairs_of(_key(case))[1]
    if box > EXACT_PAIRS * (0.6 if case["mode"] == "absorb" else 1.0):
        return None
    p = _stored(case, _particles(case, seed, "cuda"))
    cams = _cameras(case)
    fn = _exact_absorb if case["mode"] == "absorb" else _exact_additive
    images = [fn(case, c, p) for c in cams]
    if case["kind"] == "batch":
        return images
    return images[0].cpu().numpy() if case["kind"] == "host" else images[0]
