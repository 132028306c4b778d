"""What a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values.  `listed()` gives the fixed ones, `draw(rng)` one more of the
same ranges, `prepare(case, seed)` what a program holds before the call (scene, cameras,
weights, buffers; made on the GPU from the seed alone), `run(state)` one pass through the
public entry points, `work(case)` the bytes and operations the pass cannot do without and
`exact(case, seed)` the computed outputs in 64 bits by plain torch.

The kinds:
  raster  nrv_rasterize: render + resolve passes, every G-buffer plane written;
  frame   nrv_render_batch: points to RGB;
  pack    nrv_resolve_pack: a key image to the network input, with the Vel2D channels;
  shade   nrv_shade: the U-Net in one of its precisions;
  gated   nrv_gnet_shade: the gated network;
  train   one optimisation step: nrv_train_step (BF16, L1), or forward_train + recon_loss +
          backward (FP32, the L2 reconstruction term) as an autograd loop issues it;
  layer   one convolution's forward, data gradient and weight gradient (BF16).
"""
import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F

from paper_2407_19097_gb300 import nrv

DEV = "cuda:0"
ZNEAR, ZFAR, FOVY = 0.1, 2.0e5, 60.0
PRECS = {"f32": nrv.PREC_F32, "bf16": nrv.PREC_BF16, "fp8": nrv.PREC_FP8, "e4m3": nrv.PREC_FP8_E4M3}
# words read, record stride, network channels of each scene kind
SCENES = {"cube": (3, 4, 3), "grid": (5, 8, 5), "traj": (3, 4, 3), "terrain": (2, 2, 4)}
TERRAIN_VIEWS = "2160x2160 2160x2160 1920x1080 1920x1080 1920x1080 1920x1080 960x540 960x540"


def listed():
    return [
        # the plain method's tiny scene in one small view: the shortest call a viewer makes
        {"name": "raster_cube_1m_512", "kind": "raster", "scene": "cube", "points": 1_000_000, "views": "512x512"},
        # a static vector field at full HD: an ordinary single-view rasterization, 32-byte records
        {"name": "raster_grid_50m_1080p", "kind": "raster", "scene": "grid", "points": 49_836_032, "views": "1920x1080"},
        # a terrain scan in a batch of eight views of uneven sizes (a stereo pair, four monitors,
        # two thumbnails): the largest rasterization
        {"name": "raster_terrain_200m_8v", "kind": "raster", "scene": "terrain", "points": 200_000_000, "views": TERRAIN_VIEWS},
        # the headline: a 350M-point trajectory frame, points to RGB, replayed as a viewer does
        {"name": "frame_traj_350m_1080p", "kind": "frame", "scene": "traj", "points": 350_000_000, "views": "1920x1080", "prec": "bf16"},
        # a resolve with the projected-velocity channels, the input preparation of the vector
        # field's network
        {"name": "pack_vel2d_1080p", "kind": "pack", "points": 8_000_000, "views": "1920x1080", "prec": "bf16"},
        # the FP32 network on the tiny scene's view
        {"name": "shade_f32_512", "kind": "shade", "prec": "f32", "n": 1, "h": 512, "w": 512, "c": 5},
        # two thumbnails of the batch shaded together; 540 rows do not divide by 8
        {"name": "shade_bf16_2x540p", "kind": "shade", "prec": "bf16", "n": 2, "h": 540, "w": 960, "c": 6},
        # the 8-bit network at full HD
        {"name": "shade_fp8_1080p", "kind": "shade", "prec": "fp8", "n": 1, "h": 1080, "w": 1920, "c": 5},
        # the gated form of the network at full HD
        {"name": "gated_1080p", "kind": "gated", "n": 1, "h": 1080, "w": 1920, "c": 5},
        # the training step of the trajectory network: batches of 16 crops of 256 x 256
        {"name": "train_bf16_16x256", "kind": "train", "prec": "bf16", "n": 16, "h": 256, "w": 256, "c": 5},
        # FP32 training (the precision the method was trained in), gradients for an outer optimizer
        {"name": "train_f32_2x256", "kind": "train", "prec": "f32", "n": 2, "h": 256, "w": 256, "c": 5},
        # a concatenating decoder layer of a full-HD frame alone, forward and both gradients
        {"name": "layer_d1a_bf16_540p", "kind": "layer", "layer": 12, "n": 1, "h": 540, "w": 960, "c": 5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["raster", "raster", "frame", "pack", "shade", "shade", "gated", "train", "layer"])
    if kind in ("raster", "frame"):
        scene = rng.choice(sorted(SCENES))
        nv = rng.choice([1, 1, 1, 2, 4, 8])
        views = " ".join("%dx%d" % (_log(rng, 160, 2160), _log(rng, 120, 1600)) for _ in range(nv))
        c = {"kind": kind, "scene": scene, "points": _log(rng, 200_000, 120_000_000), "views": views}
        if kind == "frame":
            c["prec"] = rng.choice(["bf16", "bf16", "fp8", "f32"])
            if c["prec"] == "f32":
                c["points"] = min(c["points"], 2_000_000)
                c["views"] = views.split()[0]
        return c
    if kind == "pack":
        return {"kind": kind, "points": _log(rng, 200_000, 20_000_000), "prec": rng.choice(["f32", "bf16", "e4m3"]),
                "views": "%dx%d" % (_log(rng, 160, 2160), _log(rng, 120, 1600))}
    h, w = _log(rng, 64, 1200), _log(rng, 64, 1920)
    c = {"kind": kind, "n": rng.choice([1, 1, 2, 4]), "h": h, "w": w, "c": rng.randint(3, 8)}
    if kind == "shade":
        c["prec"] = rng.choice(["f32", "bf16", "bf16", "fp8", "e4m3"])
        if c["prec"] == "f32":
            c["h"], c["w"] = min(h, 720), min(w, 1280)
    elif kind == "train":
        c["prec"] = rng.choice(["bf16", "bf16", "f32"])
        c["n"], c["h"], c["w"] = (rng.randint(1, 16) if c["prec"] == "bf16" else rng.randint(1, 3)), _log(rng, 48, 300), _log(rng, 48, 300)
    elif kind == "layer":
        c["layer"] = rng.choice([1, 2, 3, 4, 5, 6, 7, 9, 10, 12, 13, 15, 16])
        lvl = {1: 0, 2: 1, 3: 1, 4: 2, 5: 2, 6: 3, 7: 3, 9: 2, 10: 2, 12: 1, 13: 1, 15: 0, 16: 0}[c["layer"]]
        c["h"], c["w"] = max(16, h >> lvl), max(16, w >> lvl)
    return c


# --------------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["views"].split()]


def _look(eye, target, w, h):
    """View-projection of a camera (+y up, 60 degrees vertical), built in double, rounded once."""
    e, t = np.asarray(eye, np.float64), np.asarray(target, np.float64)
    f = (t - e) / np.linalg.norm(t - e)
    s = np.cross(f, [0.0, 1.0, 0.0])
    s /= np.linalg.norm(s)
    v = np.eye(4)
    v[0, :3], v[1, :3], v[2, :3] = s, np.cross(s, f), -f
    v[:3, 3] = -v[:3, :3] @ e
    k = 1.0 / math.tan(math.radians(FOVY) / 2.0)
    p = np.zeros((4, 4))
    p[0, 0], p[1, 1], p[3, 2] = k * h / w, k, -1.0
    p[2, 2], p[2, 3] = (ZFAR + ZNEAR) / (ZNEAR - ZFAR), 2.0 * ZFAR * ZNEAR / (ZNEAR - ZFAR)
    return SimpleNamespace(viewproj=(p @ v).astype(np.float32).reshape(16), width=w, height=h, znear=ZNEAR, zfar=ZFAR, view=v)


def _cube(n, g):
    return torch.rand((n, 3), device=DEV, generator=g), torch.randn((n, 4), device=DEV, generator=g).view(torch.int32)


def _grid(n, g):
    """Jittered grid (x fastest) with a Rankine vortex about the vertical axis, speed and pressure."""
    m = max(2, round(n ** (1.0 / 3.0)))
    a = torch.arange(m, device=DEV, dtype=torch.float32)
    xyz = torch.rand((m, m, m, 3), device=DEV, generator=g)
    xyz[..., 0] += a.view(1, 1, m)
    xyz[..., 1] += a.view(1, m, 1)
    xyz[..., 2] += a.view(m, 1, 1)
    xyz = xyz.div_(m).view(-1, 3)
    rec = torch.zeros((m ** 3, 8), device=DEV)
    dx, dz = xyz[:, 0] - 0.5, xyz[:, 2] - 0.5
    r2 = (dx * dx + dz * dz).clamp_min_(1e-12)
    om = 10.0 * 0.01 / r2.clamp_min(0.01)
    rec[:, :3] = 0.05 * torch.randn((m ** 3, 3), device=DEV, generator=g)
    rec[:, 0] += om * dz
    rec[:, 2] -= om * dx
    rec[:, 3] = rec[:, :3].square().sum(1).sqrt()
    rec[:, 4] = torch.where(r2 <= 0.01, -0.5 * (2.0 - r2 / 0.01), -0.005 / r2)
    return xyz, rec.view(torch.int32)


def _traj(n, g):
    """Particle-major RK4 trajectories of up to 350 steps through eight Rankine vortex lines."""
    steps = 350 if n >= 3_500_000 else max(20, n // 10_000)
    np_ = max(64, n // steps)
    p = torch.rand((np_, 3), device=DEV, generator=g)
    ctr = torch.rand((8, 3), device=DEV, generator=g)
    ax = F.normalize(torch.randn((8, 3), device=DEV, generator=g), dim=1)
    R = 0.05 + 0.15 * torch.rand(8, device=DEV, generator=g)
    gam = (2.0 * torch.rand(8, device=DEV, generator=g) - 1.0) * R      # circulation / 2 pi
    M = torch.cat([ax, torch.linalg.cross(ax, ctr)], 1)
    off, c2, R2 = (ax * ctr).sum(1), (ctr * ctr).sum(1), R * R

    def vel(q):
        al = q @ ax.T - off
        r2 = (q * q).sum(1, keepdim=True) - 2.0 * (q @ ctr.T) + c2 - al * al
        m = (gam / torch.maximum(r2, R2)) @ M
        return torch.linalg.cross(m[:, :3], q) - m[:, 3:]

    xyz = torch.empty((np_, steps, 3), device=DEV)
    rec = torch.zeros((np_, steps, 4), device=DEV, dtype=torch.int32)
    rec[..., 2] = torch.arange(np_, device=DEV, dtype=torch.int32).view(-1, 1)
    fr = rec.view(torch.float32)
    dt = 0.01
    k1 = vel(p)
    for s in range(steps):
        k2 = vel(p + 0.5 * dt * k1)
        k3 = vel(p + 0.5 * dt * k2)
        k4 = vel(p + dt * k3)
        p = p + (dt / 6.0) * (k1 + 2.0 * (k2 + k3) + k4)
        k1 = vel(p)
        xyz[:, s] = p
        fr[:, s, 0] = (s + 1) * dt
        fr[:, s, 1] = k1.square().sum(1).sqrt()
    return xyz.view(-1, 3), rec.view(-1, 4)


def _terrain(n, g):
    """fBm heightfield over 10 km x 10 km, cells of 64 x 64 points in Morton order; records of
    RGBA bytes by height band and an intensity."""
    nc = max(1, round(math.sqrt(n) / 64))
    side = 64 * nc
    oct_ = [torch.rand((2 ** (o + 2) + 3, 2 ** (o + 2) + 3), device=DEV, generator=g) * 2 - 1 for o in range(6)]
    cx, cz = np.meshgrid(np.arange(nc), np.arange(nc))
    code = np.zeros(nc * nc, np.int64)
    for b in range(16):
        code |= (((cx.ravel() >> b) & 1) << (2 * b)) | (((cz.ravel() >> b) & 1) << (2 * b + 1))
    order = np.argsort(code, kind="stable")
    cells = torch.from_numpy(np.stack([cx.ravel()[order], cz.ravel()[order]], 1)).to(DEV)
    xyz = torch.empty((nc * nc, 64, 64, 3), device=DEV)
    rec = torch.empty((nc * nc, 64, 64, 2), device=DEV, dtype=torch.int32)
    a = torch.arange(64, device=DEV, dtype=torch.float32)
    band = torch.tensor([[40, 70, 160], [194, 178, 128], [80, 140, 60], [120, 110, 100], [240, 240, 245]], dtype=torch.int64)
    pal = (band[:, 0] | (band[:, 1] << 8) | (band[:, 2] << 16) | (255 << 24)).to(torch.int32).to(DEV)
    edges = torch.tensor([-150.0, 0.0, 150.0, 350.0], device=DEV)
    for k in range(0, nc * nc, 4096):
        c = cells[k:k + 4096].float() * 64.0
        m = c.shape[0]
        x = (c[:, 0].view(m, 1, 1) + a.view(1, 1, 64) + torch.rand((m, 64, 64), device=DEV, generator=g)) * (1.0e4 / side)
        z = (c[:, 1].view(m, 1, 1) + a.view(1, 64, 1) + torch.rand((m, 64, 64), device=DEV, generator=g)) * (1.0e4 / side)
        hgt = torch.zeros_like(x)
        for o, lat in enumerate(oct_):
            u, v = x * (2.0 ** o / 2500.0), z * (2.0 ** o / 2500.0)
            iu, iv = u.floor(), v.floor()
            fu, fv = u - iu, v - iv
            fu, fv = fu * fu * (3 - 2 * fu), fv * fv * (3 - 2 * fv)
            at = iv.int() * lat.shape[1] + iu.int()
            f = lat.view(-1)
            top = torch.lerp(f[at], f[at + 1], fu)
            bot = torch.lerp(f[at + lat.shape[1]], f[at + lat.shape[1] + 1], fu)
            hgt += (400.0 * 0.5 ** o) * torch.lerp(top, bot, fv)
        xyz[k:k + m, ..., 0], xyz[k:k + m, ..., 1], xyz[k:k + m, ..., 2] = x, hgt, z
        rec[k:k + m, ..., 0] = pal[torch.bucketize(hgt, edges)]
        rec[k:k + m, ..., 1] = torch.rand((m, 64, 64), device=DEV, generator=g).view(torch.int32)
    return xyz.view(-1, 3), rec.view(-1, 2)


def _cameras(case, scene, lo, hi, seed):
    c, diag = 0.5 * (lo + hi), float(np.linalg.norm(hi - lo))
    r = np.random.default_rng(seed)
    out = []
    for i, (w, h) in enumerate(_sizes(case)):
        if scene == "terrain":       # orbits over the field; the first two views are a stereo pair
            if i != 1:
                th, rad, up = 2 * math.pi * r.random(), 1e4 * (0.55 + 0.25 * r.random()), 1e4 * (0.25 + 0.2 * r.random())
            eye = c + np.array([rad * math.cos(th), up, rad * math.sin(th)])
            if i == 1:
                eye = eye + 0.065 * np.array([math.sin(th), 0.0, -math.cos(th)])
        elif i == 0:                 # the whole scene in the vertical field of view
            eye = c + np.array([0.05 * diag * r.random(), 0.0, 0.5 * diag / math.sin(math.radians(FOVY) / 2.0)])
        else:                        # the training hemisphere
            th, ph = 2 * math.pi * r.random(), math.pi * (1 + 6 * r.random()) / 16
            eye = c + 0.75 * diag * np.array([math.sin(ph) * math.cos(th), math.cos(ph), math.sin(ph) * math.sin(th)])
        out.append(_look(eye, c, w, h))
    return out


def _channels(scene, rec):
    """Network channels (word, fmt, comp, 1/std, -mean/std) over a sample of the records."""
    s = rec[:: max(1, rec.shape[0] // 4_000_000)]
    spec = {"cube": [(0, nrv.NRV_F32, 0), (1, nrv.NRV_F32, 0), (2, nrv.NRV_F32, 0)],
            "grid": [(j, nrv.NRV_F32, 0) for j in range(5)],
            "traj": [(0, nrv.NRV_F32, 0), (1, nrv.NRV_F32, 0), (2, nrv.NRV_U32, 0)],
            "terrain": [(0, nrv.NRV_U8X4, 0), (0, nrv.NRV_U8X4, 1), (0, nrv.NRV_U8X4, 2), (1, nrv.NRV_F32, 0)]}[scene]
    out = []
    for w, f, b in spec:
        col = s[:, w].contiguous()
        v = col.view(torch.float32).double() if f == nrv.NRV_F32 else col.double() if f == nrv.NRV_U32 else ((col >> (8 * b)) & 255).double()
        sd = float(v.std().clamp_min(1e-6))
        out.append(SimpleNamespace(word=w, fmt=f, comp=b, scale=float(np.float32(1 / sd)), offset=float(np.float32(-float(v.mean()) / sd))))
    return out


def _scene(case, seed):
    kind = case.get("scene", "grid")
    xyz, rec = {"cube": _cube, "grid": _grid, "traj": _traj, "terrain": _terrain}[kind](case["points"], _gen(seed))
    lo, hi = (t.double().cpu().numpy() for t in (xyz.min(0).values, xyz.max(0).values))
    views = _cameras(case, kind, lo, hi, seed)
    corners = np.array([[x, y, z, 1.0] for x in (lo[0], hi[0]) for y in (lo[1], hi[1]) for z in (lo[2], hi[2])])
    d = -(corners @ views[0].view[2])
    dn = max(float(d.min()), ZNEAR)
    ds = 1.0 / (max(float(d.max()), dn + 1e-6) - dn)
    return SimpleNamespace(kind=kind, xyz=xyz, rec=rec, views=views, channels=_channels(kind, rec),
                           depth=(float(np.float32(ds)), float(np.float32(-dn * ds))))


# The fixed U-Net: name, kind (0 3x3, 1 transposed, 2 head), input and output channels.
def _unet_layers(c):
    return [("e0a", 0, c, 16), ("e0b", 0, 16, 16), ("e1a", 0, 16, 32), ("e1b", 0, 32, 32), ("e2a", 0, 32, 64), ("e2b", 0, 64, 64),
            ("e3a", 0, 64, 128), ("e3b", 0, 128, 128), ("up3", 1, 128, 64), ("d2a", 0, 128, 64), ("d2b", 0, 64, 64), ("up2", 1, 64, 32),
            ("d1a", 0, 64, 32), ("d1b", 0, 32, 32), ("up1", 1, 32, 16), ("d0a", 0, 32, 16), ("d0b", 0, 16, 16), ("head", 2, 16, 3)]


def _gated_layers(c):
    return [("inj", 2, c, c), ("e0", 3, c, 16), ("e1", 3, 16 + c, 32), ("e2", 3, 32 + c, 64), ("e3", 3, 64 + c, 128), ("up2", 1, 128, 64),
            ("d2", 3, 128, 64), ("up1", 1, 64, 32), ("d1", 3, 64, 32), ("up0", 1, 32, 16), ("d0", 3, 32, 16), ("head", 2, 16, 3)]


def _shapes(kind, ci, co):
    if kind == 1:
        return [(ci, co, 2, 2), (co,)]
    one = [(co, ci, 3, 3) if kind != 2 else (co, ci), (co,)]
    return one + one if kind == 3 else one


def _params(layers, seed):
    """Xavier-uniform weights with small biases, the flat FP32 vector the library exchanges."""
    g, out = _gen(seed + 77), []
    for _, kind, ci, co in layers:
        for s in _shapes(kind, ci, co):
            u = 2.0 * torch.rand(s, device=DEV, generator=g) - 1.0
            out.append((u * (0.05 if len(s) == 1 else math.sqrt(6.0 / ((ci + co) * {0: 9, 1: 4, 2: 1, 3: 9}[kind])))).view(-1))
    return torch.cat(out)


def _split(layers, flat):
    out, o = {}, 0
    for name, kind, ci, co in layers:
        t = []
        for s in _shapes(kind, ci, co):
            n = math.prod(s)
            t.append(flat[o:o + n].view(s))
            o += n
        out[name] = t
    return out


def _netin(case, seed):
    """A packed G-buffer [n][Hn][Wn][8]: smooth normalised channels with per-point noise, depth,
    coverage over about three quarters of the view; zeros where empty, in the padding and in the
    channels past c."""
    g = _gen(seed + 5)
    n, h, w, c = case["n"], case["h"], case["w"], case["c"]
    hn, wn = (h + 7) // 8 * 8, (w + 7) // 8 * 8
    coarse = torch.randn((n, c + 1, h // 24 + 3, w // 24 + 3), device=DEV, generator=g)
    f = F.interpolate(coarse, size=(h, w), mode="bicubic", align_corners=True)
    x = torch.zeros((n, hn, wn, 8), device=DEV)
    v = f[:, :c].permute(0, 2, 3, 1) + 0.15 * torch.randn((n, h, w, c), device=DEV, generator=g)
    v[..., c - 2] = (0.5 + 0.2 * v[..., c - 2]).clamp(0, 1)
    v[..., c - 1] = 1.0
    x[:, :h, :w, :c] = v * (f[:, c] > -0.6).unsqueeze(-1)
    return x


def _target(case, seed):
    g = _gen(seed + 9)
    coarse = torch.rand((case["n"], 3, case["h"] // 16 + 2, case["w"] // 16 + 2), device=DEV, generator=g)
    return F.interpolate(coarse, size=(case["h"], case["w"]), mode="bilinear", align_corners=True).permute(0, 2, 3, 1).contiguous()


def _layer_tensors(case, seed):
    """Inputs of one layer: ReLU outputs, the gradient at its output; BF16 NHWC."""
    _, _, ci, co = _unet_layers(case["c"])[case["layer"]]
    g = _gen(seed + 13)
    n, h, w = case["n"], case["h"], case["w"]
    cat = case["layer"] in (9, 12, 15)
    x1 = torch.randn((n, h, w, ci // 2 if cat else ci), device=DEV, generator=g)
    x2 = torch.randn(x1.shape, device=DEV, generator=g).relu_().bfloat16() if cat else None
    dy = (1e-3 * torch.randn((n, h, w, co), device=DEV, generator=g)).bfloat16()
    x1 = (x1 if cat else x1.relu_()).bfloat16()      # the upsampled half has no activation
    mask = None if cat else x1
    return x1, x2, dy, mask


# --------------------------------------------------------------------------- prepare and run

def prepare(case, seed):
    kind, s = case["kind"], SimpleNamespace(case=case, kind=case["kind"])
    if kind in ("raster", "frame", "pack"):
        sc = _scene(case, seed)
        k, _, nch = SCENES[sc.kind]
        s.views, s.scene = sc.views, nrv.Scene(sc.xyz, sc.rec, k)
        if kind != "frame":
            s.key = [torch.empty((v.height, v.width), dtype=torch.int64, device=DEV) for v in s.views]
        if kind == "raster":
            s.depth = [torch.empty_like(t, dtype=torch.int32) for t in s.key]
            s.mask = [torch.empty_like(t, dtype=torch.uint8) for t in s.key]
            s.gattr = [torch.empty((k,) + tuple(t.shape), dtype=torch.int32, device=DEV) for t in s.key]
            return s
        s.prec = PRECS[case["prec"]]
        if kind == "pack":
            s.desc, _ = _pack_desc(sc)
            nrv.rasterize(s.scene, s.views, s.key)
            v = s.views[0]
            dt, c = {"f32": (torch.float32, 8), "bf16": (torch.bfloat16, 8), "e4m3": (torch.uint8, 16)}[case["prec"]]
            s.netin = torch.empty(((v.height + 7) // 8 * 8, (v.width + 7) // 8 * 8, c), dtype=dt, device=DEV)
            return s
        s.desc = nrv.make_pack_desc(sc.channels, *sc.depth)
        s.net = nrv.Net(nch + 2)
        s.net.set_params(_params(_unet_layers(nch + 2), seed))
        if s.prec == nrv.PREC_FP8:
            s.net.calibrate(_netin({"n": 1, "h": 256, "w": 256, "c": nch + 2}, seed).bfloat16(), 1, 256, 256)
        s.rgb = [torch.empty((v.height, v.width, 3), device=DEV) for v in s.views]
        return s
    c, n, h, w = case["c"], case["n"], case["h"], case["w"]
    if kind == "gated":
        s.net = nrv.GatedNet(c)
        s.net.set_params(_params(_gated_layers(c), seed))
    else:
        s.net, s.params = nrv.Net(c), _params(_unet_layers(c), seed)
        s.net.set_params(s.params)
    if kind == "layer":
        s.x1, s.x2, s.dy, s.mask = _layer_tensors(case, seed)
        s.y = torch.empty_like(s.dy)
        s.dx = torch.empty(s.x1.shape[:3] + (_unet_layers(c)[case["layer"]][2],), dtype=torch.bfloat16, device=DEV)
        s.grad = torch.zeros_like(s.params)
        return s
    s.netin = _netin(case, seed)
    if kind in ("shade", "gated"):
        s.prec = PRECS[case.get("prec", "bf16")]
        s.rgb = torch.empty((n, h, w, 3), device=DEV)
        if case.get("prec", "bf16") != "f32":
            bf = s.netin.bfloat16()
            if s.prec in (nrv.PREC_FP8, nrv.PREC_FP8_E4M3):
                s.net.calibrate(bf, n, h, w)
            if s.prec == nrv.PREC_FP8_E4M3:      # 16 stored channels, codes at the input's scale
                q = torch.zeros(s.netin.shape[:3] + (16,), device=DEV)
                q[..., :8] = s.netin / s.net.act_scales()[0]
                bf = q.clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
            s.netin = bf
        return s
    s.prec, s.target = PRECS[case["prec"]], _target(case, seed)
    s.grad, s.loss = torch.zeros_like(s.params), torch.zeros(1, device=DEV)
    if s.prec == nrv.PREC_BF16:
        s.netin = s.netin.bfloat16()
        g = _gen(seed + 21)                      # moments of a run under way
        s.m = 1e-3 * torch.randn(s.params.shape, device=DEV, generator=g)
        s.v = 1e-4 * (0.5 + torch.rand(s.params.shape, device=DEV, generator=g))
        s.step = 200
    else:
        s.rgb = torch.empty((n, h, w, 3), device=DEV)
        s.drgb = torch.empty_like(s.rgb)
    return s


def _pack_desc(sc):
    """Velocity, its projection onto the view (Vel2D) and pressure: six channels."""
    ch = [SimpleNamespace(word=0, fmt=f, comp=0, scale=sc_, offset=0.0) for f, sc_ in
          ((nrv.NRV_VEL2D_X, 1e-3), (nrv.NRV_VEL2D_Y, 1e-3), (nrv.NRV_VEL2D_ANGLE, 0.5), (nrv.NRV_VEL2D_MAG, 1e-3))]
    ch += [sc.channels[3], sc.channels[4]]
    return nrv.make_pack_desc(ch, *sc.depth), ch


def run(s):
    case, kind = s.case, s.kind
    if kind == "raster":
        nrv.rasterize(s.scene, s.views, s.key, s.depth, s.mask, s.gattr)
        return {"key": s.key, "depth": s.depth, "mask": s.mask, "attr": s.gattr}
    if kind == "frame":
        nrv.render_batch(s.scene, s.net, s.desc, s.views, s.rgb, s.prec)
        return s.rgb
    if kind == "pack":
        nrv.resolve_pack(s.scene, s.views[0], s.key[0], s.desc, s.prec, s.netin)
        return s.netin
    n, h, w = case["n"], case["h"], case["w"]
    if kind == "shade":
        s.net.shade(s.netin, n, h, w, s.prec, s.rgb)
        return s.rgb
    if kind == "gated":
        s.net.shade(s.netin, n, h, w, s.rgb)
        return s.rgb
    if kind == "layer":
        l = case["layer"]
        _run_layer(s, l, n, h, w)
        s.net.layer_dgrad(l, s.dy, s.mask, n, h, w, nrv.PREC_BF16, s.dx)
        s.net.layer_wgrad(l, s.dy, s.x1, s.x2, n, h, w, nrv.PREC_BF16, s.grad)
        return {"y": s.y, "dx": s.dx, "grad": s.grad}
    if s.prec == nrv.PREC_BF16:
        s.net.train_step(s.params, s.grad, s.m, s.v, s.step, 1e-4, s.netin, s.target, n, h, w, s.prec, s.loss)
        s.step += 1
        return {"loss": s.loss, "grad": s.grad, "params": s.params, "m": s.m, "v": s.v}
    s.net.forward_train(s.netin, n, h, w, s.prec, s.rgb)
    nrv.recon_loss(s.rgb, s.target, (0.0, 1.0, 0.0), s.loss, s.drgb)
    s.net.backward(s.drgb, s.grad)
    return {"rgb": s.rgb, "loss": s.loss, "drgb": s.drgb, "grad": s.grad}


def _run_layer(s, l, n, h, w):
    """nrv_net_run_layer through the binding's C signature (it has no method on Net)."""
    nrv.check(nrv.lib().nrv_net_run_layer(s.net.h, l, s.x1.data_ptr(), None if s.x2 is None else s.x2.data_ptr(), n, h, w,
                                          nrv.PREC_BF16, s.y.data_ptr(), torch.cuda.current_stream().cuda_stream))


# --------------------------------------------------------------------------- work

def _unet_work(case, es):
    """Bytes and FLOPs of one forward: input, output and weights; every layer's products."""
    px = case["n"] * ((case["h"] + 7) // 8 * 8) * ((case["w"] + 7) // 8 * 8)
    lv = {"e0": 0, "e1": 1, "e2": 2, "e3": 3, "d2": 2, "d1": 1, "d0": 0}
    fl = sum(2.0 * ci * co * (9 * px / 4 ** lv[nm[:2]] if k == 0 else 4 * px / 4 ** int(nm[2]) if k == 1 else px)
             for nm, k, ci, co in _unet_layers(case["c"]))
    par = sum(math.prod(s) for _, k, ci, co in _unet_layers(case["c"]) for s in _shapes(k, ci, co))
    return px * case["c"] * es + case["n"] * case["h"] * case["w"] * 12 + par * 4, fl, par


def work(case):
    kind = case["kind"]
    if kind in ("raster", "frame", "pack"):
        px = sum(w * h for w, h in _sizes(case))
        k, stride, nch = SCENES[case.get("scene", "grid")]
        if kind == "raster":
            return {"bytes": 12.0 * case["points"] + px * (8 + 4 + 1 + 8 * k), "flops": 0}
        if kind == "pack":
            return {"bytes": px * (8.0 + 32 + 12 + {"f32": 32, "bf16": 16, "e4m3": 16}[case["prec"]]), "flops": 60.0 * px}
        fl = sum(_unet_work({"n": 1, "w": w, "h": h, "c": nch + 2}, 2)[1] for w, h in _sizes(case))
        return {"bytes": 12.0 * case["points"] + px * (4.0 * k + 12), "flops": fl}
    if kind == "layer":
        _, _, ci, co = _unet_layers(case["c"])[case["layer"]]
        px = case["n"] * case["h"] * case["w"]
        # forward: x in, y out; data gradient: dy (and the mask) in, dx out; weight gradient: x, dy in
        return {"bytes": 2.0 * px * ((ci + co) + (co + ci + (0 if case["layer"] in (9, 12, 15) else ci)) + (ci + co)) + 36.0 * ci * co,
                "flops": 3 * 18.0 * px * ci * co}
    if kind == "gated":
        px = case["n"] * ((case["h"] + 7) // 8 * 8) * ((case["w"] + 7) // 8 * 8)
        lv = {"in": 0, "e0": 0, "e1": 1, "e2": 2, "e3": 3, "d2": 2, "d1": 1, "d0": 0, "he": 0}
        fl = sum(2.0 * ci * co * (18 * px / 4 ** lv[nm[:2]] if k == 3 else 4 * px / 4 ** (int(nm[2]) + 1) if k == 1 else px)
                 for nm, k, ci, co in _gated_layers(case["c"]))
        par = sum(math.prod(s) for _, k, ci, co in _gated_layers(case["c"]) for s in _shapes(k, ci, co))
        return {"bytes": px * case["c"] * 2.0 + case["n"] * case["h"] * case["w"] * 12 + par * 4, "flops": fl}
    b, fl, par = _unet_work(case, {"f32": 4, "bf16": 2, "fp8": 2, "e4m3": 1}[case["prec"]])
    if kind == "shade":
        return {"bytes": b, "flops": fl}
    # training: forward, data and weight gradients of every layer but the first's data gradient;
    # target read, parameters, moments and gradient read and written
    return {"bytes": b + case["n"] * case["h"] * case["w"] * 12.0 + 6.0 * 4 * par, "flops": 3 * fl}


# --------------------------------------------------------------------------- 64-bit results

def _unet64(x, p):
    """x [n][c][H][W] double -> [n][3][H][W]."""
    cv = lambda t, nm: F.relu(F.conv2d(t, p[nm][0], p[nm][1], padding=1))
    up = lambda t, nm: F.conv_transpose2d(t, p[nm][0], p[nm][1], stride=2)
    e0 = cv(cv(x, "e0a"), "e0b")
    e1 = cv(cv(F.avg_pool2d(e0, 2), "e1a"), "e1b")
    e2 = cv(cv(F.avg_pool2d(e1, 2), "e2a"), "e2b")
    e3 = cv(cv(F.avg_pool2d(e2, 2), "e3a"), "e3b")
    d2 = cv(cv(torch.cat([up(e3, "up3"), e2], 1), "d2a"), "d2b")
    d1 = cv(cv(torch.cat([up(d2, "up2"), e1], 1), "d1a"), "d1b")
    d0 = cv(cv(torch.cat([up(d1, "up1"), e0], 1), "d0a"), "d0b")
    return F.conv2d(d0, p["head"][0][:, :, None, None], p["head"][1])


def _gated64(x, p):
    def gt(t, nm):
        wf, bf, wg, bg = p[nm]
        return F.elu(F.conv2d(t, wf, bf, padding=1)) * torch.sigmoid(F.conv2d(t, wg, bg, padding=1))
    g = [F.conv2d(x, p["inj"][0][:, :, None, None], p["inj"][1])]
    for _ in range(3):
        g.append(F.avg_pool2d(g[-1], 2))
    e = [gt(g[0], "e0")]
    for l in (1, 2, 3):
        e.append(gt(torch.cat([F.avg_pool2d(e[l - 1], 2), g[l]], 1), "e%d" % l))
    d = e[3]
    for l in (2, 1, 0):
        d = gt(torch.cat([F.conv_transpose2d(d, p["up%d" % l][0], p["up%d" % l][1], stride=2), e[l]], 1), "d%d" % l)
    return F.conv2d(d, p["head"][0][:, :, None, None], p["head"][1])


def _visible(sc, v):
    """Key image of one view by the fixed FP32 sequence, every operation rounded on its own."""
    m = [float(t) for t in v.viewproj]
    n, npx = sc.xyz.shape[0], v.width * v.height
    key = torch.full((npx,), 2 ** 63 - 1, dtype=torch.int64, device=DEV)
    hw, hh = 0.5 * v.width, 0.5 * v.height
    for i in range(0, n, 25_000_000):
        x, y, z = (t.contiguous() for t in sc.xyz[i:i + 25_000_000].unbind(1))
        row = lambda r: ((x * m[4 * r] + y * m[4 * r + 1]) + z * m[4 * r + 2]) + m[4 * r + 3]
        w = row(3)
        sx, sy = (row(0) / w + 1.0) * hw, (1.0 - row(1) / w) * hh
        ok = (w >= ZNEAR) & (w <= np.float32(ZFAR)) & (sx >= 0) & (sx < v.width) & (sy >= 0) & (sy < v.height)
        at = ok.nonzero().view(-1)
        px = sy[at].long() * v.width + sx[at].long()
        key.scatter_reduce_(0, px, (w[at].view(torch.int32).long() << 32) | (at + i), "amin")
    return key


def _packed64(sc, v, key, channels):
    """Packed network input [8][Hn][Wn] in double from a key image."""
    hit = (key != 2 ** 63 - 1).nonzero().view(-1)
    idx, w = key[hit] & 0xFFFFFFFF, (key[hit] >> 32).int().view(torch.float32).double()
    rec, p = sc.rec[idx], torch.cat([sc.xyz[idx].double(), torch.ones((idx.numel(), 1), device=DEV, dtype=torch.float64)], 1)
    M = torch.tensor(v.viewproj.reshape(4, 4), device=DEV, dtype=torch.float64)
    c = p @ M.T
    out = torch.zeros((8, v.width * v.height), device=DEV, dtype=torch.float64)
    f32 = lambda t: t.contiguous().view(torch.float32).double()
    for j, ch in enumerate(channels):
        if nrv.NRV_VEL2D_X <= ch.fmt <= nrv.NRV_VEL2D_MAG:
            mv = torch.stack([f32(rec[:, ch.word + k]) for k in range(3)], 1) @ M[:, :3].T
            vx = 0.5 * v.width * (mv[:, 0] - c[:, 0] / c[:, 3] * mv[:, 3]) / c[:, 3]
            vy = -0.5 * v.height * (mv[:, 1] - c[:, 1] / c[:, 3] * mv[:, 3]) / c[:, 3]
            val = {nrv.NRV_VEL2D_X: vx, nrv.NRV_VEL2D_Y: vy, nrv.NRV_VEL2D_ANGLE: torch.atan2(vy, vx)}.get(ch.fmt, torch.hypot(vx, vy))
        else:
            col = rec[:, ch.word]
            val = f32(col) if ch.fmt == nrv.NRV_F32 else col.double() if ch.fmt == nrv.NRV_U32 else ((col >> (8 * ch.comp)) & 255).double()
        out[j, hit] = val * ch.scale + ch.offset
    out[len(channels), hit] = w * sc.depth[0] + sc.depth[1]
    out[len(channels) + 1, hit] = 1.0
    return F.pad(out.view(8, v.height, v.width), (0, -v.width % 8, 0, -v.height % 8))


def exact(case, seed):
    kind = case["kind"]
    if kind == "raster":
        return None                              # whole numbers and copied bits only
    if kind in ("frame", "pack"):
        sc = _scene(case, seed)
        if kind == "pack":
            if case["prec"] == "e4m3":
                return None                      # bytes
            return _packed64(sc, sc.views[0], _visible(sc, sc.views[0]), _pack_desc(sc)[1]).permute(1, 2, 0).contiguous()
        c = SCENES[sc.kind][2] + 2
        p = _split(_unet_layers(c), _params(_unet_layers(c), seed).double())
        with torch.no_grad():
            return [_unet64(_packed64(sc, v, _visible(sc, v), sc.channels)[None, :c], p)[0, :, :v.height, :v.width].permute(1, 2, 0).contiguous()
                    for v in sc.views]
    c, h, w = case["c"], case["h"], case["w"]
    if kind == "layer":
        nm, _, ci, co = _unet_layers(c)[case["layer"]]
        x1, x2, dy, mask = _layer_tensors(case, seed)
        par = _params(_unet_layers(c), seed)
        wt, b = (t.double() for t in _split(_unet_layers(c), par)[nm])
        nchw = lambda t: t.double().permute(0, 3, 1, 2)
        x, g = nchw(x1) if x2 is None else torch.cat([nchw(x1), nchw(x2)], 1), nchw(dy)
        dx = F.conv_transpose2d(g, wt, padding=1)
        if mask is not None:
            dx = dx * (nchw(mask) > 0)
        grad = torch.zeros_like(par, dtype=torch.float64)
        gw, gb = _split(_unet_layers(c), grad)[nm]
        xp = F.pad(x, (1, 1, 1, 1))
        for t in range(9):
            gw[:, :, t // 3, t % 3] = torch.einsum("nohw,nchw->oc", g, xp[:, :, t // 3:t // 3 + h, t % 3:t % 3 + w])
        gb.copy_(g.sum((0, 2, 3)))
        nhwc = lambda t: t.permute(0, 2, 3, 1).contiguous()
        return {"y": nhwc(F.relu(F.conv2d(x, wt, b, padding=1))), "dx": nhwc(dx), "grad": grad}
    x = _netin(case, seed)[..., :c].permute(0, 3, 1, 2).double()
    crop = lambda t: t[:, :, :h, :w].permute(0, 2, 3, 1).contiguous()
    if kind in ("shade", "gated"):
        ls, net = (_gated_layers(c), _gated64) if kind == "gated" else (_unet_layers(c), _unet64)
        p = _split(ls, _params(ls, seed).double())
        with torch.no_grad():
            return torch.cat([crop(net(x[i:i + 1], p)) for i in range(case["n"])])
    # training: the gradient by autograd, one image at a time
    flat = _params(_unet_layers(c), seed).double().requires_grad_()
    tgt, loss, rgb = _target(case, seed).double(), 0.0, []
    bf = case["prec"] == "bf16"
    for i in range(case["n"]):
        y = crop(_unet64(x[i:i + 1], _split(_unet_layers(c), flat)))
        part = ((y - tgt[i:i + 1]).abs() if bf else (y - tgt[i:i + 1]).square()).sum() / tgt.numel()
        part.backward()
        loss += float(part)
        rgb.append(y.detach())
    g, one = flat.grad, torch.tensor([loss], dtype=torch.float64)
    if not bf:
        rgb = torch.cat(rgb)
        return {"rgb": rgb, "loss": one, "drgb": 2.0 * (rgb - tgt) / tgt.numel(), "grad": g}
    s = prepare(case, seed)                      # the moments a run is given
    m = 0.9 * s.m.double() + 0.1 * g
    v = 0.999 * s.v.double() + 0.001 * g * g
    par = flat.detach() - 1e-4 * (m / (1 - 0.9 ** 200)) / ((v / (1 - 0.999 ** 200)).sqrt() + 1e-8)
    return {"loss": one, "grad": g, "params": par, "m": m, "v": v}
