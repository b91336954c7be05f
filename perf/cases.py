"""Performance cases: what a user of this library has it do, over the sizes it is used at.

A case is one call (or one short sequence of calls) of the public Python API on a synthetic scene:
UV spheres, triangle soups and overlapping transparent spheres of the sizes the benchmark and the
tests run, with seeded vertex noise, textures, cameras and target images.

`exact` restates the method in plain torch: float32 where the method fixes its rounding (signs,
projection, coverage, depth, UV, footprint position), float64 for everything after that.
"""
import math

import torch

import paper_2404_09758_gb300 as sge

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
F32, F64, I64 = torch.float32, torch.float64, torch.int64
EPS_POS, EPS_TEX, NEAR, LAYERS = 1e-3, 1.0 / 255.0, 0.1, 4
UNLIT, LAMBERT, GGX, TRANSPARENT = 0, 1, 2, 3
LIGHT = tuple(x / math.sqrt(0.3 ** 2 + 0.6 ** 2 + 0.74 ** 2) for x in (0.3, 0.6, 0.74))
ITER, T_ADAM = 3, 100  # a loop under way: its iteration index and Adam's step number


def listed():
    """Sizes: the benchmark's workloads and the test configurations."""
    return [
        # one iteration's estimate of the plain configuration: the smallest call, launches count
        dict(name="plain_2k_r256_1x1", call="estimate", scene="sphere", shading=UNLIT, lon=32, lat=32, w=256, h=256,
             tex=256, maps=0, views=1, pairs=1, nearest=False),
        # a soup of independent coloured triangles fitted to one image
        dict(name="soup_10k_r512_1x8", call="estimate", scene="soup", shading=UNLIT, lon=10240, lat=1, w=512, h=512,
             tex=10240, maps=0, views=1, pairs=8, nearest=False),
        # the benchmark's batched estimate
        dict(name="unlit_8k_r512_8x64", call="estimate", scene="sphere", shading=UNLIT, lon=64, lat=64, w=512, h=512,
             tex=512, maps=0, views=8, pairs=64, nearest=False),
        # the paper's own texel footprint (nearest), a ragged image and texture
        dict(name="nearest_8k_r501_4x16", call="estimate", scene="sphere", shading=UNLIT, lon=67, lat=61, w=501,
             h=397, tex=509, maps=0, views=4, pairs=16, nearest=True),
        # a whole optimiser iteration from host buffers: theta and targets in, estimate, Adam, theta and loss out
        dict(name="iterate_8k_r512_8x8", call="iterate", scene="sphere", shading=UNLIT, lon=64, lat=64, w=512, h=512,
             tex=512, maps=0, views=8, pairs=8, nearest=False),
        # the autograd form, forward and backward: RGBA albedo and normal map, Lambert
        dict(name="lambert_32k_r1024_8x16", call="autograd", scene="sphere", shading=LAMBERT, lon=128, lat=128, w=1024,
             h=1024, tex=1024, maps=1024, views=8, pairs=16, nearest=False),
        # lit maps of two sizes, a ragged image, few pairs
        dict(name="lambert_5k_r413_3x5", call="estimate", scene="sphere", shading=LAMBERT, lon=53, lat=47, w=413,
             h=311, tex=384, maps=200, views=3, pairs=5, nearest=False),
        # the scale configuration: a million triangles, four 2048^2 maps, GGX
        dict(name="ggx_1m_r2048_4x4", call="estimate", scene="sphere", shading=GGX, lon=1024, lat=512, w=2048, h=2048,
             tex=2048, maps=2048, views=4, pairs=4, nearest=False),
        # assets of uneven sizes in one batched call
        dict(name="batch_8assets_r512_4x8", call="batch", scene="sphere", shading=UNLIT, lon=1000, lat=200000, w=512,
             h=512, tex=1024, maps=8, views=4, pairs=8, nearest=False),
        # transparent geometry: three overlapping spheres, deep ID buffers
        dict(name="transparent_6k_r512_8x16", call="estimate", scene="spheres", shading=TRANSPARENT, lon=32, lat=32,
             w=512, h=512, tex=512, maps=0, views=8, pairs=16, nearest=False),
        # the forward pass alone: ID, UV and colour buffers of every view
        dict(name="render_32k_r1024_4v", call="render", scene="sphere", shading=LAMBERT, lon=128, lat=128, w=1024,
             h=1024, tex=1024, maps=1024, views=4, pairs=1, nearest=False),
        # the descent step alone at the scale configuration's 52 million parameters (Adam)
        dict(name="adam_52m", call="step", scene="sphere", shading=GGX, lon=1024, lat=512, w=64, h=64, tex=2048,
             maps=2048, views=1, pairs=16, nearest=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["estimate"] * 5 + ["autograd", "iterate", "batch", "render", "step"])
    scene = rng.choice(["sphere", "sphere", "soup", "spheres"]) if call == "estimate" else "sphere"
    shading = {"soup": UNLIT, "spheres": TRANSPARENT}.get(scene, rng.choice([UNLIT, LAMBERT, GGX]))
    if call in ("batch", "iterate"):
        shading = UNLIT
    w, h = _log_int(rng, 64, 1024), _log_int(rng, 64, 1024)
    tex = _log_int(rng, 32, 1024)
    maps = rng.choice([tex, _log_int(rng, 32, 1024)]) if shading in (LAMBERT, GGX) else 0
    lat = max(4, int(math.sqrt(_log_int(rng, 500, 20000 if scene == "spheres" else 200000) / 4)))
    lon = 2 * lat
    if scene == "soup":
        lon, lat = _log_int(rng, 1000, 100000), 1
        tex = lon
    views, pairs = 1 if scene == "soup" else rng.randint(1, 8), _log_int(rng, 1, 64)
    if call == "batch":
        lon, lat, maps, views = _log_int(rng, 300, 3000), _log_int(rng, 10000, 100000), rng.randint(2, 8), rng.randint(1, 4)
        pairs = _log_int(rng, 1, 8)
    if call in ("render", "step"):
        pairs = 1
    while w * h * views * pairs > (1 << 24) and pairs > 1:
        pairs //= 2
    return dict(call=call, scene=scene, shading=shading, lon=lon, lat=lat, w=w, h=h, tex=tex, maps=maps, views=views,
                pairs=pairs, nearest=call == "estimate" and scene != "soup" and rng.random() < 0.25)


# ------------------------------------------------------------------------------------ inputs
def _gen(seed, salt=0):
    return torch.Generator(device="cpu").manual_seed(1000003 * (seed + 1) + salt)


def _uv_sphere(n_lon, n_lat, radius=1.0):
    """Welded latitude/longitude sphere: positions [V,3] float64, triangles [T,3], uvs, uv triangles."""
    pole_s = 1 + (n_lat - 1) * n_lon
    j, i = torch.meshgrid(torch.arange(1, n_lat, device=DEV), torch.arange(n_lon, device=DEV), indexing="ij")
    phi, lam = math.pi * j.to(F64) / n_lat, 2 * math.pi * i.to(F64) / n_lon - math.pi
    ring = torch.stack([phi.sin() * lam.sin(), phi.cos(), phi.sin() * lam.cos()], -1).reshape(-1, 3)
    pole = torch.tensor([[0.0, 1.0, 0.0]], dtype=F64, device=DEV)
    pos = radius * torch.cat([pole, ring, -pole])
    jg, ig = torch.meshgrid(torch.arange(n_lat + 1, device=DEV), torch.arange(n_lon + 1, device=DEV), indexing="ij")
    uvs = torch.stack([ig.to(F64) / n_lon, jg.to(F64) / n_lat], -1).reshape(-1, 2).to(F32)
    j, i = torch.meshgrid(torch.arange(n_lat, device=DEV), torch.arange(n_lon, device=DEV), indexing="ij")
    i, j = i.reshape(-1), j.reshape(-1)

    def pid(i, j):
        inner = 1 + (j - 1) * n_lon + i % n_lon
        return torch.where(j == 0, 0, torch.where(j == n_lat, pole_s, inner))

    def tid(i, j):
        return j * (n_lon + 1) + i

    quad = [(i, j), (i + 1, j), (i, j + 1), (i + 1, j + 1)]
    order = [0, 2, 1, 1, 2, 3]
    pidx = torch.stack([pid(*quad[k]) for k in order], -1).reshape(-1, 3)
    tidx = torch.stack([tid(*quad[k]) for k in order], -1).reshape(-1, 3)
    return pos, pidx, uvs, tidx


def _waves(height, width, channels, gen, terms=6):
    """Smooth random values in [0,1], periodic in x."""
    x = (torch.arange(width, device=DEV, dtype=F32) + 0.5) / width
    y = (torch.arange(height, device=DEV, dtype=F32) + 0.5) / height
    out = torch.zeros(height, width, channels, device=DEV)
    for c in range(channels):
        for _ in range(terms):
            fx, (fy, ph, a) = int(torch.randint(1, 7, (1,), generator=gen)), torch.rand(3, generator=gen).tolist()
            out[..., c] += (0.5 + 0.5 * a) * torch.sin(2 * math.pi * (fx * x[None] + (0.5 + 5.5 * fy) * y[:, None] + ph))
    return (0.5 + 0.5 / terms * out).contiguous()


def _normal_map(height, width, gen, strength=0.3):
    g = strength * (2.0 * _waves(height, width, 2, gen) - 1.0)
    n = torch.cat([g, torch.ones(height, width, 1, device=DEV)], -1)
    return (0.5 + 0.5 * n / n.norm(dim=-1, keepdim=True)).contiguous()


def _bumps(pos, gen, amplitude, terms=4):
    g = torch.zeros(len(pos), dtype=F64, device=DEV)
    for _ in range(terms):
        d = torch.randn(3, generator=gen, dtype=F64)
        f, ph = torch.rand(2, generator=gen, dtype=F64).tolist()
        g += torch.sin((1 + 2 * f) * (pos @ (d / d.norm()).to(DEV)) + 2 * math.pi * ph) / terms
    return pos * (1 + amplitude * g)[:, None]


def _cameras(n, w, h, gen):
    """Eyes on a sphere of radius 3 looking at the origin; [n,4,4] row-major clip matrices."""
    mvps, eyes = [], []
    for _ in range(n):
        eye = torch.randn(3, generator=gen, dtype=F64)
        eye = 3 * eye / eye.norm()
        f = -eye / 3
        up = torch.tensor([0.0, 0.0, 1.0] if abs(f[1]) > 0.99 else [0.0, 1.0, 0.0], dtype=F64)
        s = torch.linalg.cross(f, up)
        s = s / s.norm()
        view = torch.eye(4, dtype=F64)
        view[0, :3], view[1, :3], view[2, :3] = s, torch.linalg.cross(s, f), -f
        view[:3, 3] = -view[:3, :3] @ eye
        fy, far = 1 / math.tan(math.radians(45) / 2), 10.0
        p = torch.zeros(4, 4, dtype=F64)
        p[0, 0], p[1, 1], p[2, 2], p[2, 3], p[3, 2] = fy * h / w, fy, far / (NEAR - far), NEAR * far / (NEAR - far), -1
        mvps.append((p @ view).to(F32))
        eyes.append(eye.to(F32))
    return torch.stack(mvps).to(DEV), torch.stack(eyes).to(DEV)


def _soup(case, seed):
    n, gen = case["lon"], _gen(seed)
    c = torch.rand(n, 3, generator=gen, dtype=F64) * torch.tensor([2.0, 2.0, 0.6]) + torch.tensor([-1.0, -1.0, 0.2])
    ang = 2 * math.pi * (torch.rand(n, 1, generator=gen, dtype=F64) + torch.tensor([[0.0, 1 / 3, 2 / 3]]))
    pos = c[:, None, :].repeat(1, 3, 1)
    pos[..., 0] += 3 / math.sqrt(n) * ang.cos()
    pos[..., 1] += 3 / math.sqrt(n) * ang.sin()
    idx = torch.arange(3 * n, device=DEV).reshape(n, 3)
    u = ((torch.arange(n, dtype=F64) + 0.5) / n).repeat_interleave(3)
    uvs = torch.stack([u, torch.full_like(u, 0.5)], 1).to(DEV, F32)
    tex = (0.25 + 0.5 * torch.rand(1, n, 3, generator=gen)).to(DEV)
    return dict(pos=pos.reshape(-1, 3).to(DEV, F32), pidx=idx, uvs=uvs, tidx=idx, maps=[(tex, 2.0 / 255.0, 0)],
                eps=2.0 / case["w"], mvp=torch.eye(4, device=DEV)[None], cam=torch.tensor([[0.0, 0.0, 3.0]], device=DEV),
                targets=_waves(case["h"], case["w"], 3, gen)[None], bg=(0.0, 0.0, 0.0), ambient=0.0, light=(1.0,) * 3)


def _maps(case, gen, start):
    """The textures a shading model reads, (data, eps, role); `start`: mid-optimisation, flatter than the target's."""
    s, m, k = case["tex"], case["maps"], (0.35 if start else 1.0)
    mix = lambda t, c: (c + k * (t - c)).contiguous()  # noqa: E731
    if case["shading"] == TRANSPARENT:
        t = _waves(s, s, 4, gen)
        t[..., 3] = 0.25 + 0.5 * t[..., 3]
        return [(t, EPS_TEX, 0)]
    if case["shading"] == UNLIT:
        return [(mix(_waves(s, s, 3, gen), 0.5), EPS_TEX, 0)]
    nrm = (_normal_map(m, m, gen, 0.3 * k), EPS_TEX, 1)
    if case["shading"] == LAMBERT:
        return [(mix(_waves(s, s, 4, gen), 0.5), EPS_TEX, 0), nrm]
    rough = mix(0.2 + 0.7 * _waves(m, m, 3, gen), 0.5)
    return [(mix(_waves(s, s, 3, gen), 0.5), EPS_TEX, 0), (rough, EPS_TEX, 2), (mix(_waves(m, m, 3, gen), 0.2), EPS_TEX, 3), nrm]


def _arrays(case, seed):
    """Everything a scene is made of, on the GPU; the target images are of another seeded shape and textures."""
    if case["scene"] == "soup":
        return _soup(case, seed)
    gen = _gen(seed)
    if case["scene"] == "spheres":
        pos, pidx, uvs, tidx = _uv_sphere(case["lon"], case["lat"], 0.6)
        off = [(-0.45, 0.0, -0.3), (0.0, 0.05, 0.0), (0.45, -0.05, 0.3)]
        nv, nt = len(pos), len(uvs)
        pos = torch.cat([pos + torch.tensor(o, dtype=F64, device=DEV) for o in off])
        pidx, tidx = torch.cat([pidx + k * nv for k in range(3)]), torch.cat([tidx + k * nt for k in range(3)])
        uvs = uvs.repeat(3, 1)
    else:
        pos, pidx, uvs, tidx = _uv_sphere(case["lon"], case["lat"])
    mvp, cam = _cameras(case["views"], case["w"], case["h"], gen)
    lit = case["shading"] in (LAMBERT, GGX)
    A = dict(pidx=pidx, uvs=uvs, tidx=tidx, eps=EPS_POS, mvp=mvp, cam=cam, ambient=0.1 if lit else 0.0,
             light=(3.0,) * 3 if case["shading"] == GGX else (1.0,) * 3,
             bg=(0.3,) * 3 if case["shading"] == TRANSPARENT else (0.0,) * 3)
    goal = dict(A, pos=_bumps(pos, gen, 0.08).to(F32), maps=_maps(case, gen, False))
    A["pos"], A["maps"] = _bumps(pos, gen, 0.05).to(F32).contiguous(), _maps(case, gen, True)
    if case["call"] in ("render", "step"):
        A["targets"] = torch.zeros(case["views"], case["h"], case["w"], 3, device=DEV)
    else:
        A["targets"] = torch.stack([_Image(case, goal, v).colour(None, 0).to(F32).reshape(case["h"], case["w"], 3)
                                    for v in range(case["views"])])
    return A


def _assets(case):
    """The scenes of a batched call: triangle counts spread over [lon, lat], texture sides around `tex`."""
    out = []
    for k in range(case["maps"]):
        t = math.exp(math.log(case["lon"]) + (k + 0.5) / case["maps"] * math.log(case["lat"] / case["lon"]))
        lat = max(2, int(round(math.sqrt(t / 4))))
        out.append(dict(case, call="estimate", lon=2 * lat, lat=lat, tex=max(16, case["tex"] * (1, 2, 4, 8)[3 * k % 4] // 4), maps=0))
    return out


def _scene(case, A):
    per_tri = 6 if case["scene"] != "soup" else 12
    tiles = -(-case["w"] // 16) * -(-case["h"] // 16)
    cap = (per_tri * len(A["pidx"]) + 24 * tiles) * case["views"]
    return sge.Scene(A["pos"], A["pidx"].to(torch.int32), A["uvs"], A["tidx"].to(torch.int32), A["maps"], A["eps"],
                     A["mvp"], A["cam"], case["w"], case["h"], targets=A["targets"], near=NEAR, shading=case["shading"],
                     light_dir=LIGHT, light_rgb=A["light"], ambient=A["ambient"], background=A["bg"],
                     max_pairs_per_call=min(64, case["pairs"]), bin_capacity=cap,
                     footprint=sge.FOOT_NEAREST if case["nearest"] else sge.FOOT_BILINEAR)


def _moments(n, seed):
    """Adam's m and v of a loop under way, and summed gradients with their counts."""
    g = torch.Generator(device=DEV).manual_seed(7 + seed)
    m = 0.1 * torch.randn(n, generator=g, device=DEV)
    v = 0.01 * (0.5 + torch.rand(n, generator=g, device=DEV))
    s = 0.1 * torch.randn(n, generator=g, device=DEV)
    return m, v, s, torch.randint(0, 40, (n,), generator=g, device=DEV, dtype=torch.int32)


class State:
    pass


def prepare(case, seed):
    st = State()
    st.case, st.seed = case, seed
    if case["call"] == "batch":
        st.parts = [prepare(c, seed + 100 * k) for k, c in enumerate(_assets(case))]
        views = list(range(case["views"]))
        st.batch = sge.Batch([(p.scene, views, p.grad, p.counts, p.loss) for p in st.parts])
        return st
    A = _arrays(case, seed)
    st.A, st.scene, st.views = A, _scene(case, A), list(range(case["views"]))
    n = st.scene.n_params
    st.lr = (EPS_POS, [t[1] for t in A["maps"]])
    if case["call"] in ("estimate", "iterate"):
        st.grad, st.counts = st.scene.new_grad_buffers()
        st.loss = torch.zeros(case["views"], device=DEV)
    if case["call"] == "step":
        st.m, st.v, st.grad, st.counts = _moments(n, seed)
    if case["call"] == "iterate":
        st.m, st.v, _, _ = _moments(n, seed)
        st.iter = sge.IterState(ITER, T_ADAM)
        st.theta_in = torch.cat([t.reshape(-1) for t in st.scene.param_groups()]).cpu().pin_memory()
        st.targets_in = A["targets"].cpu().pin_memory()
        st.theta_out, st.loss_out = torch.empty(n).pin_memory(), torch.empty(case["views"]).pin_memory()
    return st


def run(st):
    case, call = st.case, st.case["call"]
    if call == "estimate":
        st.grad.zero_(), st.counts.zero_(), st.loss.zero_()
        st.scene.estimate_grad(st.seed, ITER, st.views, case["pairs"], st.grad, st.counts, loss=st.loss)
        return [st.grad, st.counts, st.loss]
    if call == "batch":
        for p in st.parts:
            p.grad.zero_(), p.counts.zero_(), p.loss.zero_()
        st.batch.estimate_grad(st.seed, ITER, case["pairs"])
        return [[p.grad, p.counts, p.loss] for p in st.parts]
    if call == "autograd":
        loss = sge.sge_loss(st.scene, st.seed, ITER, st.views, case["pairs"])
        return [loss.detach(), *torch.autograd.grad(loss, st.scene.param_groups())]
    if call == "iterate":
        st.scene.iterate_host(st.seed, st.iter, st.views, case["pairs"], st.grad, st.counts, st.m, st.v, *st.lr,
                              loss_dev=st.loss, theta_in=st.theta_in, targets_in=st.targets_in,
                              theta_out=st.theta_out, loss_out=st.loss_out)
        return [st.theta_out, st.m, st.v, st.loss_out]
    if call == "render":
        return [list(st.scene.render_idb(v, seed=st.seed, it=ITER, pair=v, side=1)) for v in st.views]
    st.scene.step(sge.STEP_ADAM, st.grad, st.counts, case["pairs"], *st.lr, m=st.m, v=st.v, t=T_ADAM)
    return [st.m, st.v, *st.scene.param_groups()]


def work(case):
    """Bytes: indices, UVs, parameters and targets read, sums and counts written, once each; a step reads and
    writes what it updates.  Operations: coverage, UV, sampling, shading and credits of the visible triangle
    of both sides of a pixel pair, on the 57 % of the pixels a unit sphere covers."""
    if case["call"] == "batch":
        parts = [work(c) for c in _assets(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    tris = case["lon"] if case["scene"] == "soup" else 2 * case["lon"] * case["lat"] * (3 if case["scene"] == "spheres" else 1)
    verts = 3 * tris if case["scene"] == "soup" else tris / 2
    texels = {UNLIT: 3 * case["tex"] ** 2, TRANSPARENT: 4 * case["tex"] ** 2,
              LAMBERT: 4 * case["tex"] ** 2 + 3 * case["maps"] ** 2, GGX: 3 * case["tex"] ** 2 + 9 * case["maps"] ** 2}[case["shading"]]
    if case["scene"] == "soup":
        texels = 3 * case["tex"]
    d, px = 3 * verts + texels, case["w"] * case["h"] * case["views"]
    if case["call"] == "step":
        return {"bytes": 40 * d, "flops": 20 * d}
    scene = 24 * tris + 8 * verts + 4 * d
    ops = {UNLIT: 114, LAMBERT: 230, GGX: 390, TRANSPARENT: 300}[case["shading"]]
    if case["call"] == "render":
        return {"bytes": scene + 28 * px, "flops": 0.57 * px * ops / 2}
    extra = {"autograd": 4 * d, "iterate": 24 * d + 12 * px}.get(case["call"], 0)
    return {"bytes": scene + 12 * px + 8 * d + extra, "flops": 0.57 * px * case["pairs"] * ops}


# ------------------------------------------------------------------------------------ 64-bit values
_M64 = (1 << 64) - 1
_GAMMA, _MUL1, _MUL2 = 0x9E3779B97F4A7C15, 0xBF58476D1CE4E5B9, 0x94D049BB133111EB


def _signed(x):
    x &= _M64
    return x - (1 << 64) if x >> 63 else x


def _mix(z):
    z = ((z ^ (z >> 30)) * _MUL1) & _M64
    z = ((z ^ (z >> 27)) * _MUL2) & _M64
    return z ^ (z >> 31)


def _shr(x, n):
    return (x >> n) & ((1 << (64 - n)) - 1)


def _signs(seed, it, view, pair, n):
    """s_i of one estimate for i < n, +-1 float32: bit i mod 64 of SplitMix64's output i // 64."""
    key = _mix((seed + _GAMMA) & _M64)
    for x in (it, view, pair):
        key = _mix(((key ^ x) + _GAMMA) & _M64)
    z = (torch.arange(1, (n + 63) // 64 + 1, device=DEV) * _signed(_GAMMA)) + _signed(key)
    z = (z ^ _shr(z, 30)) * _signed(_MUL1)
    z = (z ^ _shr(z, 27)) * _signed(_MUL2)
    z = z ^ _shr(z, 31)
    bits = (z[:, None] >> torch.arange(64, device=DEV)) & 1
    return (1 - 2 * bits.reshape(-1)[:n]).to(F32)


def _unit(a):
    n = a.norm(dim=-1, keepdim=True)
    return torch.where(n > 0, a / n.clamp_min(1e-300), a)


class _Image:
    """One view of a scene rendered under signs s (None: unperturbed) and a side."""

    def __init__(self, case, A, view):
        self.case, self.A, self.view = case, A, view
        self.w, self.h = case["w"], case["h"]
        self.px = torch.arange(self.w * self.h, device=DEV)

    def raster(self, s, side):
        """The visible triangle of every pixel ([layers, pixels], -1: none) with the perturbed parameters."""
        A, W, H = self.A, self.w, self.h
        self.pos, self.tex, o = A["pos"], [], 3 * len(A["pos"])
        if side:
            self.pos = A["pos"] + side * s[:o].reshape(-1, 3) * torch.tensor(A["eps"], dtype=F32, device=DEV)
        for t, eps, _ in A["maps"]:
            e = torch.tensor(eps, dtype=F32, device=DEV)
            self.tex.append(t + side * s[o:o + t.numel()].reshape(t.shape) * e if side else t)
            o += t.numel()
        m, (x, y, z) = A["mvp"][self.view], self.pos.unbind(1)
        cx, cy, cz, cw = (((m[r, 0] * x + m[r, 1] * y) + m[r, 2] * z) + m[r, 3] for r in range(4))
        iw = torch.ones_like(cw) / cw
        X = ((((cx * iw) * 0.5 + 0.5) * W) * 256.0)
        Y = ((0.5 - (cy * iw) * 0.5) * H) * 256.0
        ok = (cw > NEAR) & (X.abs() < 2.0 ** 23) & (Y.abs() < 2.0 ** 23)
        X, Y = (torch.where(ok, t, torch.zeros_like(t)).round().to(I64) for t in (X, Y))
        p = A["pidx"]
        self.X, self.Y, self.z, self.iw = X[p], Y[p], (cz * iw)[p], iw[p]
        X, Y = self.X, self.Y
        area = (X[:, 1] - X[:, 0]) * (Y[:, 2] - Y[:, 0]) - (Y[:, 1] - Y[:, 0]) * (X[:, 2] - X[:, 0])
        self.sgn = torch.where(area > 0, 1, -1)
        self.inv_area = torch.ones_like(iw[:1]) / area.abs().to(F32)
        x0, x1 = ((X.amin(1) + 127) // 256).clamp_min(0), ((X.amax(1) - 128) // 256).clamp_max(W - 1)
        y0, y1 = ((Y.amin(1) + 127) // 256).clamp_min(0), ((Y.amax(1) - 128) // 256).clamp_max(H - 1)
        nx = (x1 - x0 + 1).clamp_min(0)
        n = torch.where(ok[p].all(1) & (area != 0), nx * (y1 - y0 + 1).clamp_min(0), 0)
        tri = torch.repeat_interleave(torch.arange(len(p), device=DEV), n)
        k = torch.arange(len(tri), device=DEV) - (n.cumsum(0) - n)[tri]
        px, py = x0[tri] + k % nx[tri], y0[tri] + k // nx[tri]
        inside, l = self.weights(tri, px, py, True)
        tri, pix, l = tri[inside], (py * W + px)[inside], l[inside]
        zt = self.z[tri]
        d = ((l[:, 0] * zt[:, 0] + l[:, 1] * zt[:, 1]) + l[:, 2] * zt[:, 2]).view(torch.int32).to(I64)
        key = (torch.where(d >= 0, d, d ^ 0x7FFFFFFF) << 32) | tri
        out, last = [], torch.iinfo(I64).max
        for _ in range(LAYERS if self.case["shading"] == TRANSPARENT else 1):
            best = torch.full((W * H,), last, device=DEV).scatter_reduce(0, pix, key, "amin")
            out.append(torch.where(best == last, -1, best & 0xFFFFFFFF))
            keep = key != best[pix]
            key, pix = key[keep], pix[keep]
        return torch.stack(out)

    def weights(self, tri, px, py, test=False):
        """Barycentric weights (float32) of triangles at pixel centres; with `test` also the coverage."""
        X, Y, sgn = self.X[tri], self.Y[tri], self.sgn[tri]
        qx, qy, l, inside = 256 * px + 128, 256 * py + 128, [], True
        for k in range(3):
            a, b = (k + 1) % 3, (k + 2) % 3
            dx, dy = sgn * (X[:, b] - X[:, a]), sgn * (Y[:, a] - Y[:, b])
            e = dx * (qy - Y[:, a]) + dy * (qx - X[:, a])
            l.append(e.to(F32) * self.inv_area[tri])
            if test:
                inside = inside & torch.where((dy > 0) | ((dy == 0) & (dx > 0)), e >= 0, e > 0)
        return (inside, torch.stack(l, 1)) if test else torch.stack(l, 1)

    def surface(self, tri, pix):
        """UV (float32), perspective-correct weights and each map's footprint (texel ids [N,4], weights, nearest)."""
        l = self.weights(tri, pix % self.w, pix // self.w)
        q = l * self.iw[tri]
        qs = (q[:, 0] + q[:, 1]) + q[:, 2]
        t = self.A["uvs"][self.A["tidx"][tri]]
        u, v = (((q[:, 0] * t[:, 0, c] + q[:, 1] * t[:, 1, c]) + q[:, 2] * t[:, 2, c]) / qs for c in range(2))
        feet, by_size = [], {}
        for d, _, _ in self.A["maps"]:
            th, tw = d.shape[:2]
            if (th, tw) not in by_size:
                x, y = u * tw - 0.5, v * th - 0.5
                fx, fy = ((c - c.floor()).to(F64) for c in (x, y))
                ix, iy = x.floor().to(I64), y.floor().to(I64)
                ids = torch.stack([(iy + j).clamp(0, th - 1) * tw + (ix + i) % tw for j in (0, 1) for i in (0, 1)], 1)
                wq = torch.stack([(1 - fx) * (1 - fy), fx * (1 - fy), (1 - fx) * fy, fx * fy], 1)
                near = (v * th).floor().to(I64).clamp(0, th - 1) * tw + (u * tw).floor().to(I64) % tw
                by_size[th, tw] = (ids, wq, near[:, None])
            feet.append(by_size[th, tw])
        return torch.stack([u, v], 1), q.to(F64) / qs.to(F64)[:, None], feet

    def shade(self, tri, pix):
        A, (uv, b, feet) = self.A, self.surface(tri, pix)
        val = {}
        for t, (ids, wq, _), (d, _, role) in zip(self.tex, feet, A["maps"]):
            val[role] = (t.reshape(-1, d.shape[2])[ids].to(F64) * wq[..., None]).sum(1)
        alb = val[0]
        if self.case["shading"] in (UNLIT, TRANSPARENT):
            return alb, uv, feet
        p, t = self.pos[A["pidx"][tri]].to(F64), A["uvs"][A["tidx"][tri]].to(F64)
        e1, e2, d1, d2 = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0], t[:, 1] - t[:, 0], t[:, 2] - t[:, 0]
        N = _unit(torch.linalg.cross(e1, e2))
        det = (d1[:, :1] * d2[:, 1:] - d2[:, :1] * d1[:, 1:])
        T = torch.where(det != 0, (e1 * d2[:, 1:] - e2 * d1[:, 1:]) / torch.where(det != 0, det, 1.0), e1)
        T = _unit(T - N * (N * T).sum(1, keepdim=True))
        nm = 2 * val[1] - 1
        n = T * nm[:, :1] + torch.linalg.cross(N, T) * nm[:, 1:2] + N * nm[:, 2:3]
        n = _unit(torch.where((n * n).sum(1, keepdim=True) == 0, N, n))
        f32 = lambda c: torch.tensor(c, dtype=F32, device=DEV).to(F64)  # noqa: E731
        L, light, amb = f32(LIGHT), f32(A["light"]), f32(A["ambient"])
        ndl = (n @ L).clamp_min(0)[:, None]
        if self.case["shading"] == LAMBERT:
            return alb[:, :3] * (amb + light * ndl), uv, feet
        V = _unit(A["cam"][self.view].to(F64) - (b[..., None] * p).sum(1))
        Hh = _unit(L + V)
        ndv, ndh = ((n * x).sum(1, keepdim=True) for x in (V, Hh))
        ndv, ndh, vdh = ndv.clamp_min(1e-4), ndh.clamp_min(0), (V * Hh).sum(1, keepdim=True).clamp_min(0)
        a = val[2][:, :1].clamp(0.02, 1.0) ** 2
        D = a ** 2 / (math.pi * (ndh ** 2 * (a ** 2 - 1) + 1) ** 2)
        G = (ndl / (ndl * (1 - a / 2) + a / 2)) * (ndv / (ndv * (1 - a / 2) + a / 2))
        mt = val[3][:, :1]
        F0 = 0.04 * (1 - mt) + alb * mt
        F = F0 + (1 - F0) * (1 - vdh) ** 5
        return light * ((1 - F) * (1 - mt) * alb * ndl / math.pi + D * G * F / (4 * ndv)) + amb * alb, uv, feet

    def colour(self, s, side, credits=None):
        """[pixels, 3] float64; `credits` (vertex ids, texel ids of each map per pixel) gets this render's, -1: none."""
        n, bg = self.w * self.h, torch.tensor(self.A["bg"], dtype=F32, device=DEV).to(F64)
        ids = self.raster(s, side)
        rgb, trans = torch.zeros(n, 3, dtype=F64, device=DEV), torch.ones(n, 1, dtype=F64, device=DEV)
        for tris in ids:
            pix = self.px[tris >= 0]
            tri = tris[pix]
            c, uv, feet = self.shade(tri, pix)
            al = c[:, 3:].clamp(0, 1) if self.case["shading"] == TRANSPARENT else torch.ones_like(c[:, :1])
            rgb[pix] += trans[pix] * al * c[:, :3]
            trans[pix] *= 1 - al
            if credits is not None:
                near = self.case["nearest"]
                for k, v in enumerate([self.A["pidx"][tri]] + [f[2] if near else f[0] for f in feet]):
                    credits[k].append(torch.full((n, v.shape[1]), -1, device=DEV).index_copy_(0, pix, v))
        self.uv, self.ids = torch.zeros(n, 2, device=DEV), ids
        if len(ids) == 1 and len(pix):
            self.uv[pix] = uv
        return rgb + trans * bg


def _estimate(case, A, seed):
    """For the sign seed: Eq. 9's sums [d], and per view the mean image error of the perturbed renders, in float64."""
    groups = [A["pos"]] + [t for t, _, _ in A["maps"]]
    chans = [t.shape[-1] for t in groups]
    d = sum(t.numel() for t in groups)
    total, loss = torch.zeros(d, dtype=F64, device=DEV), []
    for view in range(case["views"]):
        img, tgt = _Image(case, A, view), A["targets"][view].reshape(-1, 3).to(F64)
        f = 0.0
        for pair in range(case["pairs"]):
            s = _signs(seed, ITER, view, pair, d)
            credits = [[] for _ in groups]
            fp, fm = (((img.colour(s, side, credits) - tgt) ** 2).sum(1) for side in (1, -1))
            f += float((0.5 * (fp + fm)).sum())
            df, o = fp - fm, 0
            for t, c, ids in zip(groups, chans, credits):
                ids = torch.cat(ids, 1).sort(1).values
                once = ids >= 0
                once[:, 1:] &= ids[:, 1:] != ids[:, :-1]
                key = torch.zeros(t.numel() // c, dtype=F64, device=DEV)
                key.index_add_(0, ids[once], df[:, None].expand_as(ids)[once])
                total[o:o + t.numel()] += s[o:o + t.numel()].to(F64) * key.repeat_interleave(c)
                o += t.numel()
        loss.append(f / case["pairs"])
    return total, torch.tensor(loss, dtype=F64, device=DEV)


def _adam(theta, m, v, sums, eps, lr, n):
    f = lambda x: torch.tensor(x, dtype=F32).to(F64).item()  # noqa: E731
    b1, b2, g = f(0.9), f(0.999), sums / (2 * f(eps) * n)
    m, v = b1 * m.to(F64) + (1 - b1) * g, b2 * v.to(F64) + (1 - b2) * g * g
    return theta.to(F64) - f(lr) * (m / (1 - b1 ** T_ADAM)) / ((v / (1 - b2 ** T_ADAM)).sqrt() + f(1e-8)), m, v


def exact(case, seed):
    if case["call"] == "batch":  # each asset has its own inputs, the call one seed
        parts = [_estimate(c, _arrays(c, seed + 100 * k), seed) for k, c in enumerate(_assets(case))]
        return [[sums, None, loss] for sums, loss in parts]
    A, call = _arrays(case, seed), case["call"]
    groups = [A["pos"]] + [t for t, _, _ in A["maps"]]
    eps = [A["eps"]] + [e for _, e, _ in A["maps"]]
    if call == "render":
        out = []
        for v in range(case["views"]):
            img = _Image(case, A, v)
            s = _signs(seed, ITER, v, v, sum(t.numel() for t in groups))
            rgb = img.colour(s, 1)
            out.append([None, img.uv.to(F64).reshape(case["h"], case["w"], 2), rgb.reshape(case["h"], case["w"], 3)])
        return out
    if call == "step":
        m, v, sums, _ = _moments(sum(t.numel() for t in groups), seed)
        n = case["pairs"]
    else:
        if case["views"] * case["pairs"] * case["w"] * case["h"] > (1 << 28):
            return None
        sums, loss = _estimate(case, A, seed)
        n = case["pairs"] * case["views"]
        if call == "estimate":
            return [sums, None, loss]
        if call == "autograd":
            f = sum(float(((_Image(case, A, v).colour(None, 0) - A["targets"][v].reshape(-1, 3).to(F64)) ** 2).sum())
                    for v in range(case["views"]))
            parts = sums.split([t.numel() for t in groups])
            e32 = [float(torch.tensor(e, dtype=F32)) for e in eps]
            return [torch.tensor(f, dtype=F64), *[p.reshape(t.shape) / (2 * e * case["pairs"]) for p, t, e in zip(parts, groups, e32)]]
        m, v, _, _ = _moments(len(sums), seed)
    res, o = [], 0
    for t, e, lr in zip(groups, eps, [EPS_POS] + eps[1:]):
        sl = slice(o, o + t.numel())
        res.append(_adam(t.reshape(-1), m[sl], v[sl], sums[sl].to(F64), e, lr, n))
        o += t.numel()
    theta, m, v = zip(*res)
    if call == "iterate":
        return [torch.cat(theta), torch.cat(m), torch.cat(v), loss]
    return [torch.cat(m), torch.cat(v), *[x.reshape(t.shape) for x, t in zip(theta, groups)]]
