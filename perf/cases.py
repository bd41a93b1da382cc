"""The work that users of the library have it do, as timed cases.

Six kinds of call, each through the binding's public entry points:

- ``view``: one or more views of a resident cache (``fnr_render``), uniform samples;
- ``walk``: the same with every voxel on the ray integrated (``FNR_RENDER_VOXELS``);
- ``serve``: a burst of view requests through the request loop (``fnr_submit`` / ``fnr_wait``);
- ``mlp``: a cache built from the F_pos / F_dir networks (``fnr_build_cache`` from MLPs);
- ``arrays``: a cache built from device arrays, with the storage conversion its precision needs;
- ``uncached``: one view rendered straight from the networks (``fnr_render_mlp``).

Sizes are those of the repository's benchmark and tests (k = 64 .. 512, 64 x 64 .. 1920 x 1080 pixels,
N = 64 .. 192, D = 8 with smaller and ragged ones beside it). Scenes are spheres and thin box shells of
density 50 in the box [-1.5, 1.5]^3 with channels that are sums of sinusoids, seen from a radius-4 upper
hemisphere: the benchmark's scene family, drawn here on the GPU.
"""

import math

import numpy as np
import torch

import paper_2103_10380_gb300 as fnr

FP32, FP16, E4M3 = fnr.FNR_PREC_FP32, fnr.FNR_PREC_FP16, fnr.FNR_PREC_FP8_E4M3
LO, HI = -1.5, 1.5
NEAR, FAR, THR = 2.0, 6.0, 1e-4
RESOLUTIONS = ((256, 256), (512, 512), (800, 800), (1280, 720), (1920, 1080))
POS_FREQS, DIR_FREQS = 10, 4


def listed():
    return [
        # a thumbnail or a smoke check: one small view of a small cache, where the call itself is what is paid
        dict(name="view-thumbnail", kind="view", k=64, D=8, l=64, prec=FP32, layout=0, W=64, H=64, views=1, N=64,
             skip=0, bilinear=0, stats=1),
        # the ordinary call: one 800 x 800 view per launch of a binary32 cache at the paper's resolution
        dict(name="view-800-fp32", kind="view", k=512, D=8, l=512, prec=FP32, layout=0, W=800, H=800, views=1, N=128,
             skip=0, bilinear=0, stats=0),
        # a camera path rendered in one call from the smallest dense form, empty space skipped
        dict(name="views-720p-e4m3-skip", kind="view", k=512, D=8, l=512, prec=E4M3, layout=0, W=1280, H=720, views=4,
             N=192, skip=1, bilinear=0, stats=0),
        # odd sizes throughout, a sparse cache, fewer components, interpolated direction weights
        dict(name="view-ragged-bricks", kind="view", k=301, D=6, l=255, prec=FP16, layout=1, W=643, H=481, views=1,
             N=100, skip=1, bilinear=1, stats=1),
        # the quality mode: every voxel on the ray, over empty space
        dict(name="walk-800-fp32-skip", kind="walk", k=512, D=8, l=512, prec=FP32, W=800, H=800, skip=1, stats=1),
        # the same without skipping, half precision, a smaller cache
        dict(name="walk-512-fp16", kind="walk", k=256, D=8, l=256, prec=FP16, W=512, H=512, skip=0, stats=0),
        # a service under load: a burst of requests of mixed resolution
        dict(name="serve-burst-fp16", kind="serve", k=512, D=8, l=512, prec=FP16, requests=20, N=128),
        # a trained model turned into a cache at full size, and a preview of it
        dict(name="mlp-512-fp32", kind="mlp", k=512, D=8, l=512, prec=FP32),
        dict(name="mlp-64-fp16", kind="mlp", k=64, D=8, l=64, prec=FP16),
        # arrays from elsewhere stored as a cache: the quantised form at full size, and a sparse one of ragged size
        dict(name="arrays-512-e4m3", kind="arrays", k=512, D=8, l=512, prec=E4M3, layout=0),
        dict(name="arrays-250-fp16-bricks", kind="arrays", k=250, D=8, l=250, prec=FP16, layout=1),
        # a view straight from the networks, without a cache
        dict(name="uncached-800", kind="uncached", D=8, W=800, H=800, N=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "walk", "serve", "mlp", "arrays", "uncached"])
    k, l = _log(rng, 64, 512), _log(rng, 64, 512)
    prec = rng.choice([FP32, FP16, E4M3])
    if kind == "view":
        views = rng.choice([1, 1, 1, 2, 4])
        W, H = _log(rng, 64, 1280), _log(rng, 64, 720)
        return dict(kind=kind, k=k, D=rng.choice([4, 6, 8, 8, 8, 12]), l=l, prec=prec, layout=rng.choice([0, 0, 0, 1]),
                    W=W, H=H, views=views, N=_log(rng, 64, 192), skip=rng.choice([0, 1]),
                    bilinear=rng.choice([0, 0, 0, 1]), stats=rng.choice([0, 1]))
    if kind == "walk":
        return dict(kind=kind, k=k, D=rng.choice([4, 8, 8]), l=l, prec=prec, W=_log(rng, 64, 800),
                    H=_log(rng, 64, 800), skip=rng.choice([0, 1]), stats=rng.choice([0, 1]))
    if kind == "serve":
        return dict(kind=kind, k=k, D=rng.choice([4, 8, 8]), l=l, prec=prec, requests=rng.randint(1, 20),
                    N=_log(rng, 64, 128))
    if kind == "mlp":
        return dict(kind=kind, k=k, D=rng.choice([4, 8, 8]), l=l, prec=rng.choice([FP32, FP16]))
    if kind == "arrays":
        return dict(kind=kind, k=k, D=rng.choice([4, 6, 8, 8]), l=l, prec=prec, layout=rng.choice([0, 0, 1]))
    return dict(kind=kind, D=rng.choice([4, 8, 8]), W=_log(rng, 64, 800), H=_log(rng, 64, 800), N=_log(rng, 64, 128))


# ------------------------------------------------------------------ inputs
def _centres(n, device="cuda", dtype=torch.float64):
    return LO + (torch.arange(n, device=device, dtype=dtype) + 0.5) * ((HI - LO) / n)


def _scene(shape, rng, k, D):
    """Density [k^3] and channels [k^3, 3D] in binary32 on the GPU: 32 spheres, 16 box shells (drawn from `shape`)
    and 4 sinusoids a channel."""
    x = _centres(k)
    sigma = torch.zeros((k, k, k), device="cuda", dtype=torch.float32)

    def span(c, h):  # cells whose centres can lie within h of c
        a = int(math.floor((c - h - LO) / (HI - LO) * k)) - 1
        b = int(math.ceil((c + h - LO) / (HI - LO) * k)) + 1
        return slice(min(max(a, 0), k), min(max(b, 0), k))

    for c, r in zip(shape.uniform(-1, 1, (32, 3)), shape.uniform(0.1, 0.4, 32)):
        s = [span(c[a], r) for a in range(3)]
        d = [(x[s[a]] - c[a]) ** 2 for a in range(3)]
        inside = (d[2][:, None, None] + d[1][None, :, None] + d[0][None, None, :]) < r * r
        sigma[s[2], s[1], s[0]].masked_fill_(inside, 50.0)
    for c, h in zip(shape.uniform(-1, 1, (16, 3)), shape.uniform(0.1, 0.5, (16, 3))):
        s = [span(c[a], h[a]) for a in range(3)]
        d = [(x[s[a]] - c[a]).abs() for a in range(3)]

        def box(t):
            m = [d[a] < h[a] - t for a in range(3)]
            return m[2][:, None, None] & m[1][None, :, None] & m[0][None, None, :]

        sigma[s[2], s[1], s[0]].masked_fill_(box(0.0) & ~box(0.02), 50.0)
    # channel c at (x, y, z): sum_t a sin(2 pi f . x + phase), separated along x into 1, sin, cos of 2 pi j x
    nch, nt = 3 * D, 12 * D
    amp, phase = rng.uniform(-1, 1, nt), rng.uniform(0, 2 * math.pi, nt)
    freq = rng.integers(-2, 3, (nt, 3))
    freq[(freq == 0).all(1), 0] = 1
    dev = lambda v: torch.as_tensor(v, device="cuda", dtype=torch.float64)
    w = 2 * math.pi * x
    fy, fz, ph, am = dev(freq[:, 1]), dev(freq[:, 2]), dev(phase), dev(amp)
    # rows of the x basis: 1, cos w, sin w, cos 2w, sin 2w
    basis = torch.stack([torch.ones_like(w), w.cos(), w.sin(), (2 * w).cos(), (2 * w).sin()], 1).float()
    psin = torch.zeros((nt, 5, nch), dtype=torch.float64)
    pcos = torch.zeros((nt, 5, nch), dtype=torch.float64)
    for t in range(nt):
        f, ch = int(freq[t, 0]), t // 4  # a sin(f w + q) = a sin q cos(f w) + a cos q sin(f w)
        psin[t, 0 if f == 0 else 2 * abs(f) - 1, ch] = 1.0
        if f:
            pcos[t, 2 * abs(f), ch] = 1.0 if f > 0 else -1.0
    psin, pcos = psin.reshape(nt, -1).cuda().float(), pcos.reshape(nt, -1).cuda().float()
    uvw = torch.empty((k, k, k, nch), device="cuda", dtype=torch.float32)
    for z in range(k):
        q = w[:, None] * fy + w[z] * fz + ph
        rows = (am * q.sin()).float() @ psin + (am * q.cos()).float() @ pcos
        torch.matmul(basis, rows.reshape(k, 5, nch), out=uvw[z])
    return sigma.reshape(-1), uvw.reshape(-1)


def _directions(rng, l, D):
    """Direction weights [l, l, D]: random polynomials of degree 4 in the unit vector at the bin centres."""
    th = (torch.arange(l, device="cuda", dtype=torch.float64) + 0.5) * (math.pi / l)
    ph = (torch.arange(l, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / l)
    v = [th.sin()[:, None] * ph.cos(), th.sin()[:, None] * ph.sin(), th.cos()[:, None].expand(l, l)]
    mono = [v[0] ** a * v[1] ** b * v[2] ** c for a in range(5) for b in range(5 - a) for c in range(5 - a - b)]
    coef = torch.as_tensor(rng.normal(size=(len(mono), D)) * 0.6, device="cuda")
    return (torch.stack(mono, -1) @ coef).float().contiguous()


def _camera(rng, W, H):
    z, phi = rng.uniform(0, 0.99), rng.uniform(0, 2 * math.pi)
    s = math.sqrt(1 - z * z)
    back = np.array([s * math.cos(phi), s * math.sin(phi), z])
    right = np.cross([0.0, 0.0, 1.0], back)
    right /= np.linalg.norm(right)
    c2w = np.stack([right, np.cross(back, right), back, 4.0 * back], 1).astype(np.float32).reshape(12)
    f = np.float32(0.5 * W / math.tan(math.radians(20.0)))
    return dict(c2w=c2w, fx=f, fy=f, cx=np.float32(W / 2), cy=np.float32(H / 2), W=W, H=H)


def _network(rng, dims):
    """He-uniform layers: bf16 weights [out][in], binary32 biases."""
    out = []
    for i, o in zip(dims[:-1], dims[1:]):
        lim = math.sqrt(6.0 / i)
        out.append((torch.as_tensor(rng.uniform(-lim, lim, (o, i)), device="cuda").to(torch.bfloat16).contiguous(),
                    torch.as_tensor(rng.uniform(-0.05, 0.05, o), device="cuda", dtype=torch.float32)))
    return out


def _networks(rng, D):
    return (_network(rng, [6 * POS_FREQS] + [256] * 8 + [1 + 3 * D]),
            _network(rng, [6 * DIR_FREQS] + [128] * 4 + [D]))


class _Context:
    """A library context, given back when nothing holds it any more."""

    def __init__(self):
        self.handle = fnr.fnr_context_create(0, 0)

    def __del__(self):
        torch.cuda.synchronize()
        fnr.fnr_context_destroy(self.handle)


class _Cache:
    """A built cache: freed when neither the state nor an output that lies in it is held any more."""

    def __init__(self, context, handle):
        self.context, self.handle = context, handle

    def __del__(self):
        torch.cuda.synchronize()
        fnr.fnr_cache_free(self.context.handle, self.handle)


def _desc(c):
    return fnr.make_desc(c["k"], c["D"], c["l"], c["prec"], FP32 if c["prec"] == FP32 else FP16,
                         layout=c.get("layout", 0))


def _samples(c):
    return 3 * c["k"] if c["kind"] == "walk" else c["N"]


def _inputs(case, seed):
    """What the seed alone decides: (sigma, uvw, beta) or networks, and cameras."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    d = {}
    if kind in ("mlp", "uncached"):
        d["nets"] = _networks(rng, case["D"])
    else:
        # a sparse build's outputs are as large as the scene has occupied bricks: one geometry, appearance by the seed
        shape = np.random.default_rng(0) if kind == "arrays" and case["layout"] else rng
        d["arrays"] = (*_scene(shape, rng, case["k"], case["D"]), _directions(rng, case["l"], case["D"]))
    if kind == "serve":
        d["cams"] = [_camera(rng, *RESOLUTIONS[i % len(RESOLUTIONS)]) for i in range(case["requests"])]
    elif kind in ("view", "walk", "uncached"):
        d["cams"] = [_camera(rng, case["W"], case["H"]) for _ in range(case.get("views", 1))]
    return d


def prepare(case, seed):
    c, d, context = case, _inputs(case, seed), _Context()
    st = dict(case=c, context=context)
    if "cams" in d:
        st["cams"] = [fnr.make_camera(v) for v in d["cams"]]
        st["params"] = fnr.make_params(_samples(c), NEAR, FAR, THR, skip_empty=bool(c.get("skip")),
                                       dir_bilinear=bool(c.get("bilinear")), voxels=c["kind"] == "walk")
        pixels = [v["W"] * v["H"] for v in d["cams"]]
        if c["kind"] == "serve":
            st["rgba"] = [torch.zeros(4 * n, device="cuda") for n in pixels]
        else:
            st["rgba"] = torch.zeros(4 * sum(pixels), device="cuda")
            st["stats"] = torch.zeros(4 * sum(pixels), device="cuda", dtype=torch.int32) if c.get("stats") else None
    if c["kind"] in ("view", "walk", "serve"):
        st["cache"] = _Cache(context, fnr.fnr_build_cache(context.handle, _desc(c), *d["arrays"]))
        if c["kind"] == "serve":
            fnr.fnr_serve_start(context.handle)
    else:
        st.update(d)
        st.update(desc=_desc(c) if "k" in c else None)
    return st


# ------------------------------------------------------------------ one pass
class _Memory:
    """Device memory of a cache as an array; a tensor made of it holds this object, and so the cache."""

    def __init__(self, owner, address, shape, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = dict(shape=shape, typestr=typestr, data=(address, False), version=3)


def _stored(c, cache):
    """A built cache's memory: densities, records, direction weights and what the renders skip by."""
    lay = fnr.fnr_cache_get_layout(cache.handle)
    at = lambda address, shape, typestr: torch.as_tensor(_Memory(cache, address, shape, typestr), device="cuda")
    t, es = {FP32: ("<f4", 4), FP16: ("<f2", 2), E4M3: ("|u1", 1)}[c["prec"]]
    k, l, D = c["k"], c["l"], c["D"]
    nb = -(-k // lay.occupancy_brick)
    nj = -(-k // lay.distance_brick)
    cells = lay.n_bricks * lay.occupancy_brick ** 3 if lay.layout else k ** 3
    out = dict(sigma=at(lay.sigma_dev, (cells,), t),
               uvw=at(lay.uvw_dev, (cells, lay.record_stride // es), t)[:, :3 * D],  # without the records' padding
               beta=at(lay.beta_dev, (l, l, D), "<f4" if c["prec"] == FP32 else "<f2"),
               occupancy=at(lay.occupancy_dev, (-(-nb ** 3 // 32),), "<i4"),
               distance=at(lay.brick_distance_dev, (nj ** 3,), "|u1"))
    if c["prec"] == E4M3:
        nbo = -(-k // lay.offset_brick)
        out["scales"] = at(lay.scales_dev, (1 + 3 * D,), "<f4")
        out["offsets"] = at(lay.offsets_dev, (nbo ** 3, lay.offset_stride), "<f2")
    if lay.layout:
        out["pages"] = at(lay.page_table_dev, (nb ** 3,), "<i4")
    return out


def run(st):
    c, ctx = st["case"], st["context"].handle
    kind = c["kind"]
    if kind in ("view", "walk"):
        fnr.fnr_render(ctx, st["cache"].handle, st["cams"], st["params"], st["rgba"], st["stats"])
        return dict(rgba=st["rgba"], stats=st["stats"])
    if kind == "serve":
        tickets = [fnr.fnr_submit(ctx, fnr.make_request(st["cache"].handle, cam, st["params"], out))
                   for cam, out in zip(st["cams"], st["rgba"])]
        for t in tickets:
            if fnr.fnr_wait(ctx, t, 60000).status != fnr.FNR_OK:
                raise RuntimeError("a request failed")
        return st["rgba"]
    if kind == "uncached":
        fnr.fnr_render_mlp(ctx, *st["nets"], c["D"], st["cams"][0], st["params"], st["rgba"], st["stats"])
        return dict(rgba=st["rgba"])
    st["cache"] = None  # the cache of the pass before makes room for the new one
    if kind == "mlp":
        built = fnr.fnr_build_cache_mlp(ctx, st["desc"], *st["nets"])
    else:
        built = fnr.fnr_build_cache(ctx, st["desc"], *st["arrays"])
    st["cache"] = _Cache(st["context"], built)
    return _stored(c, st["cache"])


# ------------------------------------------------------------------ what a pass cannot do without
def _layer_flops(dims):
    return 2.0 * sum(a * b for a, b in zip(dims[:-1], dims[1:]))


def _pos_flops(D):
    return _layer_flops([6 * POS_FREQS] + [256] * 8 + [1 + 3 * D])


def _dir_flops(D):
    return _layer_flops([6 * DIR_FREQS] + [128] * 4 + [D])


def work(case):
    c, D = case, case["D"]
    kind = c["kind"]
    es = {FP32: 4, FP16: 2, E4M3: 1}[c.get("prec", FP32)]
    eb = 4 if c.get("prec", FP32) == FP32 else 2
    if kind == "mlp":
        n, m = c["k"] ** 3, c["l"] ** 2
        return dict(bytes=n * (1 + 3 * D) * es + m * D * eb, flops=n * _pos_flops(D) + m * _dir_flops(D))
    if kind == "arrays":
        n, m = c["k"] ** 3, c["l"] ** 2
        kept = 0.2 if c["layout"] else 1.0  # about a fifth of the bricks of this scene family hold density
        return dict(bytes=n * (1 + 3 * D) * (4 + kept * es) + m * D * (4 + eb), flops=4.0 * n * 3 * D)
    if kind == "serve":
        rays = sum(RESOLUTIONS[i % len(RESOLUTIONS)][0] * RESOLUTIONS[i % len(RESOLUTIONS)][1]
                   for i in range(c["requests"]))
    else:
        rays = c["W"] * c["H"] * c.get("views", 1)
    if kind == "uncached":
        inside = 0.71 * c["N"] * rays  # samples inside the box, of this camera family
        return dict(bytes=16.0 * rays, flops=inside * (_pos_flops(D) + 6 * D) + rays * _dir_flops(D))
    # per ray of this scene family, as counted on the benchmark's views: densities looked up and samples shaded
    if kind == "walk":
        looked, shaded = (0.11 if c["skip"] else 0.93) * c["k"], 0.057 * c["k"]
    else:
        looked, shaded = (0.054 if c.get("skip") or c.get("layout") else 0.47) * c["N"], 0.029 * c["N"]
    per_ray = looked * es + shaded * 3 * D * es + D * eb + 16 + (16 if c.get("stats") else 0)
    return dict(bytes=rays * per_ray, flops=rays * (shaded * (6 * D + 20) + looked * 6))


# ------------------------------------------------------------------ the same in 64 bits
def _fma(a, b, c):
    return (a.double() * b.double() + torch.as_tensor(c).double()).float()


def _rays(cam):
    """Unit directions [H * W, 3] in binary32 by the library's documented sequence, and the eye."""
    W, H = cam["W"], cam["H"]
    f = lambda v: torch.tensor(float(v), device="cuda", dtype=torch.float32)
    px = torch.arange(W, device="cuda", dtype=torch.float32).repeat(H)
    py = torch.arange(H, device="cuda", dtype=torch.float32).repeat_interleave(W)
    dx = ((px + 0.5) - f(cam["cx"])) / f(cam["fx"])
    dy = -(((py + 0.5) - f(cam["cy"])) / f(cam["fy"]))
    m = cam["c2w"]
    w = [_fma(f(m[4 * r]), dx, _fma(f(m[4 * r + 1]), dy, -f(m[4 * r + 2]))) for r in range(3)]
    n = _fma(w[0], w[0], _fma(w[1], w[1], w[2] * w[2])).sqrt()
    return torch.stack([v / n for v in w], 1), [f(m[3]), f(m[7]), f(m[11])]


def _direction_cell(d, l):
    j = torch.arange(1, l, device="cuda", dtype=torch.float64)
    ct = torch.cos(j * math.pi / l).float()

    def key(x, y):
        zero = (x == 0) & (y == 0)
        q = torch.where(y >= 0, torch.where(x >= 0, y / (x + y), 1 + (-x) / (y + (-x))),
                        torch.where(x < 0, 2 + (-y) / ((-x) + (-y)), 3 + x / (x + (-y))))
        return torch.where(zero, torch.zeros_like(q), q)

    a = 2 * math.pi * j / l
    it = torch.searchsorted((-ct).contiguous(), (-d[:, 2]).contiguous(), right=True)  # #{dz <= cos_j}
    ip = torch.searchsorted(key(a.cos(), a.sin()).float().contiguous(), key(d[:, 0], d[:, 1]).contiguous(),
                            right=True)
    return it * l + ip


def _ray_beta(c, d, beta):
    """Direction weights [rays, D] in 64 bits, nearest bin or bilinear."""
    l = c["l"]
    b = (beta if c["prec"] == FP32 else beta.half()).reshape(l * l, -1)
    if not c.get("bilinear"):
        return b[_direction_cell(d, l)].double()
    v = d.double()
    u = torch.atan2(torch.hypot(v[:, 0], v[:, 1]), v[:, 2]) * (l / math.pi) - 0.5
    w = torch.remainder(torch.atan2(v[:, 1], v[:, 0]), 2 * math.pi) * (l / (2 * math.pi)) - 0.5
    fu, fw = u.floor(), w.floor()
    a, e = (u - fu)[:, None], (w - fw)[:, None]
    i0, i1 = fu.long().clamp(0, l - 1), (fu.long() + 1).clamp(0, l - 1)
    j0, j1 = fw.long() % l, (fw.long() + 1) % l
    at = lambda i, j: b[i * l + j].double()
    return (1 - a) * ((1 - e) * at(i0, j0) + e * at(i0, j1)) + a * ((1 - e) * at(i1, j0) + e * at(i1, j1))


def _e4m3(v):
    return v.clamp(-448, 448).to(torch.float8_e4m3fn).float()


def _as_stored(c, sigma, uvw):
    """The values a cache of the case's precision holds (binary32 arithmetic as documented)."""
    k, nch = c["k"], 3 * c["D"]
    if c["prec"] == FP32:
        return sigma, uvw.reshape(-1, nch)
    if c["prec"] == FP16:
        return sigma.half(), uvw.reshape(-1, nch).half()
    s0 = sigma.max() / 448
    s0 = torch.where(s0 > 0, s0, torch.ones_like(s0))
    Bo = 4
    while -(-k // Bo) > 64:
        Bo *= 2
    nb = -(-k // Bo)
    u = uvw.reshape(k, k, k, nch)
    out = torch.empty_like(u)
    brick = (torch.arange(k, device="cuda") // Bo)
    mids = []
    for c0 in range(nch):  # channel by channel: bounded temporaries
        g = torch.nn.functional.pad(u[..., c0], (0, nb * Bo - k) * 3, value=math.nan)
        g = g.reshape(nb, Bo, nb, Bo, nb, Bo)
        lo = torch.nan_to_num(g, nan=math.inf).amin((1, 3, 5))
        hi = torch.nan_to_num(g, nan=-math.inf).amax((1, 3, 5))
        mids.append(((lo + hi) * 0.5).half().float())
        m = mids[-1][brick][:, brick][:, :, brick]
        r = u[..., c0] - m
        s = r.abs().max() / 448
        s = torch.where(s > 0, s, torch.ones_like(s))
        out[..., c0] = (m.double() + s.double() * _e4m3(r / s).double()).float()
    return _e4m3(sigma / s0) * s0, out.reshape(-1, nch)


def _shade(c, beta, rec):
    x = (beta[:, None, :] * rec.reshape(rec.shape[0], 3, c["D"]).double()).sum(2)
    return 1 / (1 + torch.exp(-x))


class _Blend:
    """Eq. 1 per ray in 64 bits, with the exact integer termination."""

    def __init__(self, n, thr):
        z = lambda: torch.zeros(n, device="cuda", dtype=torch.float64)
        self.T, self.C, self.thr = z() + 1, torch.zeros((n, 3), device="cuda", dtype=torch.float64), thr
        self.S = z().long()
        self.live = torch.ones(n, device="cuda", dtype=torch.bool)

    def add(self, at, sigma, length, colour, depth):
        """Rays `at` pass one sample of density sigma over `length`."""
        e = torch.exp(-sigma.double() * length.double())
        self.C[at] += (self.T[at] * (1 - e))[:, None] * colour
        self.T[at] *= e
        self.S[at] += (depth.double() * 4294967296.0).floor().long()
        self.live[at] = self.S[at] < self.thr

    def rgba(self):
        return torch.cat([self.C + self.T[:, None], 1 - self.T[:, None]], 1).reshape(-1)


def _grid_line(d, o, k):
    """g_a(t) = t u_a + w_a in binary32: u [rays, 3], w [3]."""
    s = torch.tensor(k / (HI - LO), device="cuda", dtype=torch.float64).float()
    return d * s, torch.stack([(v - LO) * s for v in o])


def _view64(c, cam, stored, beta):
    k, N = c["k"], c["N"]
    sigma, rec = stored
    d, o = _rays(cam)
    u, w = _grid_line(d, o, k)
    dt = (torch.tensor(FAR, device="cuda") - torch.tensor(NEAR, device="cuda")) / N
    e, f = u * dt, _fma(torch.tensor(NEAR, device="cuda"), u, w)
    b = _ray_beta(c, d, beta)
    blend = _Blend(d.shape[0], math.ceil(math.log(1.0 / np.float64(np.float32(THR))) / float(dt) * 2.0 ** 32))
    for i in range(N):
        g = _fma(torch.tensor(i + 0.5, device="cuda"), e, f).floor()
        at = (((g >= 0) & (g < k)).all(1) & blend.live).nonzero()[:, 0]
        q = g[at].long()
        cell = (q[:, 2] * k + q[:, 1]) * k + q[:, 0]
        s = sigma[cell].float()
        hit = (s > 0).nonzero()[:, 0]
        at, cell, s = at[hit], cell[hit], s[hit]
        blend.add(at, s, dt.expand(len(at)), _shade(c, b[at], rec[cell]), s)
    return blend.rgba()


def _walk64(c, cam, stored, beta):
    k = c["k"]
    sigma, rec = stored
    d, o = _rays(cam)
    u, w = _grid_line(d, o, k)
    b = _ray_beta(c, d, beta)
    w = w.expand_as(u)
    lo, hi = (-w) / u, (float(k) - w) / u
    lo, hi = torch.minimum(lo, hi), torch.maximum(lo, hi)
    still = u == 0
    out = (still & ~((w >= 0) & (w < k))).any(1)
    lo, hi = lo.masked_fill(still, -math.inf), hi.masked_fill(still, math.inf)
    t = lo.amax(1).clamp(min=NEAR)
    t1 = hi.amin(1).clamp(max=FAR)
    blend = _Blend(d.shape[0], math.ceil(math.log(1.0 / np.float64(np.float32(THR))) * 2.0 ** 32))
    blend.live &= (t < t1) & ~out
    cell = _fma(t[:, None], u, w).floor().clamp(0, k - 1)
    step = torch.where(u > 0, 1.0, -1.0)

    def crossing(cc):
        return ((torch.where(u > 0, cc + 1, cc) - w) / u).masked_fill(still, math.inf)

    for _ in range(3 * k):
        tn, axis = crossing(cell).min(1)  # the first smallest: x, then y, then z
        length = torch.minimum(tn, t1) - t
        idx = cell.long()
        idx = (idx[:, 2] * k + idx[:, 1]) * k + idx[:, 0]
        at = (blend.live & (length > 0)).nonzero()[:, 0]
        if not len(at) and not bool(blend.live.any()):
            break
        s = sigma[idx[at]].float()
        hit = (s > 0).nonzero()[:, 0]
        at, s = at[hit], s[hit]
        blend.add(at, s, length[at], _shade(c, b[at], rec[idx[at]]), s * length[at])
        moved = cell + torch.nn.functional.one_hot(axis, 3) * step
        blend.live &= (tn < t1) & ((moved >= 0) & (moved < k)).all(1)
        cell = torch.where(blend.live[:, None], moved, cell)
        t = torch.maximum(t, tn)
    return blend.rgba()


def _encode64(x, freqs):
    """sin / cos(2^j pi x) per coordinate, rounded to bf16 as the network's input is."""
    q = x.double()[:, :, None] * (2.0 ** torch.arange(freqs, device="cuda", dtype=torch.float64)) * math.pi
    return torch.stack([q.sin(), q.cos()], -1).reshape(x.shape[0], -1).to(torch.bfloat16).double()


def _network64(layers, x, freqs):
    """The network in 64 bits with bf16 inputs to every layer."""
    out = []
    for part in x.split(1 << 18):
        h = _encode64(part, freqs)
        for i, (W, b) in enumerate(layers):
            h = h @ W.double().T + b.double()
            if i + 1 < len(layers):
                h = h.clamp(min=0).to(torch.bfloat16).double()
        out.append(h)
    return torch.cat(out)


#: 64-bit arithmetic runs at about 1 TFLOP/s on this GPU: networks over more work than this are not evaluated in it
_FLOPS64 = 6e12


def _mlp64(c, nets):
    k, l = c["k"], c["l"]
    h = np.float32((HI - LO) / k)
    g = _fma(torch.arange(k, device="cuda", dtype=torch.float32) + 0.5, torch.tensor(float(h), device="cuda"), LO)
    z, y, x = torch.meshgrid(g, g, g, indexing="ij")
    out = _network64(nets[0], torch.stack([x, y, z], -1).reshape(-1, 3), POS_FREQS)
    th = (torch.arange(l, device="cuda", dtype=torch.float64) + 0.5) * (math.pi / l)
    ph = (torch.arange(l, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / l)
    v = torch.stack([th.sin()[:, None] * ph.cos(), th.sin()[:, None] * ph.sin(), th.cos()[:, None].expand(l, l)], -1)
    beta = _network64(nets[1], v.reshape(-1, 3), DIR_FREQS).reshape(l, l, -1)
    return dict(sigma=out[:, 0].clamp(min=0), uvw=out[:, 1:], beta=beta, occupancy=None, distance=None)


def _uncached64(c, nets, cam):
    D, N = c["D"], c["N"]
    d, o = _rays(cam)
    dt = (torch.tensor(FAR, device="cuda") - torch.tensor(NEAR, device="cuda")) / N
    beta = _network64(nets[1], d, DIR_FREQS)
    blend = _Blend(d.shape[0], math.ceil(math.log(1.0 / np.float64(np.float32(THR))) / float(dt) * 2.0 ** 32))
    for i in range(N):
        t = _fma(torch.tensor(i + 0.5, device="cuda"), dt, torch.tensor(NEAR, device="cuda"))
        p = torch.stack([_fma(t, d[:, a], o[a]) for a in range(3)], 1)
        at = (((p >= LO) & (p < HI)).all(1) & blend.live).nonzero()[:, 0]
        if not len(at):
            continue
        out = _network64(nets[0], p[at], POS_FREQS)
        hit = (out[:, 0] > 0).nonzero()[:, 0]
        at, out = at[hit], out[hit]
        blend.add(at, out[:, 0], dt.expand(len(at)), _shade(c, beta[at], out[:, 1:]), out[:, 0].float())
    return dict(rgba=blend.rgba())


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "arrays":
        return None  # stored bytes: they are equal or they are not
    if kind in ("mlp", "uncached") and work(c)["flops"] > _FLOPS64:
        return None
    d = _inputs(c, seed)
    if kind == "mlp":
        return _mlp64(c, d["nets"])
    if kind == "uncached":
        return _uncached64(c, d["nets"], d["cams"][0])
    sigma, uvw, beta = d["arrays"]
    stored = _as_stored(c, sigma, uvw)
    del uvw, d["arrays"]
    images = [(_walk64 if kind == "walk" else _view64)(c, cam, stored, beta) for cam in d["cams"]]
    return images if kind == "serve" else dict(rgba=torch.cat(images), stats=None)
