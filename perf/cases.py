"""Performance cases: what a program does with this library, over the range of sizes, formats
and filters it is used for.

A case is a dict of plain values; its "kind" names the entry point:

  filter  apply_filter on one volume (handles and filter kept, as a program that filters a
          stream of volumes keeps them): separable or dense, any pair of voxel formats, whole
          volume or a region
  batch   apply_filter_batch over a mixed set of small volumes
  train   apply_filter_autograd, forward and backward, over a batch of float32 volumes
  clahe   clahe3d
  render  render
  bricks  brick_decompose

Inputs are synthetic: CT-like volumes (Gaussian blobs and noise, quantised to the integer
formats), a turbulence-like float32 field (64 Fourier modes), random kernels.
"""
import math

import numpy as np
import torch

import paper_2203_10213_gb300 as vkt

SIZE = {"u8": 1, "u16": 2, "f32": 4}
QMAX = {"u8": 255, "u16": 65535}
DTYPE = {"u8": torch.uint8, "u16": torch.uint16, "f32": torch.float32}


# ------------------------------------------------------------------ the cases

def _filter(name, dims, src, dst, weights, k, roi=0.0):
    """roi: the region's share of each axis (0: the whole volume)."""
    c = {"kind": "filter", "nx": dims[0], "ny": dims[1], "nz": dims[2], "src": src, "dst": dst,
         "weights": weights, "k": k, "roi": roi}
    return {"name": name, **c} if name else c


def listed():
    return [
        # an interactive preview or a simulation's small block: one launch, latency counts
        _filter("small_dense3_f32", (64, 64, 64), "f32", "f32", "gauss_dense", 3),
        # denoising a scan in its own format; rows of 302 bytes, as the paper's Heptane volume has
        _filter("scan302_gauss5_u8", (302, 302, 302), "u8", "u8", "gauss", 5),
        # the benchmark's workload: a blur and an edge filter of a CT volume into float32
        _filter("ct512_gauss5_u8_f32", (512, 512, 512), "u8", "f32", "gauss", 5),
        _filter("ct512_laplace3_u8_f32", (512, 512, 512), "u8", "f32", "laplace", 3),
        # denoising a 16-bit scan in its own format
        _filter("ct_gauss5_u16", (512, 512, 256), "u16", "u16", "gauss", 5),
        # a user's own dense kernel on an 8-bit scan, in its own format
        _filter("ct256_kernel5_u8", (256, 256, 256), "u8", "u8", "random", 5),
        # a wide dense kernel on a large simulation field
        _filter("dns_kernel7_f32", (1024, 1024, 512), "f32", "f32", "random", 7),
        # many small volumes of mixed sizes, formats and filters in one call
        {"name": "batch128_mixed", "kind": "batch", "n": 128, "dmin": 16, "dmax": 256, "recipe": 1},
        # one training step of a learnable kernel: forward, input and weight gradients
        {"name": "train8_128_k5", "kind": "train", "batch": 8, "nx": 128, "ny": 128, "nz": 128, "k": 5},
        # the paper's CLAHE case study size
        {"name": "clahe256", "kind": "clahe", "bx": 8, "by": 8, "bz": 8, "sx": 32, "sy": 32, "sz": 32,
         "clip": 2.0},
        # one frame of a CT volume
        {"name": "render512", "kind": "render", "src": "u8", "nx": 512, "ny": 512, "nz": 512,
         "width": 1024, "height": 768, "step": 0.5},
        # splitting a volume into bricks with the ghost cells a 5^3 filter needs
        {"name": "bricks512", "kind": "bricks", "src": "u8", "nx": 512, "ny": 512, "nz": 512, "bx": 128,
         "by": 128, "bz": 128, "ghost": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["filter"] * 7 + ["batch", "train", "clahe", "render", "bricks"])
    if kind == "filter":
        src = rng.choice(["u8", "u8", "u16", "f32"])
        dst = rng.choice(["f32", src])
        weights = rng.choice(["gauss", "gauss", "random", "laplace", "gauss_dense"])
        k = 3 if weights in ("laplace", "gauss_dense") else rng.choice([3, 5, 7, 9] if weights == "gauss" else [3, 5, 7])
        # up to the size of the largest listed volume for float32 results; dense kernels into
        # integer formats up to what costs as much
        most = 1 << 28
        if weights != "gauss":
            most = min(most, int(9e10 / k ** 3) if dst == "f32" else int(4e9 / k ** 3))
        while True:
            dims = tuple(_log(rng, 24, 900) for _ in range(3))
            if rng.random() < 0.5:
                dims = (max(32, dims[0] // 32 * 32),) + dims[1:]
            if 1 << 15 <= dims[0] * dims[1] * dims[2] <= most:
                break
        roi = round(rng.uniform(0.4, 0.9), 2) if rng.random() < 0.2 else 0.0
        return _filter("", dims, src, dst, weights, k, roi)
    if kind == "batch":
        return {"kind": "batch", "n": _log(rng, 16, 128), "dmin": 16, "dmax": rng.choice([64, 128, 256]),
                "recipe": rng.randrange(1000)}
    if kind == "train":
        return {"kind": "train", "batch": rng.randint(1, 8), "nx": 4 * rng.randint(8, 40),
                "ny": rng.randint(32, 150), "nz": rng.randint(32, 128), "k": rng.choice([3, 5, 7])}
    if kind == "clahe":
        return {"kind": "clahe", "bx": rng.randint(4, 10), "by": rng.randint(4, 10), "bz": rng.randint(3, 8),
                "sx": rng.randint(12, 48), "sy": rng.randint(12, 40), "sz": rng.randint(8, 32),
                "clip": rng.choice([0.0, 1.5, 2.0, 4.0])}
    if kind == "render":
        return {"kind": "render", "src": rng.choice(["u8", "u16", "f32"]), "nx": _log(rng, 64, 512),
                "ny": _log(rng, 64, 512), "nz": _log(rng, 64, 512), "width": rng.randint(200, 1024),
                "height": rng.randint(150, 768), "step": rng.choice([0.5, 0.75, 1.0])}
    return {"kind": "bricks", "src": rng.choice(["u8", "u16", "f32"]), "nx": 16 * rng.randint(8, 30),
            "ny": _log(rng, 60, 400), "nz": _log(rng, 60, 400), "bx": 16 * rng.randint(8, 12),
            "by": rng.randint(100, 160), "bz": rng.randint(100, 160), "ghost": rng.choice([0, 1, 2, 3])}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _blobs(g, nx, ny, nz, noise=0.02):
    """CT-like float32 field in [0, 1]: 32 Gaussian blobs (sigma 8 to 64 voxels in a volume of
    512^3, in proportion in others) and noise."""
    r = torch.rand((5, 32), generator=g, device="cuda")
    sigma, amp = (8.0 + 56.0 * r[3]) * ((nx * ny * nz) ** (1.0 / 3.0) / 512.0), 0.2 + 0.8 * r[4]
    ex, ey, ez = (torch.exp(-0.5 * ((torch.arange(n, device="cuda") - r[a, :, None] * n) / sigma[:, None]) ** 2)
                  for a, n in ((0, nx), (1, ny), (2, nz)))
    out = torch.empty((nz, ny, nx), device="cuda")
    for z0 in range(0, nz, 64):
        zs = ez[:, z0:z0 + 64] * amp[:, None]
        v = (zs[:, :, None] * ey[:, None, :]).reshape(32, -1).t() @ ex
        v = v.reshape(-1, ny, nx)
        v += noise * torch.randn(v.shape, generator=g, device="cuda")
        out[z0:z0 + 64] = v.clamp_(0.0, 1.0)
    return out


def _fourier(g, nx, ny, nz):
    """Turbulence-like float32 field: 64 modes, amplitude |k|^(-5/3)."""
    r = torch.rand((2, 64), generator=g, device="cuda")
    d = torch.randn((3, 64), generator=g, device="cuda")
    kk = 1.0 + 31.0 * r[0]
    d = d / d.norm(dim=0) * kk * (2.0 * math.pi)
    ax, ay, az = (d[a][:, None] * (torch.arange(n, device="cuda") / n) for a, n in ((0, nx), (1, ny), (2, nz)))
    az = az + 2.0 * math.pi * r[1][:, None]
    amp = kk ** (-5.0 / 3.0)
    b = torch.cat([amp[:, None] * torch.cos(ax), -amp[:, None] * torch.sin(ax)])
    out = torch.empty((nz, ny, nx), device="cuda")
    for z0 in range(0, nz, 64):
        zy = az[:, z0:z0 + 64, None] + ay[:, None, :]
        a = torch.cat([torch.cos(zy), torch.sin(zy)]).reshape(128, -1)
        out[z0:z0 + 64] = (a.t() @ b).reshape(-1, ny, nx)
    return out


def _volume(g, fmt, nx, ny, nz, field="blobs"):
    v = _fourier(g, nx, ny, nz) if field == "fourier" else _blobs(g, nx, ny, nz)
    if fmt == "f32":
        return v
    q = v.mul_(QMAX[fmt]).add_(0.5).floor_()
    return q.to(torch.uint8) if fmt == "u8" else q.to(torch.int32).to(torch.uint16)


def _gauss(k, sigma):
    """The sampled Gaussian, normalised in 64 bits, as float32."""
    d = np.arange(k) - (k - 1) // 2
    e = np.exp(-(d * d) / (2.0 * float(np.float32(sigma)) ** 2))
    return (e / e.sum()).astype(np.float32)


def _weights(case, seed):
    """(the three vectors or None, the dense k^3 float32 weights or None)"""
    k, kind = case["k"], case["weights"]
    if kind == "gauss":
        g = _gauss(k, 0.3 * k)
        return (g, g, g), None
    if kind == "gauss_dense":
        g = _gauss(k, 1.0).astype(np.float64)
        return None, (g[:, None, None] * g[None, :, None] * g[None, None, :]).astype(np.float32)
    if kind == "laplace":
        w = np.zeros((3, 3, 3), np.float32)
        w[1, 1, 1] = -6.0
        w[0, 1, 1] = w[2, 1, 1] = w[1, 0, 1] = w[1, 2, 1] = w[1, 1, 0] = w[1, 1, 2] = 1.0
        return None, w
    w = np.random.RandomState(1000 + seed % 100000).standard_normal((k, k, k)) + 0.5
    return None, (w / w.sum()).astype(np.float32)


def _ranges(case):
    """Value ranges of source and destination: a Laplacian has negative results."""
    return (0.0, 1.0), ((-1.0, 1.0) if case["weights"] == "laplace" else (0.0, 1.0))


def _roi(case):
    if not case["roi"]:
        return None
    lo, hi = [], []
    for n in (case["nx"], case["ny"], case["nz"]):
        s = max(1, int(n * case["roi"]))
        lo.append((n - s) // 3)
        hi.append((n - s) // 3 + s)
    return tuple(lo), tuple(hi)


def _batch_items(case):
    """Dims, formats and Gaussian filters of the volumes of a batch (the same for every seed)."""
    r = np.random.RandomState(case["recipe"])
    items = []
    for _ in range(case["n"]):
        d = np.exp(r.uniform(math.log(case["dmin"]), math.log(case["dmax"]), 3)).round().astype(int)
        items.append((tuple(int(x) for x in d), ("u8", "u16", "f32")[r.randint(3)], (3, 5, 7)[r.randint(3)]))
    return items


def _train_inputs(case, seed):
    g = _gen(seed)
    shape = (case["batch"], case["nz"], case["ny"], case["nx"])
    x = torch.stack([_blobs(g, case["nx"], case["ny"], case["nz"]) for _ in range(case["batch"])])
    w = 0.1 * torch.randn((case["k"],) * 3, generator=g, device="cuda")
    gy = torch.randn(shape, generator=g, device="cuda") * (2.0 / x.numel())
    return x, w, gy


def _render_inputs(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    v = _volume(_gen(seed), case["src"], nx, ny, nz)
    lut = np.array([[0.0, 0.0, 0.2, 0.0], [0.1, 0.4, 0.7, 0.005], [0.9, 0.6, 0.2, 0.02],
                    [1.0, 1.0, 0.9, 0.06]], np.float32)
    far = float(max(nx, ny, nz))
    cam = {"eye": (0.5 * nx, 0.5 * ny + 0.1 * far, -1.2 * far), "center": (0.5 * nx, 0.5 * ny, 0.5 * nz),
           "up": (0.0, 1.0, 0.0), "fovy": 0.8}
    return v, lut, cam


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    kind = case["kind"]
    if kind == "filter":
        src = _volume(_gen(seed), case["src"], case["nx"], case["ny"], case["nz"],
                      "fourier" if case["src"] == "f32" and case["dst"] == "f32" else "blobs")
        dst = torch.zeros(src.shape, dtype=DTYPE[case["dst"]], device="cuda")
        sep, dense = _weights(case, seed)
        srange, drange = _ranges(case)
        return {"kind": kind, "out": dst, "src": vkt.StructuredVolume.from_tensor(src, *srange),
                "dst": vkt.StructuredVolume.from_tensor(dst, *drange), "roi": _roi(case),
                "filter": vkt.Filter.separable(*sep) if sep else vkt.Filter.dense(dense)}
    if kind == "batch":
        g = _gen(seed)
        items = _batch_items(case)
        # the destinations of each format lie in one buffer, each on a 16-byte boundary
        total = {f: 0 for f in SIZE}
        offsets = []
        for (nx, ny, nz), fmt, _ in items:
            offsets.append(total[fmt])
            total[fmt] += -(-nx * ny * nz // 16) * 16
        out = {f: torch.zeros(max(n, 1), dtype=DTYPE[f], device="cuda") for f, n in total.items()}
        srcs, dsts, filters = [], [], []
        for ((nx, ny, nz), fmt, k), o in zip(items, offsets):
            srcs.append(vkt.StructuredVolume.from_tensor(_volume(g, fmt, nx, ny, nz)))
            dsts.append(vkt.StructuredVolume.from_tensor(out[fmt][o:o + nx * ny * nz].view(nz, ny, nx)))
            filters.append(vkt.Filter.gaussian(k, k / 3.0))
        return {"kind": kind, "out": out, "srcs": srcs, "dsts": dsts, "filters": filters}
    if kind == "train":
        x, w, gy = _train_inputs(case, seed)
        return {"kind": kind, "x": x.requires_grad_(), "w": w.requires_grad_(), "gy": gy}
    if kind == "clahe":
        v = _volume(_gen(seed), "u8", case["bx"] * case["sx"], case["by"] * case["sy"], case["bz"] * case["sz"])
        return {"kind": kind, "src": v, "out": torch.empty_like(v), "bricks": (case["bx"], case["by"], case["bz"]),
                "clip": case["clip"]}
    if kind == "render":
        v, lut, cam = _render_inputs(case, seed)
        return {"kind": kind, "src": v, "lut": lut, "cam": cam, "width": case["width"], "height": case["height"],
                "step": case["step"],
                "out": torch.empty((case["height"], case["width"], 4), dtype=torch.float32, device="cuda")}
    v = _volume(_gen(seed), case["src"], case["nx"], case["ny"], case["nz"])
    return {"kind": kind, "src": v, "brick": (case["bx"], case["by"], case["bz"]), "ghost": case["ghost"]}


def _bits(t):
    """uint16 codes as int16, which torch can index; the same bytes."""
    return t.view(torch.int16) if t.dtype == torch.uint16 else t


def run(state):
    kind = state["kind"]
    if kind == "filter":
        vkt.apply_filter(state["dst"], state["src"], state["filter"], roi=state["roi"])
        return _bits(state["out"])
    if kind == "batch":
        vkt.apply_filter_batch(state["dsts"], state["srcs"], state["filters"])
        return {f: _bits(t) for f, t in state["out"].items()}
    if kind == "train":
        y = vkt.apply_filter_autograd(state["x"], state["w"])
        gx, gw = torch.autograd.grad(y, (state["x"], state["w"]), state["gy"])
        return {"y": y.detach(), "gx": gx, "gw": gw}
    if kind == "clahe":
        return vkt.clahe3d(state["src"], state["bricks"], state["clip"], out=state["out"])
    if kind == "render":
        c = state["cam"]
        return vkt.render(state["src"], state["width"], state["height"], c["eye"], c["center"], c["up"], c["fovy"],
                          state["step"], state["lut"], out=state["out"])
    return [_bits(t) for t in vkt.brick_decompose(state["src"], state["brick"], state["ghost"])]


# ------------------------------------------------------------------ what a pass cannot do without

def _ray_samples(case):
    """About how many samples a frame of _render_inputs' camera takes: the rays through a grid
    of pixels, clipped to the volume."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    far = float(max(nx, ny, nz))
    o = np.array([0.5 * nx, 0.5 * ny + 0.1 * far, -1.2 * far])
    f = np.array([0.5 * nx, 0.5 * ny, 0.5 * nz]) - o
    f /= np.linalg.norm(f)
    r = np.cross(f, [0.0, 1.0, 0.0])
    r /= np.linalg.norm(r)
    u = np.cross(r, f)
    t = math.tan(0.4)
    s = np.linspace(-0.98, 0.98, 50)
    d = f + s[None, :, None] * t * case["width"] / case["height"] * r + s[:, None, None] * t * u
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    a, b = -o / d, (np.array([nx, ny, nz]) - o) / d
    near, last = np.minimum(a, b).max(-1).clip(0), np.maximum(a, b).min(-1)
    return float((last - near).clip(0).mean()) / case["step"] * case["width"] * case["height"]


def work(case):
    kind = case["kind"]
    if kind == "filter":
        lo, hi = _roi(case) or ((0, 0, 0), (case["nx"], case["ny"], case["nz"]))
        n = math.prod(b - a for a, b in zip(lo, hi))
        k = case["k"]
        return {"bytes": n * (SIZE[case["src"]] + SIZE[case["dst"]]),
                "flops": n * 2 * (3 * k if case["weights"] == "gauss" else 7 if case["weights"] == "laplace" else k ** 3)}
    if kind == "batch":
        items = [(math.prod(d), SIZE[f], k) for d, f, k in _batch_items(case)]
        return {"bytes": sum(2 * n * s for n, s, _ in items), "flops": sum(n * 6 * k for n, _, k in items)}
    if kind == "train":
        n = case["batch"] * case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 16 * n, "flops": 6 * n * case["k"] ** 3}
    if kind == "clahe":
        n = case["bx"] * case["by"] * case["bz"] * case["sx"] * case["sy"] * case["sz"]
        return {"bytes": 2 * n, "flops": 14 * n}
    if kind == "render":
        return {"bytes": case["nx"] * case["ny"] * case["nz"] * SIZE[case["src"]] + 16 * case["width"] * case["height"],
                "flops": 60 * _ray_samples(case)}
    n, m = case["nx"] * case["ny"] * case["nz"], 1
    for d, b in (("nx", "bx"), ("ny", "by"), ("nz", "bz")):
        m *= case[d] + 2 * case["ghost"] * -(-case[d] // case[b])
    return {"bytes": SIZE[case["src"]] * (n + m), "flops": 0}


# ------------------------------------------------------------------ the results in 64 bits

def _axis(v, w, dim):
    """One clamped 1-D pass along dim."""
    r, n = (len(w) - 1) // 2, v.shape[dim]
    at = torch.arange(n, device=v.device)
    out = torch.zeros_like(v)
    for i, x in enumerate(w):
        out.add_(v.index_select(dim, (at + i - r).clamp_(0, n - 1)), alpha=float(x))
    return out


def _separable64(v, g):
    for dim, w in ((2, g[0]), (1, g[1]), (0, g[2])):
        v = _axis(v, w, dim)
    return v


def _dense64(v, w):
    """The clamped correlation, in slabs of z."""
    k = w.shape[0]
    r = (k - 1) // 2
    nz, ny, nx = v.shape
    out = torch.empty_like(v)
    at = torch.arange(-r, nz + r, device=v.device).clamp_(0, nz - 1)
    for z0 in range(0, nz, 128):
        z1 = min(z0 + 128, nz)
        p = torch.nn.functional.pad(v[at[z0:z1 + 2 * r]][None, None], (r, r, r, r, 0, 0), mode="replicate")[0, 0]
        o = out[z0:z1].zero_()
        for c in range(k):
            for b in range(k):
                for a in range(k):
                    if w[c, b, a] != 0:
                        o.add_(p[c:c + z1 - z0, b:b + ny, a:a + nx], alpha=float(w[c, b, a]))
    return out


def _values64(t, fmt):
    return t.double() if fmt == "f32" else t.to(torch.int32).double() / QMAX[fmt]


def _filter64(case, seed):
    if case["dst"] != "f32":
        return None
    src = _volume(_gen(seed), case["src"], case["nx"], case["ny"], case["nz"],
                  "fourier" if case["src"] == "f32" else "blobs")
    v = _values64(src, case["src"])
    sep, dense = _weights(case, seed)
    full = _separable64(v, sep) if sep else _dense64(v, dense)
    roi = _roi(case)
    if roi is None:
        return full
    (x0, y0, z0), (x1, y1, z1) = roi
    out = torch.zeros_like(full)
    out[z0:z1, y0:y1, x0:x1] = full[z0:z1, y0:y1, x0:x1]
    return out


def _batch64(case, seed):
    g, parts = _gen(seed), [torch.zeros(0, dtype=torch.float64, device="cuda")]
    for (nx, ny, nz), fmt, k in _batch_items(case):
        v = _volume(g, fmt, nx, ny, nz)
        if fmt == "f32":
            w = _gauss(k, k / 3.0)
            o = _separable64(v.double(), (w, w, w)).reshape(-1)
            parts.append(torch.nn.functional.pad(o, (0, -o.numel() % 16)))
    flat = torch.cat(parts)
    return {"u8": None, "u16": None, "f32": flat if flat.numel() else torch.zeros_like(flat).new_zeros(1)}


def _train64(case, seed):
    x, w, gy = (t.double() for t in _train_inputs(case, seed))
    k = case["k"]
    r = (k - 1) // 2
    nz, ny, nx = x.shape[1:]
    x.requires_grad_()
    p = torch.nn.functional.pad(x[:, None], (r,) * 6, mode="replicate")[:, 0]
    pd = p.detach()
    y, gp, gw = torch.zeros_like(gy), torch.zeros_like(pd), torch.zeros_like(w)
    for c in range(k):
        for b in range(k):
            for a in range(k):
                s = (slice(None), slice(c, c + nz), slice(b, b + ny), slice(a, a + nx))
                y += w[c, b, a] * pd[s]
                gp[s] += w[c, b, a] * gy
                gw[c, b, a] = (pd[s] * gy).sum()
    return {"y": y, "gx": torch.autograd.grad(p, x, gp)[0], "gw": gw}


def _render64(case, seed):
    """Ray marching: one pass over the sample index, all pixels at once."""
    t, lut, cam = _render_inputs(case, seed)
    vol = (t if case["src"] != "u16" else t.to(torch.int32)).reshape(-1)
    scale = 1.0 if case["src"] == "f32" else 1.0 / QMAX[case["src"]]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    W, H, step = case["width"], case["height"], float(np.float32(case["step"]))
    dev, f64 = "cuda", torch.float64
    vec = lambda v: np.asarray(v, np.float32).astype(np.float64)  # noqa: E731
    o, f = vec(cam["eye"]), vec(cam["center"]) - vec(cam["eye"])
    f /= np.linalg.norm(f)
    r = np.cross(f, vec(cam["up"]))
    r /= np.linalg.norm(r)
    u = np.cross(r, f)
    th = math.tan(float(np.float32(cam["fovy"])) / 2)
    px = (2 * (torch.arange(W, device=dev, dtype=f64) + 0.5) / W - 1) * th * W / H
    py = (1 - 2 * (torch.arange(H, device=dev, dtype=f64) + 0.5) / H) * th
    d = [(f[a] + px[None, :] * r[a] + py[:, None] * u[a]).reshape(-1) for a in range(3)]
    norm = (d[0] ** 2 + d[1] ** 2 + d[2] ** 2).sqrt()
    d = [x / norm for x in d]
    near, last = torch.zeros_like(norm), torch.full_like(norm, math.inf)
    for a, n in enumerate((nx, ny, nz)):
        lo, hi = (0.0 - o[a]) / d[a], (n - o[a]) / d[a]
        near, last = torch.maximum(near, torch.minimum(lo, hi)), torch.minimum(last, torch.maximum(lo, hi))
    out = torch.zeros((W * H, 4), dtype=f64, device=dev)
    rays = torch.nonzero(last > near)[:, 0]
    d, near, last = [x[rays] for x in d], near[rays], last[rays]
    table = torch.from_numpy(lut).to(dev).double()
    C = torch.zeros((rays.numel(), 4), dtype=f64, device=dev)
    k = 0
    while True:
        tt = near + (k + 0.5) * step
        live = tt < last
        if not bool(live.any()):
            break
        i0, i1, w = [], [], []
        for a, n in enumerate((nx, ny, nz)):
            q = o[a] + tt * d[a] - 0.5
            b = q.floor()
            w.append(q - b)
            i0.append(b.long().clamp_(0, n - 1))
            i1.append((b.long() + 1).clamp_(0, n - 1))
        v = torch.zeros_like(tt)
        for cz, wz in ((i0[2], 1 - w[2]), (i1[2], w[2])):
            for cy, wy in ((i0[1], 1 - w[1]), (i1[1], w[1])):
                base, wzy = (cz * ny + cy) * nx, wz * wy
                v += wzy * ((1 - w[0]) * vol[base + i0[0]].double() + w[0] * vol[base + i1[0]].double())
        p = (v * scale).clamp_(0, 1) * (lut.shape[0] - 1)
        e = p.floor().long().clamp_(0, lut.shape[0] - 2)
        s = torch.lerp(table[e], table[e + 1], (p - e)[:, None])
        alpha = 1 - (1 - s[:, 3]) ** step
        add = torch.cat([s[:, :3] * alpha[:, None], alpha[:, None]], 1) * (1 - C[:, 3:])
        C += torch.where(live[:, None], add, torch.zeros_like(add))
        k += 1
    out[rays] = C
    return out.reshape(H, W, 4)


def exact(case, seed):
    kind = case["kind"]
    if kind == "filter":
        return _filter64(case, seed)
    if kind == "batch":
        return _batch64(case, seed)
    if kind == "train":
        return _train64(case, seed)
    if kind == "render":
        return _render64(case, seed)
    return None   # codes and copies
