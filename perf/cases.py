"""What a program that uses this framework has it do, as measurable cases.

Each case is one call (or one short sequence of calls) of the public binding
``paper_1709_05418_gb300.api.Context``: renders, the stages of a render on their own
(descriptor rows, the network in its three arithmetics), training steps, label generation
and the per-volume preprocessing.  Sizes are those of the benchmark's workloads, the tests
and the paper's images, with ragged ones between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1709_05418_gb300 import api
from paper_1709_05418_gb300 import workloads as W

K, S, DIN, STRIDE, STRIDE8, H = api.K, api.S, api.DIN, api.DESC_STRIDE, api.DESC_STRIDE_FP8, api.H
NP = api.NPARAMS
FLOP_ROW = 2 * (10 * 226 * 200 + 9 * 200 * 200 + 10 * 200 * 200 + 2 * 200 * 200 + 200)
PREC = {"f32": api.F32, "bf16": api.BF16, "fp8": api.FP8}
DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.uint8}


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # a thumbnail of a small cloud with the default arithmetic: launches and latency
        {"name": "render_thumb_f32", "kind": "render", "cloud": "blob", "nx": 64, "ny": 64, "nz": 64,
         "grid": "f32", "width": 64, "height": 64, "spp": 1, "prec": "f32", "mode": "rpnn"},
        # the benchmark's render: 256^3 cloud, 512 x 512, tensor-core network
        {"name": "render_512_bf16", "kind": "render", "cloud": "fbm", "nx": 256, "ny": 256, "nz": 256,
         "grid": "f32", "width": 512, "height": 512, "spp": 1, "prec": "bf16", "mode": "rpnn"},
        # a final frame at the paper's image size from a large FP16 grid, several samples a pixel
        {"name": "render_720p_bf16", "kind": "render", "cloud": "fbm", "nx": 384, "ny": 288, "nz": 352,
         "grid": "f16", "width": 1280, "height": 720, "spp": 3, "prec": "bf16", "mode": "rpnn"},
        # the plain path tracer a prediction is judged by
        {"name": "render_path", "kind": "render", "cloud": "fbm", "nx": 160, "ny": 128, "nz": 192,
         "grid": "f32", "width": 256, "height": 192, "spp": 1, "prec": "f32", "mode": "path"},
        # descriptors of training records: FP32 rows, a light direction of its own for each query
        {"name": "descriptors_f32", "kind": "desc", "cloud": "fbm", "nx": 160, "ny": 192, "nz": 144,
         "rows": 30011, "dtype": "f32"},
        # the network on its own, in the default arithmetic (validation loss, FP32 renders)
        {"name": "network_f32", "kind": "net", "rows": 20011, "prec": "f32"},
        # ... on the tensor cores
        {"name": "network_bf16", "kind": "net", "rows": 100003, "prec": "bf16"},
        # ... with E4M3 operands
        {"name": "network_fp8", "kind": "net", "rows": 65536, "prec": "fp8"},
        # a training step in the default arithmetic on a small ragged minibatch
        {"name": "train_f32", "kind": "train", "rows": 1000, "prec": "f32"},
        # the benchmark's training step: mixed precision, 4,096 BF16 records
        {"name": "train_bf16", "kind": "train", "rows": 4096, "prec": "bf16"},
        # a new density in the same volume (a frame of an animation): statistics, majorants and
        # pyramid, then descriptors from it
        {"name": "volume_256", "kind": "volume", "cloud": "fbm", "nx": 256, "ny": 256, "nz": 256, "rows": 1000},
        # path-traced training labels (Sec. 5.1's stopping rule under a path cap)
        {"name": "records", "kind": "records", "cloud": "fbm", "nx": 128, "ny": 160, "nz": 128,
         "rows": 1024, "n_min": 64, "n_max": 1024},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    return {"cloud": rng.choice(["blob", "fbm"]), "nx": _log(rng, lo, hi), "ny": _log(rng, lo, hi),
            "nz": _log(rng, lo, hi)}


def draw(rng):
    kind = rng.choice(["render", "render", "render", "path", "desc", "net", "net", "net", "train", "train",
                       "volume", "records"])
    if kind == "render":
        w = _log(rng, 48, 1280)
        return {"kind": kind, **_grid(rng, 48, 320), "grid": rng.choice(["f32", "f16"]), "width": w,
                "height": max(32, int(w * rng.uniform(0.5, 1.0))), "spp": rng.choice([1, 1, 2, 3]),
                "prec": rng.choice(["f32", "bf16", "bf16"]) if w <= 400 else "bf16", "mode": "rpnn"}
    if kind == "path":
        w = _log(rng, 48, 320)
        return {"kind": "render", **_grid(rng, 48, 200), "grid": rng.choice(["f32", "f16"]), "width": w,
                "height": max(32, int(w * rng.uniform(0.5, 1.0))), "spp": rng.choice([1, 2]), "prec": "f32",
                "mode": "path"}
    if kind == "desc":
        return {"kind": kind, **_grid(rng, 48, 256), "rows": _log(rng, 100, 100000),
                "dtype": rng.choice(["f32", "bf16", "fp8"])}
    if kind == "net":
        prec = rng.choice(["f32", "bf16", "fp8"])
        return {"kind": kind, "rows": _log(rng, 100, 60000 if prec == "f32" else 300000), "prec": prec}
    if kind == "train":
        return {"kind": kind, "rows": _log(rng, 128, 8192), "prec": rng.choice(["f32", "bf16"])}
    if kind == "volume":
        return {"kind": kind, **_grid(rng, 48, 320), "rows": _log(rng, 100, 3000)}
    return {"kind": kind, **_grid(rng, 48, 200), "rows": _log(rng, 64, 2048), "n_min": 64,
            "n_max": _log(rng, 128, 1024)}


# ------------------------------------------------------------------------------- inputs
def _density(case, seed):
    """Extinction grid [nz][ny][nx] on the GPU: a sum of Gaussian blobs, or a thresholded
    fractal-noise cloud (generated at half size and resampled where the grid is large)."""
    shape = (case["nz"], case["ny"], case["nx"])
    if case["cloud"] == "blob":
        n, m = max(shape), 96
        small = torch.from_numpy(W.blob_cloud(min(n, m), nblobs=8, seed=seed)).cuda()
    else:
        half = 2 if max(shape) > 288 else 1
        small = torch.from_numpy(W.fbm_cloud(seed=seed, shape=tuple((e + half - 1) // half for e in shape))).cuda()
    if tuple(small.shape) != shape:
        small = torch.nn.functional.interpolate(small[None, None], size=shape, mode="trilinear",
                                                align_corners=False)[0, 0]
    d = small.contiguous()
    return d.half() if case.get("grid") == "f16" else d


def _params(seed):
    """He-initialised parameters with small random biases."""
    p = W.he_init(seed=seed + 11)
    rng = np.random.default_rng(seed + 12)
    parts = W.split_params(p)
    for name in parts:
        if name.startswith("b"):
            parts[name] = rng.uniform(0.0, 0.05, size=parts[name].shape).astype(np.float32)
    return torch.from_numpy(W.join_params(parts).astype(np.float32)).cuda()


def _rows(n, seed, dtype):
    """Descriptor rows as shading points inside a cloud have them: densities around the mean
    near the point, more and more zeros on the coarse levels (outside the cloud), then the
    angle to the light and zero padding."""
    g = torch.Generator(device="cuda").manual_seed(seed + 21)
    z = torch.zeros((n, K, STRIDE), device="cuda")
    base = torch.rand((n, 1, 1), generator=g, device="cuda") + 0.4
    r = torch.randn((n, K, S), generator=g, device="cuda") * 0.7 + base
    inside = torch.tensor([0.95, 0.9, 0.8, 0.6, 0.4, 0.25, 0.1, 0.03, 0.01, 0.005], device="cuda")
    keep = torch.rand((n, K, S), generator=g, device="cuda") < inside[None, :, None]
    z[:, :, :S] = torch.relu(r) * keep
    z[:, :, S] = torch.acos(torch.rand((n, 1), generator=g, device="cuda") * 2.0 - 1.0)
    if dtype == torch.uint8:
        out = torch.zeros((n, K, STRIDE8), device="cuda")
        out[:, :, :STRIDE] = z
        return out.to(torch.float8_e4m3fn).view(torch.uint8)
    return z.to(dtype)


def _queries(shape, n, seed):
    """Shading points inside the grid, tracing directions and light directions (FP32)."""
    x, d = W.random_queries(shape, n, seed=seed + 31)
    _, wl = W.random_queries(shape, n, seed=seed + 32)
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()  # noqa: E731
    return f(x), f(d), f(wl)


def prepare(case, seed):
    kind = case["kind"]
    ctx = api.Context()
    s = {"case": case, "ctx": ctx}
    if kind in ("render", "desc", "volume", "records"):
        dens = _density(case, seed)
        s["vol"] = ctx.load_volume(dens, albedo=0.99, hg_g=0.85)
        ctx.build_mips(s["vol"])
    if kind == "render":
        ctx.set_weights(_params(seed))
        s["cam"] = W.camera(tuple(dens.shape), case["width"], case["height"], spp=case["spp"], seed=seed + 3,
                            light_seed=seed + 4)
    elif kind in ("desc", "volume"):
        s["x"], s["d"], s["wl"] = _queries(tuple(dens.shape), case["rows"], seed)
    elif kind == "net":
        ctx.set_weights(_params(seed))
        s["z"] = _rows(case["rows"], seed, DTYPE[case["prec"]])
        if case["prec"] == "fp8":
            ctx.calibrate_fp8(_rows(2048, seed + 1, torch.float32))
    elif kind == "train":
        s.update(_train_state(case, seed))
        ctx.set_train_precision(PREC[case["prec"]])
        ctx.set_weights(s["p"])
        s["loss"] = torch.empty(1, dtype=torch.float64, device="cuda")
    elif kind == "records":
        s["seed"] = seed + 41
    return s


def _train_state(case, seed):
    """A resumed run: parameters, Adam moments of a thousand earlier steps, a minibatch."""
    g = torch.Generator(device="cuda").manual_seed(seed + 51)
    p = _params(seed)
    return {"p": p, "z": _rows(case["rows"], seed, DTYPE[case["prec"]]),
            "t": torch.rand(case["rows"], generator=g, device="cuda") * 2.0,
            "m": torch.randn(NP, generator=g, device="cuda") * 1e-4,
            "v": torch.rand(NP, generator=g, device="cuda") * 1e-6 + 1e-8, "step": 1000}


# ------------------------------------------------------------------------------- one pass
def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "render":
        mode = api.MODE_PATH if case["mode"] == "path" else api.MODE_RPNN
        return ctx.render(s["vol"], s["cam"], precision=PREC[case["prec"]], mode=mode)
    if kind == "desc":
        return ctx.extract_descriptors(s["vol"], s["x"], s["d"], s["wl"], dtype=DTYPE[case["dtype"]])
    if kind == "net":
        return ctx.mlp_forward(s["z"], precision=PREC[case["prec"]])
    if kind == "train":
        s["step"] += 1
        ctx.train_step(s["z"], s["t"], s["p"], s["m"], s["v"], s["step"], lr=1e-4, loss=s["loss"])
        return {"loss": s["loss"], "p": s["p"], "m": s["m"], "v": s["v"]}
    if kind == "volume":
        ctx.build_mips(s["vol"])
        info = ctx.get_volume_info(s["vol"])
        return {"mean": info["mean"], "majorant": info["majorant"], "nonzero": info["nonzero"],
                "bricks": ctx.copy_brick_majorants(s["vol"]),
                "desc": ctx.extract_descriptors(s["vol"], s["x"], s["d"], s["wl"])}
    x, d, wl, label, npaths = ctx.gen_records(s["vol"], 0, case["rows"], s["seed"], rel_ci=0.02,
                                              n_min=case["n_min"], n_max=case["n_max"])
    return {"x": x, "d": d, "wl": wl, "label": label, "npaths": npaths}


# ------------------------------------------------------------------------------- what it needs
def work(case):
    kind = case["kind"]
    vox = case.get("nx", 0) * case.get("ny", 0) * case.get("nz", 0)
    if kind == "render":
        # the grid and the weights in, the image out; about two thirds of the samples meet the cloud
        q = 0.65 * case["width"] * case["height"] * case["spp"]
        b = vox * 4 + case["width"] * case["height"] * 4
        if case["mode"] == "path":
            return {"bytes": b, "flops": 0}
        return {"bytes": b + NP * (4 if case["prec"] == "f32" else 2), "flops": q * FLOP_ROW}
    if kind == "desc":
        size = {"f32": 4, "bf16": 2, "fp8": 1}[case["dtype"]]
        width = STRIDE8 if case["dtype"] == "fp8" else STRIDE
        return {"bytes": case["rows"] * (K * width * size + 36), "flops": case["rows"] * K * S * 23}
    if kind == "net":
        size = {"f32": 4, "bf16": 2, "fp8": 1}[case["prec"]]
        width = STRIDE8 if case["prec"] == "fp8" else STRIDE
        return {"bytes": case["rows"] * (K * width * size + 4) + NP * size, "flops": case["rows"] * FLOP_ROW}
    if kind == "train":
        size = 4 if case["prec"] == "f32" else 2
        return {"bytes": case["rows"] * (K * STRIDE * size + 4) + NP * 4 * 6, "flops": 3 * case["rows"] * FLOP_ROW}
    if kind == "volume":
        return {"bytes": vox * 4 + vox // 512 * 4 + case["rows"] * (K * STRIDE * 4 + 36), "flops": vox * 7 * 2}
    return {"bytes": vox * 4 + case["rows"] * 44, "flops": 0}


# ------------------------------------------------------------------------------- in 64 bits
def _net64(p, z):
    """The network of the flat parameters p on rows z [n][10][...], in FP64 torch."""
    off = 0

    def take(*shape):
        nonlocal off
        n = math.prod(shape)
        t = p[off:off + n].reshape(shape)
        off += n
        return t

    o = None
    for k in range(K):
        V = take(H, DIN)
        W1 = take(H, H) if k else None
        b1, W2, b2 = take(H), take(H, H), take(H)
        f = z[:, k, :DIN] @ V.t() + b1
        if k:
            f = f + o @ W1.t()
        f = torch.relu(f) @ W2.t() + b2
        o = torch.relu(f if o is None else f + o)
    for n in (H, H, 1):
        T, b = take(n, H), take(n)
        o = torch.relu(o @ T.t() + b)
    return o[:, 0]


def _e4m3(z):
    return z.view(torch.float8_e4m3fn).double()


def _filter64(n, level):
    """Matrix [ceil(n / 2^level)][n] of the level's Gaussian (sigma = 2^level voxels, cut at
    three sigma, normalised, zero outside the grid) along one axis."""
    sig = 2.0 ** level
    m = -(-n // 2 ** level)
    c = (torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) * sig - 0.5
    i = torch.arange(n, dtype=torch.float64, device="cuda")
    d = i[None, :] - c[:, None]
    w = torch.exp(-d * d / (2.0 * sig * sig)) * (d.abs() <= 3.0 * sig + 1e-9)
    r = math.floor(3.0 * sig) + 1
    t = torch.arange(-r, r + 1, dtype=torch.float64) + (0.0 if level == 0 else 0.5)
    t = t[t.abs() <= 3.0 * sig]
    return w / float(torch.exp(-t * t / (2.0 * sig * sig)).sum())


def _mean64(dens):
    d = dens.double()
    return float(d.sum() / (d > 0).sum())


def _descriptors64(dens, x, d, wl):
    """Descriptor rows [q][10][240] in FP64 from the density grid."""
    nz, ny, nx = dens.shape
    nmax = max(nx, ny, nz)
    rho = dens.double() / _mean64(dens)
    mfp = 1.0 / _mean64(dens)
    levels = 1 + max(0, math.ceil(math.log2(nmax)))
    x, w, ez = x.double(), -d.double(), wl.double()
    ex = torch.linalg.cross(ez, w)
    ex = ex / ex.norm(dim=1, keepdim=True)
    ey = torch.linalg.cross(ez, ex)
    gamma = torch.acos((w * ez).sum(1).clamp(-1.0, 1.0))
    r = torch.arange(5, dtype=torch.float64, device="cuda") * 0.5 - 1.0
    oz, oy, ox = torch.meshgrid(torch.arange(9, dtype=torch.float64, device="cuda") * 0.5 - 1.0, r, r, indexing="ij")
    off = torch.stack([ox.flatten(), oy.flatten(), oz.flatten()], 1)
    out = torch.zeros((x.shape[0], K, STRIDE), dtype=torch.float64, device="cuda")
    mips = {}
    for k in range(K):
        sp = 0.5 * mfp * 2.0 ** k * nmax
        m = min(max(math.floor(math.log2(sp)), 0), levels - 1)
        if m not in mips:
            f = torch.einsum("ax,zyx->zya", _filter64(nx, m), rho)
            f = torch.einsum("by,zya->zba", _filter64(ny, m), f)
            f = torch.einsum("cz,zba->cba", _filter64(nz, m), f)
            mips[m] = torch.nn.functional.pad(f, (1, 1, 1, 1, 1, 1))
        f = mips[m]
        dims = torch.tensor([f.shape[2], f.shape[1], f.shape[0]], device="cuda")
        for a in range(0, x.shape[0], 4096):
            b = slice(a, min(a + 4096, x.shape[0]))
            p = (ex[b, None] * off[None, :, 0:1] + ey[b, None] * off[None, :, 1:2] + ez[b, None] * off[None, :, 2:3])
            u = (x[b, None] + p * (mfp * 2.0 ** k)) * (nmax / 2.0 ** m) + 0.5      # padded voxel coordinates
            inside = ((u >= 0.0) & (u < (dims - 1).double())).all(2)
            c = torch.minimum(u.clamp(min=0.0).floor().long(), dims - 2)
            t = (u - c).clamp(0.0, 1.0)
            v = torch.zeros(u.shape[:2], dtype=torch.float64, device="cuda")
            for corner in range(8):
                e = [(corner >> i) & 1 for i in range(3)]
                wt = 1.0
                for i in range(3):
                    wt = wt * (t[..., i] if e[i] else 1.0 - t[..., i])
                v += wt * f[c[..., 2] + e[2], c[..., 1] + e[1], c[..., 0] + e[0]]
            out[b, k, :S] = v * inside
            out[b, k, S] = gamma[b]
    return out


def _bricks64(dens):
    """Largest voxel of 8 b - 1 .. 8 b + 8 per axis, for every brick of 8^3 voxels."""
    v = dens.double()[None, None]
    n = [-(-e // 8) for e in dens.shape]
    pad = []
    for e, m in zip(reversed(dens.shape), reversed(n)):
        pad += [1, 8 * m + 1 - e]
    return torch.nn.functional.max_pool3d(torch.nn.functional.pad(v, pad), 10, stride=8)[0, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "net":
        z = _rows(case["rows"], seed, DTYPE[case["prec"]])
        p = _params(seed).double()
        n = 32768
        return torch.cat([_net64(p, _e4m3(c) if case["prec"] == "fp8" else c.double()) for c in z.split(n)])
    if kind == "train":
        s = _train_state(case, seed)
        p = s["p"].double().requires_grad_(True)
        g = _net64(p, s["z"].double())
        r = torch.log1p(g) - torch.log1p(s["t"].double())
        loss = (r * r).mean()
        loss.backward()
        b1, b2, eps, lr, step = 0.9, 0.999, 1e-8, 1e-4, s["step"] + 1
        m = b1 * s["m"].double() + (1.0 - b1) * p.grad
        v = b2 * s["v"].double() + (1.0 - b2) * p.grad * p.grad
        q = p.detach() - lr * (m / (1.0 - b1 ** step)) / ((v / (1.0 - b2 ** step)).sqrt() + eps)
        return {"loss": loss.detach().reshape(1), "p": q, "m": m, "v": v}
    if kind == "desc":
        dens = _density(case, seed)
        x, d, wl = _queries(tuple(dens.shape), case["rows"], seed)
        out = _descriptors64(dens, x, d, wl)
        # (E4M3 rows are bytes: compared as they are)
        return None if case["dtype"] == "fp8" else out
    if kind == "volume":
        dens = _density(case, seed)
        x, d, wl = _queries(tuple(dens.shape), case["rows"], seed)
        return {"mean": _mean64(dens), "majorant": float(dens.max()), "nonzero": int((dens > 0).sum()),
                "bricks": _bricks64(dens), "desc": _descriptors64(dens, x, d, wl)}
    # Monte Carlo images and labels: each value is a sum over random decisions made in FP32
    return None
