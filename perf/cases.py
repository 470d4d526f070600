"""Performance cases of the neural-texture decode.

Each case is one whole call of ``Decoder.decode`` (device buffers) or
``Decoder.decode_host`` (host buffers): bucketing by decoder, gather, MLP, output
rows in the caller's order.  ``listed()`` names the calls a renderer makes in
earnest; ``draw()`` gives more of the same ranges (query counts, set and decoder
counts, grid sizes, shapes, types, addressing).

Inputs are drawn on the GPU from the seed: latents N(0, 0.5) in fp16 with box-filtered
mip chains, Xavier-uniform weights, a balanced random set -> decoder map, and query
streams of three kinds -- texel-centre rasters, uniform random queries, and
G-buffers (Voronoi regions in 8x4-pixel tile order, an affine UV map each).

``exact()`` evaluates the same decode in 64 bits with torch alone.  Texel
coordinates and the bilinear and mip fractions are the decode's defined fp32
round-to-nearest expressions; everything after them (blend, encoding, MLP,
sigmoid) is fp64.
"""
import math

import numpy as np
import torch

from paper_2608_27888_gb300 import ntc
from paper_2608_27888_gb300 import workloads as W

# Every field of a case, with the default it has when a case does not name it.
DEFAULTS = dict(
    stream="gbuffer",   # raster | uniform | gbuffer
    n=0,                # queries of a uniform stream
    width=0, height=0,  # screen of a raster or G-buffer stream, any size
    frames=1, regions=200,
    lod="round",        # G-buffer: "round" = integer mip from the texel density, "real" = U[0, 3) per region
    sets=1, T=256, mips=1, decoders=1,
    levels=2, channels=8, pe=0,
    hidden=64, layers=2, leaky=False, out_dim=8,
    clamp=False, precision="fp16", output="fp32", host=False,
)


def full(case):
    return dict(DEFAULTS, **{k: v for k, v in case.items() if k != "name"})


def listed():
    return [
        # the smallest calls: a batch of ray hits or feedback probes, a few hundred
        # queries of random sets; launches and latency are the whole cost
        dict(name="probe-1k-uniform", stream="uniform", n=1013, sets=16, T=256, mips=1, decoders=16),
        # one 256^2 texture transcoded through its decoder (single set, nothing to sort)
        dict(name="raster-256", stream="raster", width=256, height=256, sets=1, T=256),
        # incoherent secondary-ray shading: uniform set ids and UVs, a decoder per set
        dict(name="uniform-4m", stream="uniform", n=4194304, sets=16, T=1024, decoders=16),
        # a 1080p shading pass, non-shared baseline: one decoder per set
        dict(name="gbuffer-1080p-identity", width=1920, height=1080, sets=32, T=1024, mips=4, decoders=32),
        # the same pass with clustered decoders, bf16 operands, fp16 rows, clamped UVs
        dict(name="gbuffer-1080p-clustered-bf16", width=1920, height=1080, sets=32, T=1024, mips=4, decoders=4,
             precision="bf16", output="fp16", clamp=True),
        # the 586-texture library with a decoder per texture: many small buckets
        dict(name="gbuffer-1080p-586-decoders", width=1920, height=1080, regions=600, sets=586, T=512, mips=4,
             decoders=586),
        # a 2160p pass over 2k textures, nine output channels
        dict(name="gbuffer-2160p-8", width=3840, height=2160, regions=800, sets=64, T=2048, mips=4, decoders=8,
             out_dim=9),
        # the largest: four 2160p frames, trilinear, wide decoders
        dict(name="gbuffer-2160p-x4-trilinear", width=3840, height=2160, frames=4, regions=2000, lod="real", sets=128,
             T=2048, mips=4, decoders=8, hidden=128, out_dim=9),
        # host buffers in and out: an offline or remote renderer's frame, fp16 rows
        dict(name="gbuffer-2160p-host", width=3840, height=2160, regions=2000, lod="real", sets=32, T=2048, mips=4,
             decoders=8, hidden=128, out_dim=9, output="fp16", host=True),
        # the decoder of the paper's experiments: 256^2 x 4 grid, encoding, LeakyReLU, 64 x 3
        dict(name="paper-decoder-1080p", width=1920, height=1080, lod="real", sets=16, T=256, mips=4, decoders=4,
             levels=1, channels=4, pe=4, leaky=True, out_dim=9),
        # its widest, deepest size of the MLP ablation, bf16, on an odd-sized view
        dict(name="paper-128x5-bf16", width=1283, height=717, lod="real", sets=16, T=256, mips=4, decoders=4, levels=1,
             channels=4, pe=4, leaky=True, hidden=128, layers=4, out_dim=9, precision="bf16"),
        # fp32 throughout: reference renders
        dict(name="gbuffer-1080p-fp32", width=1920, height=1080, sets=32, T=1024, mips=4, decoders=4,
             precision="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["standard"] * 5 + ["general"] * 3 + ["fp32", "host"])
    n = _log_int(rng, 600, {"standard": 24e6, "general": 4e6, "fp32": 1.2e6, "host": 6e6}[kind])
    c = dict(stream=rng.choice(["uniform", "gbuffer", "gbuffer", "gbuffer", "raster"]))
    if c["stream"] == "uniform":
        c["n"] = n
    else:
        c["width"] = max(5, min(8000, int(round(math.sqrt(n * rng.uniform(0.5, 2.0))))))
        c["height"] = max(5, n // c["width"])
        if c["stream"] == "gbuffer":
            c["regions"] = rng.randint(3, 1200)
            c["lod"] = rng.choice(["round", "real"])
    c["sets"] = _log_int(rng, 1, 600)
    c["decoders"] = c["sets"] if rng.random() < 0.3 else _log_int(rng, 1, c["sets"])
    c["T"] = _log_int(rng, 64, max(65, min(2048, int(math.sqrt(48e6 / c["sets"])))))
    c["mips"] = rng.choice([1, 2, 4, 4])
    c["out_dim"] = rng.choice([1, 3, 4, 8, 8, 9, 9, 12, 16])
    c["clamp"] = rng.random() < 0.3
    if kind == "fp32":
        c["precision"] = "fp32"
    else:
        c["precision"] = rng.choice(["fp16", "fp16", "bf16"])
        c["output"] = rng.choice(["fp32", "fp32", "fp16"])
    c["host"] = kind == "host"
    if kind == "general":
        c.update(levels=rng.choice([1, 1, 2]), channels=rng.choice([4, 4, 8]), pe=rng.randint(0, 6),
                 leaky=rng.random() < 0.8, hidden=rng.choice([16, 32, 64, 64, 128]), layers=rng.randint(1, 4))
    else:
        c["hidden"] = rng.choice([64, 64, 128])
    return c


# ------------------------------------------------------------------------ inputs

def count(c):
    return c["n"] if c["stream"] == "uniform" else c["width"] * c["height"] * c["frames"]


def in_dim(c):
    return c["levels"] * c["channels"] + 4 * c["pe"]


def grid_sizes(c):
    """Mip-0 edge of every latent level: half and a quarter of the texture; a single level keeps T."""
    return [c["T"]] if c["levels"] == 1 else [max(1, c["T"] // 2), max(1, c["T"] // 4)]


def _latents(c, g):
    """fp16 [sets, texels of a set * channels]: level by level, mip by mip, channel-last."""
    parts = []
    for e in grid_sizes(c):
        m = torch.randn((c["sets"], e, e, c["channels"]), generator=g, device="cuda", dtype=torch.float16) * 0.5
        parts.append(m.reshape(c["sets"], -1))
        for _ in range(1, c["mips"]):
            e = max(1, e // 2)
            f = m.float().permute(0, 3, 1, 2)
            f = torch.nn.functional.avg_pool2d(f, (2, 2)) if f.shape[-1] > 1 else f
            m = f.permute(0, 2, 3, 1).half()
            parts.append(m.reshape(c["sets"], -1))
    return torch.cat(parts, 1)


def _layers(c):
    H = c["hidden"]
    dims = [in_dim(c)] + [H] * c["layers"] + [c["out_dim"]]
    return list(zip(dims[:-1], dims[1:]))


def _weights(c, g):
    """fp32 [decoders, parameters]: per layer W [out][in] Xavier-uniform, b U(+-1/sqrt(in))."""
    parts = []
    for i, o in _layers(c):
        for k, a in ((o * i, math.sqrt(6.0 / (i + o))), (o, 1.0 / math.sqrt(i))):
            parts.append((torch.rand((c["decoders"], k), generator=g, device="cuda") * 2.0 - 1.0) * a)
    return torch.cat(parts, 1)


def _screen(w, h):
    """Pixel coordinates in emission order: 8x4-pixel tiles, row-major inside a tile."""
    tx, ty = -(-w // 8), -(-h // 4)
    k = torch.arange(tx * ty * 32, device="cuda")
    tile, p = k // 32, k % 32
    x, y = (tile % tx) * 8 + p % 8, (tile // tx) * 4 + p // 8
    inside = (x < w) & (y < h)
    return x[inside], y[inside]


def _gbuffer(c, g, x, y):
    w, R = c["width"], c["regions"]

    def rand():
        return torch.rand(R, generator=g, device="cuda", dtype=torch.float64)

    sx, sy = (rand() * w).floor().float(), (rand() * c["height"]).floor().float()
    sid = torch.randint(c["sets"], (R,), generator=g, device="cuda")
    scale, th, ou, ov, real = 1.0 + 7.0 * rand(), 2.0 * math.pi * rand(), rand(), rand(), 3.0 * rand()
    lod = real if c["lod"] == "real" else (torch.log2(scale * c["T"] / w).clamp(min=0.0) + 0.5).floor()
    near = torch.empty(len(x), dtype=torch.int64, device="cuda")
    step = max(1, (1 << 27) // R)
    for b in range(0, len(x), step):
        px, py = x[b:b + step].float()[:, None], y[b:b + step].float()[:, None]
        near[b:b + step] = ((px - sx) ** 2 + (py - sy) ** 2).argmin(1)
    q = torch.empty((len(x), 4), dtype=torch.float32, device="cuda")
    px, py = (x.double() + 0.5) / w, (y.double() + 0.5) / w
    s, co, si = scale[near], torch.cos(th)[near], torch.sin(th)[near]
    q[:, 1] = (s * (co * px - si * py) + ou[near]).float()
    q[:, 2] = (s * (si * px + co * py) + ov[near]).float()
    q[:, 3] = lod[near].float()
    q.view(torch.int32)[:, 0] = sid[near].int()
    return q


def _queries(c, g):
    """int32 [n, 4] records on the GPU: set id, then the bits of u, v, lod."""
    if c["stream"] == "uniform":
        q = torch.zeros((c["n"], 4), dtype=torch.float32, device="cuda")
        q[:, 1:3] = torch.rand((c["n"], 2), generator=g, device="cuda")
        q.view(torch.int32)[:, 0] = torch.randint(c["sets"], (c["n"],), generator=g, device="cuda").int()
        return q.view(torch.int32)
    x, y = _screen(c["width"], c["height"])
    if c["stream"] == "raster":
        q = torch.zeros((len(x), 4), dtype=torch.float32, device="cuda")
        q[:, 1], q[:, 2] = (x.float() + 0.5) / c["width"], (y.float() + 0.5) / c["height"]
        q.view(torch.int32)[:, 0] = int(torch.randint(c["sets"], (1,), generator=g, device="cuda"))
        return q.view(torch.int32)
    return torch.cat([_gbuffer(c, g, x, y) for _ in range(c["frames"])]).view(torch.int32)


def _inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    lat, wts, q = _latents(c, g), _weights(c, g), _queries(c, g)
    cmap = torch.empty(c["sets"], dtype=torch.int64, device="cuda")  # balanced random partition
    cmap[torch.randperm(c["sets"], generator=g, device="cuda")] = torch.arange(c["sets"], device="cuda") % c["decoders"]
    return lat, wts, cmap, q


def prepare(case, seed):
    """The context a program keeps (latents, weights and map uploaded), a batch of queries and its output rows."""
    c = full(case)
    lat, wts, cmap, q = _inputs(c, seed)
    sizes = grid_sizes(c)
    dims, offs, total = W.pyramid_layout(c["sets"], [[(e, e) for e in sizes]] * c["sets"], c["mips"])
    assert total * c["channels"] == lat.numel()
    a = W.Assets(num_sets=c["sets"], num_levels=c["levels"], num_mips=c["mips"], channels=c["channels"], level_dims=dims,
                 latent_offsets=offs, latents=lat.reshape(-1).cpu().numpy().view(np.uint16), num_decoders=c["decoders"],
                 in_dim=in_dim(c), hidden=c["hidden"], num_hidden_layers=c["layers"], out_dim=c["out_dim"],
                 weights=wts.cpu().numpy(), set_to_decoder=cmap.cpu().numpy().astype(np.uint32),
                 address_mode=int(c["clamp"]), pe_frequencies=c["pe"], activation=int(c["leaky"]), leaky_slope=0.01)
    del lat, wts
    dec = ntc.Decoder(a, c["precision"], c["output"])
    out = torch.empty((q.shape[0], c["out_dim"]), dtype=dec.out_dtype(), device="cpu" if c["host"] else "cuda",
                      pin_memory=c["host"])
    if c["host"]:
        q = q.cpu().pin_memory()
    return {"decoder": dec, "queries": q, "out": out, "host": c["host"]}


def run(state):
    if state["host"]:
        return state["decoder"].decode_host(state["queries"], state["out"])
    return state["decoder"].decode(state["queries"], state["out"])


# ----------------------------------------------------------- work and tolerance

def work(case):
    """Bytes: every record read and every row written once, the weights, and the latent texels a
    stream touches (a random query its own taps, up to the whole grids; a coherent one about
    one texel of every mip it blends, since neighbouring taps overlap)."""
    c = full(case)
    n = count(c)
    texel = 2 * c["channels"]
    total = sum(e * e for e in grid_sizes(c)) * c["sets"] * texel * (4 / 3 if c["mips"] > 1 else 1)
    if c["stream"] == "uniform":
        lat = total * (1.0 - math.exp(-n * 4 * c["levels"] * texel / total))
    else:
        lat = min(total, n * texel * (2 if c["lod"] == "real" and c["mips"] > 1 else 1))
    elem = 4 if c["precision"] == "fp32" else 2
    params = sum(i * o + o for i, o in _layers(c))
    row = c["out_dim"] * (2 if c["output"] == "fp16" else 4)
    return {"bytes": n * (16 + row) + lat + c["decoders"] * params * elem,
            "flops": 2.0 * n * sum(i * o for i, o in _layers(c))}


def tolerance(case):
    """Relative error another correct decode at the same precision shows: about four times
    what was measured against exact() (fp32 5e-8, with the sums in another order several times
    that; fp16 3e-5 to 9e-5, 2.2e-4 with fp16 rows; bf16 3.3e-4 to 6.6e-4)."""
    c = full(case)
    if c["precision"] == "fp32":
        return {"rel": 1e-6}
    if c["precision"] == "bf16":
        return {"rel": 2.6e-3}
    return {"rel": 1e-3 if c["output"] == "fp16" else 4e-4}


# ------------------------------------------------------------------------- exact

def _axis(x, e, clamp):
    """Texel pair and fraction of one axis, in the decode's fp32 round-to-nearest expressions."""
    x = (x if clamp else x - torch.floor(x)) * e - 0.5
    x0 = torch.floor(x)
    f = (x - x0).double()
    if clamp:
        i = x0.clamp(min=-1.0)
        i = torch.minimum(i, e).long()
        hi = e.long() - 1
        return torch.minimum(i.clamp(min=0), hi), torch.minimum((i + 1).clamp(min=0), hi), f
    i, n = x0.long(), e.long()
    return i % n, (i + 1) % n, f


def _features(c, lat, sid, u, v, lod):
    """fp64 [rows, in_dim]: each level's bilinear (two mips blended when the lod is fractional), then the encoding."""
    M, ch = c["mips"], c["channels"]
    lam = lod.clamp(min=0.0)
    lo = torch.floor(lam).clamp(max=M - 1)
    t = torch.where(lo == M - 1, torch.zeros_like(lam), lam - lo).double()
    lo = lo.long()
    per_set = lat.shape[1] // ch
    flat = lat.reshape(-1, ch)
    feats, base = [], 0
    for e0 in grid_sizes(c):
        edge = torch.tensor([max(1, e0 >> m) for m in range(M)], device="cuda")
        start = torch.cumsum(edge * edge, 0) - edge * edge + base
        base += int((edge * edge).sum())
        f = 0.0
        for k, wt in ((0, 1.0 - t), (1, t)):
            m = (lo + k).clamp(max=M - 1)
            e = edge[m].float()
            i0, i1, fx = _axis(u, e, c["clamp"])
            j0, j1, fy = _axis(v, e, c["clamp"])
            b, w = sid * per_set + start[m], edge[m]
            for i, j, wij in ((i0, j0, (1 - fx) * (1 - fy)), (i1, j0, fx * (1 - fy)), (i0, j1, (1 - fx) * fy),
                              (i1, j1, fx * fy)):
                f = f + (wij * wt)[:, None] * flat[b + j * w + i].double()
        feats.append(f)
    if c["pe"]:
        uu, vv = ((u, v) if c["clamp"] else (u - torch.floor(u), v - torch.floor(v)))
        for k in range(c["pe"]):
            for x in (uu.double(), vv.double()):
                a = 2.0 * math.pi * 2.0 ** k * x
                feats.append(torch.stack((torch.sin(a), torch.cos(a)), 1))
    return torch.cat(feats, 1)


def exact(case, seed):
    c = full(case)
    lat, wts, cmap, q = _inputs(c, seed)
    sid, f = q[:, 0].long(), q.view(torch.float32)
    out = torch.empty((q.shape[0], c["out_dim"]), dtype=torch.float64, device="cuda")
    dec = cmap[sid]
    order = torch.argsort(dec)
    ends = torch.cumsum(torch.bincount(dec, minlength=c["decoders"]), 0).tolist()
    del dec
    begin = 0
    for d, end in enumerate(ends):
        for b in range(begin, end, 1 << 19):
            at = order[b:min(end, b + (1 << 19))]
            x = _features(c, lat, sid[at], f[at, 1], f[at, 2], f[at, 3])
            o, last = 0, len(_layers(c)) - 1
            for k, (i, h) in enumerate(_layers(c)):
                w = wts[d, o:o + i * h].reshape(h, i).double()
                x = x @ w.T + wts[d, o + i * h:o + i * h + h].double()
                o += i * h + h
                if k < last:
                    x = torch.where(x > 0, x, x * (float(np.float32(0.01)) if c["leaky"] else 0.0))
            out[at] = torch.sigmoid(x)
        begin = end
    return out
