"""The library's work as its users call it, as cases that a timing program can
prepare, run and check: tiled global attention (GPA) forward and training
steps in BF16 and FP32, noise-gated attention, posterior-sampling steps, the
serving engine, temporal compression and factorised linear attention.

Sizes follow the workloads of ``paper_2604_16590_gb300/inputs.py`` (grids,
tilings, heads, input laws), with fewer heads or frames where the full
workload would take seconds.
"""
from __future__ import annotations

import math
import weakref

import torch

from paper_2604_16590_gb300 import gattn

# FP64 operations above which exact() gives no value (about 10 s of FP64 on this GPU).
EXACT_FLOPS = 6.0e12


def listed():
    return [
        # One 32 x 64 frame of patch tokens, 8 heads: the latency of a single inference call, where launches and
        # host work count (the smallest request of the serving workload has 8 such frames).
        gpa("frame_forward", 1, 8, 64, (1, 32, 64), (1, 16, 16), (0, 4, 4), train=False),
        # The plain method on a 64 x 64 frame (workload c1_4k): a training step of one FP32 head.
        gpa("frame_train_fp32", 1, 1, 64, (1, 64, 64), (1, 16, 16), (0, 4, 4), dtype="fp32"),
        # A short clip in FP32, tiles as wide as the paper regime's: the form used to check BF16 training.
        gpa("clip_train_fp32", 1, 4, 64, (4, 64, 128), (4, 16, 32), (0, 4, 8), dtype="fp32"),
        # The headline: 32 frames x 64 x 128, 16 tiles (workload c2_262k_p), one batch element of 16 heads.
        gpa("paper_train", 1, 16, 64, (32, 64, 128), (32, 16, 32), (0, 4, 8)),
        # The same grid in 1024 per-frame tiles (workload c2_262k_s): tiles of 24 x 24 tokens, four covers per token.
        gpa("small_tiles_train", 1, 16, 64, (32, 64, 128), (1, 16, 16), (0, 4, 4)),
        # Long temporal context at d = 128 (workload c3_4m_p): two of its 16 tiles of 128 frames, one head.
        gpa("long_train_d128", 1, 1, 128, (256, 32, 64), (128, 32, 64), (8, 0, 0)),
        # A regional crop whose extents are multiples of nothing: short last tiles and halos in all three dimensions.
        gpa("ragged_train_d128", 2, 6, 128, (7, 45, 77), (3, 14, 19), (1, 3, 5)),
        # The serving engine on a mix of requests (frames of 32 x 64 tokens, small tiles), 4 denoising steps each.
        serve("serve_mix", requests=6, t_min=8, t_max=96, steps=4),
        # Folding a history of 512 frames of 32 x 64 locations into one frame (workload h3_512).
        compress("compress_history", 1, 8, 128, 512, 2048),
        # Factorised linear attention over 262144 tokens, training step.
        linear("linear_train", 1, 16, 262144),
        # One posterior-sampling step of an 8-frame state: forward, likelihood gradient, update.
        dps("posterior_step", 1, 8, 64, (8, 64, 128), (1, 16, 16), (0, 4, 4)),
        # Self + cross attention of one current frame per batch element, blended by the noise gate.
        gated("gated_forward", 4, 16, 64, (1, 64, 128), (1, 16, 16), (0, 4, 4)),
    ]


# ---------------------------------------------------------------- the cases' plain values
def _tiled(kind, B, nh, d, grid, core, halo, dtype, window):
    c = {"kind": kind, "B": B, "nh": nh, "d": d, "dtype": dtype, "window": window}
    for a, n in enumerate("tyx"):
        c["grid_" + n], c["core_" + n], c["halo_" + n] = grid[a], core[a], halo[a]
    return c


def _named(c, name):
    return {"name": name, **c} if name else c


def gpa(name, B, nh, d, grid, core, halo, dtype="bf16", window="hann", train=True):
    return _named({**_tiled("gpa", B, nh, d, grid, core, halo, dtype, window), "train": train}, name)


def dps(name, B, nh, d, grid, core, halo, dtype="bf16"):
    return _named(_tiled("dps", B, nh, d, grid, core, halo, dtype, "hann"), name)


def gated(name, B, nh, d, grid, core, halo, dtype="bf16"):
    return _named(_tiled("gated", B, nh, d, grid, core, halo, dtype, "hann"), name)


def serve(name, requests, t_min, t_max, steps, d=64):
    return _named({"kind": "serve", "requests": requests, "t_min": t_min, "t_max": t_max, "steps": steps, "d": d}, name)


def compress(name, B, nh, d, S, M, dtype="bf16"):
    return _named({"kind": "compress", "B": B, "nh": nh, "d": d, "S": S, "M": M, "dtype": dtype}, name)


def linear(name, B, nh, N):
    return _named({"kind": "linear", "B": B, "nh": nh, "N": N}, name)


def _grid(c):
    return tuple(tuple(c[p + n] for n in "tyx") for p in ("grid_", "core_", "halo_"))


def _extents(G, core, halo):
    """(start, end) of every clipped extended tile along one dimension."""
    return [(max(0, k * core - halo), min(G, (k + 1) * core + halo)) for k in range(-(-G // core))]


def _pairs(c):
    """Query-key pairs of one (batch, head): the sum of the tiles' squared sizes."""
    return math.prod(sum((e - s) ** 2 for s, e in _extents(*a)) for a in zip(*_grid(c)))


def _frames(c):
    """(frames, heads) of a serving case's requests: frames in geometric steps, 8 and 16 heads in turn."""
    n = c["requests"]
    return [(round(c["t_min"] * (c["t_max"] / c["t_min"]) ** (i / max(1, n - 1))), 8 if i % 2 else 16) for i in range(n)]


SERVE_YX, SERVE_CORE, SERVE_HALO, SERVE_C = (32, 64), (1, 16, 16), (0, 4, 4), 0.5
SIGMA, SIGMA_NEXT, LAM, OBSERVED = 0.5, 0.45, 0.5, 0.25


def _serve_pairs(T):
    c = _tiled("gpa", 1, 1, 64, (T, *SERVE_YX), SERVE_CORE, SERVE_HALO, "bf16", "hann")
    return _pairs(c)


# ---------------------------------------------------------------- draws
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_tiled(rng, make, lo, hi, flops_per_pair, d, **kw):
    """A tiled case whose work lies near a log-uniform target in [lo, hi] operations."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    best = None
    for _ in range(400):
        per_frame = rng.random() < 0.5
        core = (1 if per_frame else _log_int(rng, 1, 32), _log_int(rng, 8, 32), _log_int(rng, 8, 48))
        halo = (0 if per_frame or rng.random() < 0.6 else rng.randint(0, max(0, core[0] // 2)),
                rng.randint(0, core[1] // 2), rng.randint(0, core[2] // 2))
        grid = (_log_int(rng, 1, 48), _log_int(rng, 16, 128), _log_int(rng, 24, 192))
        if rng.random() < 0.5:  # a grid the tiles divide
            grid = tuple(c * max(1, round(g / c)) for g, c in zip(grid, core))
        B, nh = rng.choice([1, 1, 2]), rng.choice([1, 2, 4, 6, 8, 16])
        case = make(None, B, nh, d, grid, core, halo, **kw)
        rows = math.prod(sum(e - s for s, e in _extents(*a)) for a in zip(*_grid(case)))
        flops = flops_per_pair * d * B * nh * _pairs(case)
        if flops > hi or B * nh * rows * d > 2.5e9:
            continue
        off = abs(math.log(flops / target))
        if best is None or off < best[0]:
            best = (off, case)
        if off < 0.3:
            break
    return best[1]


def draw(rng):
    kind = rng.choices(["bf16", "forward", "fp32", "gated", "dps", "serve", "compress", "linear"],
                       [8, 3, 3, 1, 1, 2, 2, 3])[0]
    if kind == "bf16":
        return _draw_tiled(rng, gpa, 1e10, 6e13, 12, rng.choice([64, 64, 128]), window=rng.choice(["hann"] * 4 + ["flat"]))
    if kind == "forward":
        return _draw_tiled(rng, gpa, 3e8, 2e13, 4, rng.choice([64, 64, 128]), train=False)
    if kind == "fp32":
        return _draw_tiled(rng, gpa, 3e9, 7e11, 12, rng.choice([32, 64, 64, 128]), dtype="fp32")
    if kind == "gated":
        return _draw_tiled(rng, gated, 1e10, 1e13, 8, rng.choice([64, 64, 128]))
    if kind == "dps":
        return _draw_tiled(rng, dps, 1e10, 1e13, 12, 64)
    if kind == "serve":
        t_min = _log_int(rng, 8, 24)
        return serve(None, rng.randint(1, 10), t_min, _log_int(rng, t_min, 96), rng.randint(2, 5))
    if kind == "compress":
        dtype = rng.choice(["bf16", "bf16", "fp32"])
        B, nh, d, M = rng.choice([1, 2]), rng.choice([2, 4, 8, 16]), rng.choice([64, 128]), _log_int(rng, 60, 4096)
        most = 4.3e9 / (2 * B * nh * M * d * (2 if dtype == "bf16" else 4))
        return compress(None, B, nh, d, _log_int(rng, 8, max(9, min(20000, most))), M, dtype)
    nh = rng.choice([1, 2, 4, 8, 16])
    return linear(None, rng.choice([1, 1, 2]), nh, _log_int(rng, 2000, min(1500000, 4194304 // nh // 2)))


# ---------------------------------------------------------------- inputs
DTYPE = {"bf16": torch.bfloat16, "fp32": torch.float32}


def _normal(gen, shape, std, dtype):
    t = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    return t.mul_(std).to(dtype)


def _inputs(case, seed):
    """The case's input tensors by name, from the seed alone (the laws of inputs.py: BF16 draws of std 0.5, FP32 of
    std 1, upstream gradients of std 1, learned queries FP32 of std 1)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    k = case["kind"]
    if k == "serve":
        return {"z%d" % i: _normal(gen, (nh, T * SERVE_YX[0] * SERVE_YX[1], case["d"]), 0.5, torch.bfloat16)
                for i, (T, nh) in enumerate(_frames(case))}
    dtype = DTYPE[case.get("dtype", "bf16")]
    std = 0.5 if dtype == torch.bfloat16 else 1.0
    if k == "compress":
        shape = tuple(case[n] for n in ("B", "nh", "S", "M", "d"))
        return {"k": _normal(gen, shape, std, dtype), "v": _normal(gen, shape, std, dtype),
                "q": _normal(gen, (case["nh"], case["d"]), 1.0, torch.float32)}
    if k == "linear":
        shape = (case["B"], case["nh"], case["N"], 64)
    else:
        shape = (case["B"], case["nh"], math.prod(_grid(case)[0]), case["d"])
    if k == "dps":
        z = _normal(gen, shape, 1.0, torch.float32)
        y = _normal(gen, shape, 1.0, torch.float32)
        eps = _normal(gen, shape, 1.0, torch.float32)
        mask = torch.rand((shape[0], shape[2]), generator=gen, device="cuda") < OBSERVED
        return {"z": z, "y": y, "eps": eps, "mask": mask.to(torch.uint8)}
    x = {n: _normal(gen, shape, std, dtype) for n in ("q", "k", "v")}
    if k == "gated":
        x.update({n: _normal(gen, shape, std, dtype) for n in ("kc", "vc")})
        x["gate"] = torch.rand(case["nh"], generator=gen, device="cuda")
    elif k == "linear" or case["train"]:
        x["dout"] = _normal(gen, shape, 1.0, dtype)
    return x


def _tiling(case):
    # the posterior sampler's synthetic denoiser runs at attention scale 1/d
    return gattn.Tiling(*_grid(case), window=case["window"], scale=1.0 / case["d"] if case["kind"] == "dps" else 0.0)


def prepare(case, seed):
    s = {"case": case, **_inputs(case, seed)}
    k = case["kind"]
    if k == "serve":
        s["server"] = gattn.Server(gattn.serve_cfg(
            d=case["d"], Y=SERVE_YX[0], X=SERVE_YX[1], core=SERVE_CORE, halo=SERVE_HALO, steps=case["steps"], c=SERVE_C,
            max_active=64, hbm_budget=60 * 10**9))
        weakref.finalize(s["server"], gattn.gattn_serve_destroy, s["server"].h)  # closed with the state
        s["states"] = [s.pop("z%d" % i) for i in range(case["requests"])]
        s["results"] = [torch.empty_like(z) for z in s["states"]]
        return s
    if k == "dps":
        s["sampler"] = gattn.PosteriorSampler(s["z"], _tiling(case), attn_dtype=case["dtype"])
    elif k != "compress":
        s["tiling"] = _tiling(case) if k != "linear" else None
    if "dout" in s:
        for n in ("q", "k", "v"):
            s[n].requires_grad_(True)
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "serve":
        srv = s["server"]
        ids = [srv.submit(z) for z in s["states"]]
        active = waiting = 1
        while active or waiting:
            active, waiting = srv.step()
        for rid, out in zip(ids, s["results"]):
            srv.result(rid, out=out)
        return list(s["results"])
    if k == "compress":
        out, lse = gattn.compress_forward(s["q"], s["k"], s["v"])
        return {"out": out, "lse": lse}
    if k == "dps":
        smp = s["sampler"]
        z = smp.step(s["y"], s["mask"], s["eps"], SIGMA, SIGMA_NEXT, LAM)
        return {"z": z} if smp.zb is None else {"z": z, "zb": smp.zb}
    if k == "gated":
        return gattn.gated_forward(s["q"], s["k"], s["v"], s["kc"], s["vc"], s["gate"], s["tiling"])
    q, kk, v = s["q"], s["k"], s["v"]
    if k == "gpa" and not case["train"]:
        with torch.no_grad():
            return gattn.global_attention(q, kk, v, s["tiling"])
    out = gattn.linear_attention(q, kk, v) if k == "linear" else gattn.global_attention(q, kk, v, s["tiling"])
    dq, dk, dv = torch.autograd.grad(out, (q, kk, v), s["dout"])
    return {"out": out, "dq": dq, "dk": dk, "dv": dv}


# ---------------------------------------------------------------- the work of one pass
def work(case):
    """Bytes: every input read once, every output written once.  Operations: the products of the method (GPA: 4 d per
    query-key pair forward, 8 d backward; linear attention: 2 products of 2 d^2 per token forward, 5 backward)."""
    k = case["kind"]
    if k == "serve":
        nd = [nh * T * SERVE_YX[0] * SERVE_YX[1] * case["d"] for T, nh in _frames(case)]
        pairs = [nh * _serve_pairs(T) for T, nh in _frames(case)]
        return {"bytes": 2.0 * 2 * case["steps"] * sum(nd), "flops": 4.0 * case["d"] * case["steps"] * sum(pairs)}
    es = 2 if case.get("dtype", "bf16") == "bf16" else 4
    if k == "compress":
        loc = case["B"] * case["nh"] * case["M"]
        return {"bytes": 2.0 * es * loc * case["S"] * case["d"] + loc * (case["d"] * es + 4) + 4 * case["nh"] * case["d"],
                "flops": 4.0 * loc * case["S"] * case["d"]}
    if k == "linear":
        tok = case["B"] * case["nh"] * case["N"]
        return {"bytes": 8.0 * tok * 64 * 2, "flops": 7.0 * 2 * tok * 64 * 64}
    bh = case["B"] * case["nh"]
    nd = bh * math.prod(_grid(case)[0]) * case["d"]
    pairs = bh * _pairs(case) * case["d"]
    if k == "gated":
        return {"bytes": 6.0 * es * nd, "flops": 8.0 * pairs}
    if k == "dps":  # z in and out, its BF16 copy in and out, observations, noise, mask
        return {"bytes": 16.0 * nd + (4.0 * nd if es == 2 else 0) + nd / case["d"] / case["nh"], "flops": 12.0 * pairs}
    return {"bytes": (8.0 if case["train"] else 4.0) * es * nd, "flops": (12.0 if case["train"] else 4.0) * pairs}


# ---------------------------------------------------------------- the same in 64 bits
def _window(G, core, halo, window, k):
    """Window factor of tile k along one dimension at its clipped positions."""
    s, e = _extents(G, core, halo)[k]
    n = torch.arange(s, e, device="cuda", dtype=torch.float64) - (k * core - halo)
    if window == "flat" or (G <= core and halo == 0):
        return torch.ones_like(n)
    return torch.sin(math.pi * (n + 0.5) / (core + 2 * halo)) ** 2


def _tiles(case):
    """(token indexes, window weights) of every extended tile."""
    grid, core, halo = _grid(case)
    ext = [_extents(*a) for a in zip(grid, core, halo)]
    ar = torch.arange(math.prod(grid), device="cuda").view(grid)
    for t, (t0, t1) in enumerate(ext[0]):
        for y, (y0, y1) in enumerate(ext[1]):
            for x, (x0, x1) in enumerate(ext[2]):
                w = [_window(*a, case["window"], i) for a, i in zip(zip(grid, core, halo), (t, y, x))]
                yield ar[t0:t1, y0:y1, x0:x1].reshape(-1), (w[0][:, None, None] * w[1][:, None] * w[2]).reshape(-1)


def _gpa64(case, q, k, v, dout=None, scale=None):
    """GPA of [BH, N, d] tensors in FP64: out, or (out, dq, dk, dv) with an upstream gradient."""
    scale = scale or 1.0 / math.sqrt(q.shape[-1])
    tiles = list(_tiles(case))
    total = torch.zeros(q.shape[1], device="cuda", dtype=torch.float64)
    for idx, w in tiles:
        total[idx] += w
    out = torch.zeros(q.shape, device="cuda", dtype=torch.float64)
    grads = [torch.zeros_like(out) for _ in range(3)] if dout is not None else []
    for idx, w in tiles:
        c = (w / total[idx])[:, None]
        step = max(1, int(2e8 // len(idx) ** 2))
        for b in range(0, q.shape[0], step):
            h = slice(b, b + step)
            qt, kt, vt = (t[h][:, idx].double() for t in (q, k, v))
            p = torch.softmax(qt @ kt.transpose(1, 2) * scale, -1)
            o = p @ vt
            out[h, idx] += c * o
            if dout is None:
                continue
            g = c * dout[h][:, idx].double()
            grads[2][h, idx] += p.transpose(1, 2) @ g
            ds = p * (g @ vt.transpose(1, 2) - (g * o).sum(-1, keepdim=True)) * scale
            grads[0][h, idx] += ds @ kt
            grads[1][h, idx] += ds.transpose(1, 2) @ qt
    return (out, *grads) if dout is not None else out


def _linear64(q, k, v, g):
    """Factorised linear attention with phi = elu + 1 and its gradients, one [N, 64] head in FP64."""
    q, k, v, g = (t.double() for t in (q, k, v, g))

    def phi(x):
        return torch.where(x > 0, x + 1, torch.exp(x)), torch.where(x > 0, torch.ones_like(x), torch.exp(x))

    (fq, gq), (fk, gk) = phi(q), phi(k)
    S, z = fk.T @ v, fk.sum(0)
    den = (fq @ z)[:, None]
    out = fq @ S / den
    go = (g * out).sum(-1, keepdim=True)
    dS, dz = fq.T @ (g / den), -(fq * (go / den)).sum(0)
    return out, (g @ S.T - go * z) / den * gq, (v @ dS.T + dz) * gk, fk @ dS


def exact(case, seed):
    k = case["kind"]
    x = _inputs(case, seed)
    if k == "linear":
        parts = [_linear64(*(x[n][b, h] for n in ("q", "k", "v", "dout"))) for b in range(case["B"]) for h in range(case["nh"])]
        return {n: torch.stack([p[i] for p in parts]).view(x["q"].shape) for i, n in enumerate(("out", "dq", "dk", "dv"))}
    if k == "compress":
        out, lse = [], []
        for b in range(case["B"]):
            for h in range(case["nh"]):
                kk, vv = x["k"][b, h].double(), x["v"][b, h].double()
                s = (kk @ x["q"][h].double()) / math.sqrt(case["d"])  # [S, M]
                lse.append(torch.logsumexp(s, 0))
                out.append(torch.einsum("sm,smd->md", torch.softmax(s, 0), vv))
        lead = (case["B"], case["nh"], case["M"])
        return {"out": torch.stack(out).view(*lead, case["d"]), "lse": torch.stack(lse).view(lead)}
    if k == "serve":
        if work(case)["flops"] > EXACT_FLOPS:
            return None
        res = []
        for i, (T, nh) in enumerate(_frames(case)):
            c = _tiled("gpa", 1, nh, case["d"], (T, *SERVE_YX), SERVE_CORE, SERVE_HALO, "bf16", "hann")
            z = x["z%d" % i]
            for _ in range(case["steps"]):  # the state is BF16 between steps
                z64 = z.double()
                z = (z64 + SERVE_C * (_gpa64(c, z64, z64, z64) - z64)).to(torch.bfloat16)
            res.append(z.double())
        return res
    if work(case)["flops"] * 14 / 12 > EXACT_FLOPS:
        return None
    shape = (case["B"] * case["nh"], -1, case["d"])
    if k == "dps":
        z, y, eps = (x[n].reshape(shape).double() for n in ("z", "y", "eps"))
        a = z if case["dtype"] == "fp32" else x["z"].to(torch.bfloat16).reshape(shape).double()
        mask = (x["mask"] != 0).repeat_interleave(case["nh"], 0)[:, :, None]
        scale = 1.0 / case["d"]
        D = _gpa64(case, a, a, a, scale=scale)
        r = torch.where(mask, D - y, torch.zeros_like(D))
        if case["dtype"] == "bf16":
            r = r.to(torch.bfloat16)  # the residual enters the backward in the input type
        _, dq, dk, dv = _gpa64(case, a, a, a, r, scale=scale)
        delta = SIGMA**2 - SIGMA_NEXT**2
        zn = z + delta * ((D - z) / SIGMA**2 - LAM * (dq + dk + dv)) + math.sqrt(delta) * eps
        zn = zn.view(x["z"].shape)
        return {"z": zn} if case["dtype"] == "fp32" else {"z": zn, "zb": zn}
    h = {n: t.reshape(shape) for n, t in x.items() if n != "gate"}
    if k == "gated":
        g = x["gate"].double().repeat(case["B"])[:, None, None]
        out = g * _gpa64(case, h["q"], h["k"], h["v"]) + (1 - g) * _gpa64(case, h["q"], h["kc"], h["vc"])
        return out.view(x["q"].shape)
    if not case["train"]:
        return _gpa64(case, h["q"], h["k"], h["v"]).view(x["q"].shape)
    res = _gpa64(case, h["q"], h["k"], h["v"], h["dout"])
    return {n: t.view(x["q"].shape) for n, t in zip(("out", "dq", "dk", "dv"), res)}
