"""Performance cases of the library: what they are, how their inputs are made, one pass through the public calls.

A case is a dict of plain values; `kind` says which operators it runs.  All tensors are synthetic, drawn on the device from
the seed alone with the distributions the operators meet in use (activations and their gradients normal(0, 1), kernels and
weights scaled by their fan-in, fields uniform in [-1, 1)).  A tensor that lives in several shards is kept in one buffer,
every shard starting on a 256-byte boundary, as a program that allocates its memory once would hold it; the operators get
the shards.
"""

import math

import torch

import paper_2006_03108_b200 as distdl

DEV = "cuda"
DTYPES = {"f32": (torch.float32, distdl.F32, 4), "bf16": (torch.bfloat16, distdl.BF16, 2), "f64": (torch.float64, distdl.F64, 8)}


# ---------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------

def listed():
    return [
        # The smallest exchange: a 2-D field on four workers, one ghost cell a side, H on the field and H* on its gradient,
        # as between the steps of a small solver: latency and launches.
        {"name": "halo_256x256_h1", "kind": "halo", "shape": "256,256", "parts": "2,2", "halo": "1,1", "dtype": "f32", "periodic": False},
        # The volumetric exchange (an eighth-order stencil on a seismic volume), H and H*.
        {"name": "halo_512cube_h4", "kind": "halo", "shape": "512,512,512", "parts": "4,4,4", "halo": "4,4,4", "dtype": "f32", "periodic": False},
        # Row blocks to column blocks and back with extents that divide by nothing: the change of partition between two layers.
        {"name": "repartition_6001x7003", "kind": "repartition", "shape": "6001,7003", "src": "8,1", "dst": "1,8", "dtype": "f32"},
        # Parameters sent to eight workers, their gradients summed back.
        {"name": "broadcast_sum_4096_k8", "kind": "fan", "n": 4096 * 4096, "k": 8, "dtype": "f32"},
        # One training step of the depthwise convolution layer on large images.
        {"name": "conv5_16x16x1024", "kind": "conv", "shape": "16,16,1024,1024", "parts": "4,4", "k": 5},
        # The same step on images whose rows are no whole number of vectors, on an uneven partition.
        {"name": "conv3_4x12x515x509", "kind": "conv", "shape": "4,12,515,509", "parts": "3,2", "k": 3},
        # One training step of the affine layer (forward, input gradient, weight and bias gradients).
        {"name": "affine_256x8192_train", "kind": "affine", "nb": 256, "bfi": 2048, "bfo": 2048, "pfo": 4, "pfi": 4, "train": True},
        # The affine layer applied to a handful of samples: inference, bound by the weights.
        {"name": "affine_16x8192_infer", "kind": "affine", "nb": 16, "bfi": 2048, "bfo": 2048, "pfo": 4, "pfi": 4, "train": False},
        # Max pooling on unbalanced halos, forward and backward, behind a large convolution.
        {"name": "pool3s2_16x16x1024", "kind": "pool", "shape": "16,16,1024,1024", "parts": "4,4", "k": 3, "s": 2, "pad": 1, "mode": "max"},
        # Forward and adjoint of the eighth-order star stencil on a volume: a step of a wave equation and of its gradient.
        {"name": "stencil_512cube_r4", "kind": "stencil", "shape": "512,512,512", "parts": "4,4,4", "r": 4},
        # One training step of the convolution layer with channel partitions on large images.
        {"name": "convg5_4x16x1024", "kind": "convg", "shape": "4,16,1024,1024", "nco": 16, "pci": 2, "pco": 2, "parts": "2,2", "k": 5},
        # The same step on small images in a large batch (a digit classifier's second layer on four workers).
        {"name": "convg5_256x6x28", "kind": "convg", "shape": "256,6,28,28", "nco": 16, "pci": 1, "pco": 1, "parts": "2,2", "k": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _text(v):
    return ",".join(str(int(x)) for x in v)


def draw(rng):
    kind = rng.choice(["halo", "repartition", "fan", "conv", "affine", "pool", "stencil", "convg"])
    if kind == "halo":
        rank = rng.choice([2, 3, 4])
        dtype = rng.choice(["f32", "f32", "bf16", "f64"])
        h = rng.randint(1, 4)
        if rank == 2:
            parts = [rng.randint(1, 4), rng.randint(2, 4)]
            shape = [_log_int(rng, 64, 4096), _log_int(rng, 64, 4096)]
            halo = [h, h]
        elif rank == 3:
            parts = [rng.randint(1, 4), rng.randint(1, 4), rng.randint(2, 4)]
            shape = [_log_int(rng, 32, 384) for _ in range(3)]
            halo = [h, h, h]
        else:
            parts = [1, 1, rng.randint(1, 4), rng.randint(2, 4)]
            shape = [rng.randint(1, 8), rng.randint(1, 16), _log_int(rng, 32, 768), _log_int(rng, 32, 768)]
            halo = [0, 0, h, h]
        return {"kind": kind, "shape": _text(shape), "parts": _text(parts), "halo": _text(halo), "dtype": dtype,
                "periodic": rng.random() < 0.25}
    if kind == "repartition":
        p = rng.choice([2, 3, 4, 8])
        src, dst = ([p, 1], [1, p]) if rng.random() < 0.5 else ([1, p], [p, 1])
        return {"kind": kind, "shape": _text([_log_int(rng, 64, 7000), _log_int(rng, 64, 7000)]), "src": _text(src), "dst": _text(dst),
                "dtype": rng.choice(["f32", "f32", "bf16"])}
    if kind == "fan":
        return {"kind": kind, "n": _log_int(rng, 1 << 12, 1 << 24), "k": rng.randint(2, 8), "dtype": rng.choice(["f32", "f32", "bf16"])}
    if kind == "conv":
        n, c = _log_int(rng, 1, 16), _log_int(rng, 1, 16)
        return {"kind": kind, "shape": _text([n, c, _log_int(rng, 32, 1024), _log_int(rng, 32, 1024)]),
                "parts": _text([rng.randint(1, 4), rng.randint(1, 4)]), "k": rng.choice([3, 5, 7])}
    if kind == "affine":
        pfo, pfi = rng.choice([1, 2, 3, 4]), rng.choice([1, 2, 3, 4])
        return {"kind": kind, "nb": _log_int(rng, 1, 256), "bfi": 8 * _log_int(rng, 16, 256), "bfo": 8 * _log_int(rng, 16, 256),
                "pfo": pfo, "pfi": pfi, "train": rng.random() < 0.5}
    if kind == "pool":
        k, s, pad = rng.choice([(2, 2, 0), (3, 2, 1), (3, 2, 1), (3, 1, 1)])
        return {"kind": kind, "shape": _text([_log_int(rng, 1, 16), _log_int(rng, 1, 16), _log_int(rng, 48, 1024), _log_int(rng, 48, 1024)]),
                "parts": _text([rng.randint(1, 4), rng.randint(1, 4)]), "k": k, "s": s, "pad": pad, "mode": rng.choice(["max", "avg"])}
    if kind == "stencil":
        return {"kind": kind, "shape": _text([_log_int(rng, 40, 384) for _ in range(3)]),
                "parts": _text([rng.randint(1, 4) for _ in range(3)]), "r": rng.randint(1, 4)}
    side = _log_int(rng, 24, 512)
    n = max(1, min(256, _log_int(rng, 1, 512) * 28 * 28 // (side * side)))
    return {"kind": "convg", "shape": _text([n, rng.randint(2, 16), side, max(24, side + rng.randint(-7, 7))]), "nco": rng.randint(2, 16),
            "pci": rng.randint(1, 2), "pco": rng.randint(1, 2), "parts": _text([rng.randint(1, 2), rng.randint(1, 2)]), "k": rng.choice([3, 5, 5, 7])}


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------

def _ints(text):
    return [int(v) for v in text.split(",")]


def _prod(v):
    n = 1
    for x in v:
        n *= x
    return n


def _shards(shapes, dtype, fill):
    """One buffer and its shards; fill(n) gives n values of the dtype."""
    step = 256 // torch.empty((), dtype=dtype).element_size()
    at, total = [], 0
    for s in shapes:
        at.append(total)
        total += -(-_prod(s) // step) * step
    buf = fill(total)
    return buf, [buf[o:o + _prod(s)].view(s) for o, s in zip(at, shapes)]


class _Draw:
    """Values on the device from the seed alone."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))

    def normal(self, dtype=torch.float32, std=1.0):
        return lambda n: (torch.randn(n, device=DEV, generator=self.g, dtype=torch.float32) * std).to(dtype)

    def uniform(self, dtype=torch.float32):
        return lambda n: (torch.rand(n, device=DEV, generator=self.g, dtype=torch.float32) * 2 - 1).to(dtype)

    @staticmethod
    def zeros(dtype=torch.float32):
        return lambda n: torch.zeros(n, device=DEV, dtype=dtype)


def _padded(part):
    return [part.padded_shape(w) for w in range(part.num_workers)]


def _bulk(part):
    return [part.bulk_shape(w) for w in range(part.num_workers)]


def _prepare_halo(c, d):
    dt, code, _ = DTYPES[c["dtype"]]
    shape, parts, halo = _ints(c["shape"]), _ints(c["parts"]), _ints(c["halo"])
    per = [h > 0 for h in halo] if c["periodic"] else None
    part = distdl.Partition(shape, parts, halo, halo, dtype=code, periodic=per)
    x, xs = _shards(_padded(part), dt, d.uniform(dt))
    g, gs = _shards(_padded(part), dt, d.uniform(dt))
    return {"part": part, "x": x, "xs": xs, "g": g, "gs": gs}


def _run_halo(s):
    distdl.halo_fwd(s["part"], s["xs"])
    distdl.halo_adj(s["part"], s["gs"])
    return s["x"], s["g"]


def _prepare_repartition(c, d):
    dt, code, _ = DTYPES[c["dtype"]]
    rep = distdl.Repartition(_ints(c["shape"]), _ints(c["src"]), _ints(c["dst"]), code)
    src = [rep.shard_shape(w) for w in range(rep.num_src)]
    dst = [rep.shard_shape(w, destination=True) for w in range(rep.num_dst)]
    _, xs = _shards(src, dt, d.normal(dt))
    y, ys = _shards(dst, dt, d.zeros(dt))
    _, gs = _shards(dst, dt, d.normal(dt))
    dx, dxs = _shards(src, dt, d.zeros(dt))
    return {"rep": rep, "xs": xs, "y": y, "ys": ys, "gs": gs, "dx": dx, "dxs": dxs}


def _run_repartition(s):
    distdl.repartition_fwd(s["rep"], s["xs"], s["ys"])
    distdl.repartition_adj(s["rep"], s["gs"], s["dxs"])
    return s["y"], s["dx"]


def _prepare_fan(c, d):
    dt, _, _ = DTYPES[c["dtype"]]
    n, k = c["n"], c["k"]
    copies, cs = _shards([(n,)] * k, dt, d.zeros(dt))
    _, gs = _shards([(n,)] * k, dt, d.normal(dt))
    return {"p": d.normal(dt)(n), "copies": copies, "cs": cs, "gs": gs, "sum": torch.zeros(n, device=DEV, dtype=dt)}


def _run_fan(s):
    distdl.broadcast_fwd(s["p"], s["cs"])
    distdl.sumreduce_fwd(s["gs"], s["sum"])
    return s["copies"], s["sum"]


def _prepare_conv(c, d):
    shape, parts, k = _ints(c["shape"]), _ints(c["parts"]), c["k"]
    halo = (0, 0, k // 2, k // 2)
    part = distdl.Partition(shape, (1, 1) + tuple(parts), halo, halo)
    _, xs = _shards(_padded(part), torch.float32, d.normal())
    y, ys = _shards(_bulk(part), torch.float32, d.zeros())
    _, gs = _shards(_bulk(part), torch.float32, d.normal())
    dx, dxs = _shards(_padded(part), torch.float32, d.zeros())
    C = shape[1]
    return {"part": part, "k": k, "xs": xs, "y": y, "ys": ys, "gs": gs, "dx": dx, "dxs": dxs,
            "w": d.normal(std=0.5 / k)(C * k * k).view(C, k, k), "b": d.normal()(C),
            "dw": torch.zeros(C, k, k, device=DEV), "db": torch.zeros(C, device=DEV),
            "ws": torch.empty(distdl.conv_adj_params_workspace(part, k, k), dtype=torch.uint8, device=DEV)}


def _run_conv(s):
    distdl.conv_fwd(s["part"], s["xs"], s["w"], s["b"], s["ys"])
    distdl.conv_adj(s["part"], s["gs"], s["w"], s["dxs"])
    distdl.conv_adj_params(s["part"], s["xs"], s["gs"], (s["k"], s["k"]), s["dw"], s["db"], s["ws"])
    return s["y"], s["dx"], s["dw"], s["db"]


def _prepare_affine(c, d):
    nb, bfi, bfo, pfo, pfi = c["nb"], c["bfi"], c["bfo"], c["pfo"], c["pfi"]
    bf = torch.bfloat16
    _, xs = _shards([(nb, bfi)] * pfi, bf, d.normal(bf))
    _, ws = _shards([(bfo, bfi)] * (pfo * pfi), bf, d.normal(bf, 1.0 / math.sqrt(bfi * pfi)))
    _, bs = _shards([(bfo,)] * pfo, torch.float32, d.normal())
    y, ys = _shards([(nb, bfo)] * pfo, torch.float32, d.zeros())
    s = {"dims": (nb, bfi * pfi, bfo * pfo, pfo, pfi), "xs": xs, "ws": ws, "bs": bs, "y": y, "ys": ys, "train": c["train"]}
    if c["train"]:
        _, s["gs"] = _shards([(nb, bfo)] * pfo, bf, d.normal(bf))
        s["dx"], s["dxs"] = _shards([(nb, bfi)] * pfi, torch.float32, d.zeros())
        s["dw"], s["dws"] = _shards([(bfo, bfi)] * (pfo * pfi), torch.float32, d.zeros())
        s["db"], s["dbs"] = _shards([(bfo,)] * pfo, torch.float32, d.zeros())
    return s


def _run_affine(s):
    distdl.affine_fwd(*s["dims"], s["xs"], s["ws"], s["bs"], s["ys"])
    if not s["train"]:
        return s["y"]
    distdl.affine_adj(*s["dims"], s["gs"], s["ws"], s["dxs"])
    distdl.affine_adj_params(*s["dims"], s["gs"], s["xs"], s["dws"], s["dbs"])
    return s["y"], s["dx"], s["dw"], s["db"]


def _pool_widths(c):
    shape, parts = _ints(c["shape"]), _ints(c["parts"])
    return [distdl.halo_widths_1d(shape[2 + i], parts[i], c["k"], c["s"], 1, c["pad"], c["pad"])[:2] for i in range(2)]


def _pool_out(c):
    """Extents of the workers' blocks of the output, rows and columns."""
    shape, parts = _ints(c["shape"]), _ints(c["parts"])
    out = []
    for i in range(2):
        m, p = (shape[2 + i] + 2 * c["pad"] - c["k"]) // c["s"] + 1, parts[i]
        out.append([m // p + (1 if w < m % p else 0) for w in range(p)])
    return out


def _prepare_pool(c, d):
    shape, parts = _ints(c["shape"]), _ints(c["parts"])
    (hlo, hhi), (wlo, whi) = _pool_widths(c)
    part = distdl.Partition(shape, (1, 1) + tuple(parts), [0, 0, hlo, wlo], [0, 0, hhi, whi])
    oh, ow = _pool_out(c)
    outs = [(shape[0], shape[1], a, b) for a in oh for b in ow]
    x, xs = _shards(_padded(part), torch.float32, d.normal())
    y, ys = _shards(outs, torch.float32, d.zeros())
    a, ars = _shards(outs, torch.int32, d.zeros(torch.int32)) if c["mode"] == "max" else (None, None)
    _, gs = _shards(outs, torch.float32, d.normal())
    dx, dxs = _shards(_padded(part), torch.float32, d.zeros())
    return {"part": part, "kernel": (c["k"], c["k"]), "stride": (c["s"], c["s"]), "pad": ((c["pad"],) * 2,) * 2,
            "mode": distdl.POOL_MAX if c["mode"] == "max" else distdl.POOL_AVG,
            "x": x, "xs": xs, "y": y, "ys": ys, "a": a, "as": ars, "gs": gs, "dx": dx, "dxs": dxs}


def _run_pool(s):
    distdl.pool_fwd(s["part"], s["xs"], s["kernel"], s["stride"], s["pad"], s["mode"], s["ys"], s["as"])
    distdl.pool_adj(s["part"], s["gs"], s["as"], s["kernel"], s["stride"], s["pad"], s["mode"], s["dxs"])
    return s["y"], s["a"], s["dx"], s["x"]


def _prepare_stencil(c, d):
    shape, parts, r = _ints(c["shape"]), _ints(c["parts"]), c["r"]
    part = distdl.Partition(shape, parts, (r,) * 3, (r,) * 3)
    _, xs = _shards(_padded(part), torch.float32, d.uniform())
    y, ys = _shards(_bulk(part), torch.float32, d.zeros())
    _, gs = _shards(_bulk(part), torch.float32, d.uniform())
    dx, dxs = _shards(_padded(part), torch.float32, d.zeros())
    taps = (d.normal(std=0.5)(3 * (2 * r + 1)).cpu().view(3, 2 * r + 1)).tolist()
    return {"part": part, "taps": taps, "xs": xs, "y": y, "ys": ys, "gs": gs, "dx": dx, "dxs": dxs}


def _run_stencil(s):
    distdl.stencil3d_fwd(s["part"], s["xs"], s["taps"], s["ys"])
    distdl.stencil3d_adj(s["part"], s["gs"], s["taps"], s["dxs"])
    return s["y"], s["dx"]


def _split(n, p):
    return [n // p + (1 if i < n % p else 0) for i in range(p)]


def _prepare_convg(c, d):
    n, ci, h, w = _ints(c["shape"])
    parts, k, co, pci, pco = _ints(c["parts"]), c["k"], c["nco"], c["pci"], c["pco"]
    halo = (0, 0, k // 2, k // 2)
    part = distdl.Partition((n, ci, h, w), (1, pci) + tuple(parts), halo, halo)
    ypart = distdl.Partition((n, co, h, w), (1, pco) + tuple(parts))
    _, xs = _shards(_padded(part), torch.float32, d.normal())
    y, ys = _shards(_bulk(ypart), torch.float32, d.zeros())
    _, gs = _shards(_bulk(ypart), torch.float32, d.normal())
    dx, dxs = _shards(_padded(part), torch.float32, d.zeros())
    blocks = [(a, b, k, k) for a in _split(co, pco) for b in _split(ci, pci)]
    _, ws = _shards(blocks, torch.float32, d.normal(std=1.0 / math.sqrt(ci * k * k)))
    _, bs = _shards([(a,) for a in _split(co, pco)], torch.float32, d.normal())
    dw, dws = _shards(blocks, torch.float32, d.zeros())
    db, dbs = _shards([(a,) for a in _split(co, pco)], torch.float32, d.zeros())
    return {"part": part, "nco": co, "pco": pco, "k": k, "xs": xs, "y": y, "ys": ys, "gs": gs, "dx": dx, "dxs": dxs,
            "w": ws, "b": bs, "dw": dw, "dws": dws, "db": db, "dbs": dbs,
            "ws": torch.empty(distdl.convg_adj_params_workspace(part, co, pco, k, k), dtype=torch.uint8, device=DEV)}


def _run_convg(s):
    distdl.convg_fwd(s["part"], s["nco"], s["pco"], s["xs"], s["w"], s["b"], s["ys"])
    distdl.convg_adj(s["part"], s["nco"], s["pco"], s["gs"], s["w"], s["dxs"])
    distdl.convg_adj_params(s["part"], s["nco"], s["pco"], s["xs"], s["gs"], (s["k"], s["k"]), s["dws"], s["dbs"], s["ws"])
    return s["y"], s["dx"], s["dw"], s["db"]


def prepare(case, seed):
    s = globals()["_prepare_" + case["kind"]](case, _Draw(seed))
    s["kind"] = case["kind"]
    return s


def run(state):
    return globals()["_run_" + state["kind"]](state)


# ---------------------------------------------------------------------------------------------
# Work and tolerances
# ---------------------------------------------------------------------------------------------

def _halo_cells(c):
    """(ghost cells, ghost cells with an owner, bulk cells that some ghost copies), all workers together."""
    shape, parts, halo = _ints(c["shape"]), _ints(c["parts"]), _ints(c["halo"])
    ghosts = owned = receiving = 0
    dims = []
    for n, p, h in zip(shape, parts, halo):
        wrap = c["periodic"] and h > 0
        dims.append([(b, b + 2 * h, b + (h if wrap or i > 0 else 0) + (h if wrap or i + 1 < p else 0),
                      max(0, b - (h if wrap or i > 0 else 0) - (h if wrap or i + 1 < p else 0))) for i, b in enumerate(_split(n, p))])
    for w in range(_prod(parts)):
        at = []
        for p in reversed(parts):
            at.append(w % p)
            w //= p
        d = [dims[k][i] for k, i in enumerate(reversed(at))]
        bulk = _prod(v[0] for v in d)
        ghosts += _prod(v[1] for v in d) - bulk
        owned += _prod(v[2] for v in d) - bulk
        receiving += bulk - _prod(v[3] for v in d)
    return ghosts, owned, receiving


def _padded_cells(shape, parts, lo, hi):
    """Cells of all padded shards; lo, hi: ghost widths per dimension (one number, or one per worker)."""
    n = 1
    for k, p in enumerate(parts):
        a = lo[k] if isinstance(lo[k], (list, tuple)) else [lo[k]] * p
        b = hi[k] if isinstance(hi[k], (list, tuple)) else [hi[k]] * p
        n *= shape[k] + sum(a) + sum(b)
    return n


def work(case):
    """Bytes and operations of a pass: every call of it reads its inputs once and writes its outputs once."""
    c, kind = case, case["kind"]
    if kind == "halo":
        size = DTYPES[c["dtype"]][2]
        ghosts, owned, receiving = _halo_cells(c)
        # H: ghosts written, their owners' cells read.  H*: owned ghosts read, all cleared, receiving cells read and written.
        return {"bytes": size * (2 * ghosts + 2 * owned + 2 * receiving), "flops": owned}
    if kind == "repartition":
        return {"bytes": 4 * _prod(_ints(c["shape"])) * DTYPES[c["dtype"]][2], "flops": 0}
    if kind == "fan":
        return {"bytes": 2 * (c["k"] + 1) * c["n"] * DTYPES[c["dtype"]][2], "flops": (c["k"] - 1) * c["n"]}
    if kind == "affine":
        nb, nfi, nfo = c["nb"], c["bfi"] * c["pfi"], c["bfo"] * c["pfo"]
        fwd = 2 * nb * nfi + 2 * nfi * nfo + 4 * nfo + 4 * nb * nfo
        if not c["train"]:
            return {"bytes": fwd, "flops": 2 * nb * nfi * nfo}
        adj = 2 * nb * nfo + 2 * nfi * nfo + 4 * nb * nfi
        par = 2 * nb * nfo + 2 * nb * nfi + 4 * nfi * nfo + 4 * nfo
        return {"bytes": fwd + adj + par, "flops": 6 * nb * nfi * nfo + nb * nfo}
    shape = _ints(c["shape"])
    cells = _prod(shape)
    if kind == "conv":
        h = c["k"] // 2
        padded = _padded_cells(shape, [1, 1] + _ints(c["parts"]), [0, 0, h, h], [0, 0, h, h])
        return {"bytes": 4 * (2 * cells + cells + padded + 2 * cells), "flops": 3 * 2 * c["k"] ** 2 * cells}
    if kind == "pool":
        (hlo, hhi), (wlo, whi) = _pool_widths(c)
        padded = _padded_cells(shape, [1, 1] + _ints(c["parts"]), [0, 0, hlo, wlo], [0, 0, hhi, whi])
        oh, ow = _pool_out(c)
        out = shape[0] * shape[1] * sum(oh) * sum(ow) * (2 if c["mode"] == "max" else 1)
        return {"bytes": 4 * (cells + out + out + padded), "flops": 2 * c["k"] ** 2 * shape[0] * shape[1] * sum(oh) * sum(ow)}
    if kind == "stencil":
        padded = _padded_cells(shape, _ints(c["parts"]), [c["r"]] * 3, [c["r"]] * 3)
        return {"bytes": 4 * (2 * cells + cells + padded), "flops": 2 * 2 * (6 * c["r"] + 3) * cells}
    h = c["k"] // 2
    n, ci, co = shape[0], shape[1], c["nco"]
    px = shape[2] * shape[3]
    padded = _padded_cells(shape, [1, c["pci"]] + _ints(c["parts"]), [0, 0, h, h], [0, 0, h, h])
    wts = ci * co * c["k"] ** 2
    return {"bytes": 4 * (3 * wts + n * px * (2 * ci + 3 * co) + padded), "flops": 3 * 2 * n * px * wts}


# Relative errors of fp32 (affine: bf16 inputs, fp32 sums) against the same operators in 64 bits, measured on the listed and on
# sixty drawn cases and taken four times: 2-norm, then the largest difference over the root mean square (or the value).
#   conv     y, dx 1.3e-7;  dw, db (sums over up to 16.8 M pixels) 1.0e-6 / 3.2e-6
#   convg    y, dx 4.6e-7 / 3.9e-6;  dw, db 8.7e-7 / 3.4e-6
#   stencil  9.6e-8 / 8.3e-7;  pool: a few sums of at most nine terms, positions of maxima exact
#   affine   y, dx 6.5e-6 / 2.9e-5 (8192 products a sum);  dw 2.3e-7
TOLERANCE = {
    "conv": {"rel": 4e-6, "max": 1.3e-5},
    "convg": {"rel": 4e-6, "max": 1.6e-5},
    "stencil": {"rel": 4e-7, "max": 4e-6},
    "pool": {"rel": 4e-7, "max": 4e-6},
    "affine": {"rel": 2.6e-5, "max": 1.2e-4},
}


def tolerance(case):
    # copies, and sums whose order the operator fixes
    return dict(TOLERANCE[case["kind"]]) if case["kind"] in TOLERANCE else "exact"
