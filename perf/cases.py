"""Timed cases of the particle compressor, through its public entry points.

A case is a dict of plain values.  ``listed()`` gives the fixed ones and
``draw(rng)`` one more of the same ranges; ``prepare`` makes what a program holds
before the call (positions or streams on the GPU, buffers sized for them),
``run`` makes one call and returns its whole output, ``work`` says what a call
cannot do without, and ``exact`` gives decoded positions in 64 bits.

Fields: ``kind`` is compress, decompress, batch_compress or batch_decompress;
``gen`` the particle set (uniform, cosmology, fluid); ``n`` particles; ``f64``
the coordinate type; ``mode`` abs or rel with its bound ``eb``; ``leaf`` the leaf
size (0: the default of 4096); ``perm`` asks for the permutation; ``autotune``,
``reduce``, ``reorder`` and ``widest`` are the config's flags.  A batch has
``count`` snapshots of ``n_lo`` to ``n_hi`` particles, evenly spread over the
logarithm, cosmology and fluid, both types and three bounds in turn.

The particle sets follow the repository's generators: uniform in [0, 256)^3; 70 %
in 20,000 Gaussian clumps of Pareto weights with 30 % background (stored in
random order); a jittered lattice with half of it displaced by a smooth flow,
stored in lattice order.
"""
import math
import struct

import numpy as np
import torch

import paper_2404_02826_gb300 as pc

BOX = 256.0
FLUID_DIMS = (384, 192, 228)
FLUID_MAX = 1 << 24
LARGEST = 1 << 27


def _case(name, kind, gen, n, f64=False, mode="rel", eb=1e-4, leaf=0, perm=False, autotune=False, reduce=False,
          reorder=False, widest=False):
    return {"name": name, "kind": kind, "gen": gen, "n": n, "f64": f64, "mode": mode, "eb": eb, "leaf": leaf,
            "perm": perm, "autotune": autotune, "reduce": reduce, "reorder": reorder, "widest": widest}


def listed():
    return [
        # a large simulation snapshot written out at a tight bound
        _case("compress-cosmology-2e27", "compress", "cosmology", 1 << 27),
        # the same snapshot read back for analysis
        _case("decompress-cosmology-2e27", "decompress", "cosmology", 1 << 27),
        # one mid-size snapshot, plain method
        _case("compress-uniform-2e20", "compress", "uniform", 1 << 20, eb=1e-3),
        # a fluid run's double-precision output, in lattice order, absolute bound
        _case("compress-fluid-2e24-f64", "compress", "fluid", 1 << 24, f64=True, mode="abs"),
        _case("decompress-fluid-2e24-f64", "decompress", "fluid", 1 << 24, f64=True, mode="abs"),
        # a served request whose other fields are permuted to the decoded order
        _case("compress-perm-3000017", "compress", "cosmology", 3_000_017, eb=1e-3, perm=True),
        # the smallest snapshots of a batch: latency and launches
        _case("compress-10007", "compress", "cosmology", 10_007, eb=1e-2),
        # the smallest served read
        _case("decompress-100003", "decompress", "uniform", 100_003, eb=1e-3),
        # leaf size searched for the smallest stream
        _case("compress-autotune-6000011", "compress", "cosmology", 6_000_011, autotune=True),
        # the paper's extra passes for ratio: bit-box reduction and reordering
        _case("compress-reduce-reorder-2e21", "compress", "cosmology", 1 << 21, eb=1e-3, reduce=True, reorder=True),
        # many snapshots of uneven size in one call, written and read
        {"name": "batch-compress-48", "kind": "batch_compress", "count": 48, "n_lo": 10_000, "n_hi": 10_000_000},
        {"name": "batch-decompress-48", "kind": "batch_decompress", "count": 48, "n_lo": 10_000,
         "n_hi": 10_000_000},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.random()
    if what < 0.15:
        n_hi = _log_int(rng, 200_000, 10_000_000)
        kind = rng.choice(["batch_compress", "batch_decompress"])
        return {"kind": kind, "count": rng.randint(4, 48), "n_lo": 10_000, "n_hi": n_hi}
    kind = "compress" if what < 0.70 else "decompress"
    gen = rng.choice(["cosmology", "cosmology", "uniform", "fluid"])
    f64 = gen == "fluid" if rng.random() < 0.75 else gen != "fluid"
    extra = rng.choice(["", "", "", "perm", "autotune", "reduce", "reorder", "widest"])
    cap = LARGEST
    if f64:
        cap //= 2
    if extra in ("perm", "widest"):
        cap //= 4
    if extra == "autotune":
        cap //= 8
    if extra in ("reduce", "reorder"):
        cap = 1 << 22
    if gen == "fluid":
        cap = min(cap, FLUID_MAX)
    n = _log_int(rng, 10_000, cap)
    if rng.random() < 0.7:
        n |= 1
    n = min(n, cap)
    if gen == "fluid" and rng.random() < 0.7:
        mode, eb = "abs", math.exp(rng.uniform(math.log(3e-5), math.log(1e-3)))
    else:
        mode, eb = "rel", math.exp(rng.uniform(math.log(1e-4), math.log(1e-2)))
    leaf = 0 if extra in ("autotune", "reduce") or rng.random() < 0.7 else _log_int(rng, 512, 8192)
    c = _case("", kind, gen, n, f64, mode, eb, leaf, extra == "perm", extra == "autotune", extra == "reduce",
              extra == "reorder", extra == "widest")
    del c["name"]
    return c


# ---- particle sets -----------------------------------------------------------


def _positions(gen, n, f64, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float64 if f64 else torch.float32
    chunk = 1 << 24
    if gen == "cosmology":
        kw = dict(generator=g, device="cuda")
        centres = torch.rand((20000, 3), dtype=dt, **kw) * BOX
        sigma = torch.exp(math.log(0.05) + math.log(40.0) * torch.rand(20000, dtype=dt, **kw))
        weight = (1.0 - torch.rand(20000, dtype=torch.float64, **kw)) ** (-1.0 / 1.8)
        cum = torch.cumsum(weight, 0)
        cum = (cum / cum[-1]).float()
    out = torch.empty((n, 3), dtype=dt, device="cuda")
    for a in range(0, n, chunk):
        b = min(n, a + chunk)
        m = b - a
        if gen == "fluid":
            out[a:b] = _fluid(a, b, g)
            continue
        p = torch.rand((m, 3), generator=g, dtype=dt, device="cuda") * BOX
        if gen == "cosmology":
            own = torch.searchsorted(cum, torch.rand(m, generator=g, device="cuda")).clamp_(max=19999)
            q = torch.randn((m, 3), generator=g, dtype=dt, device="cuda") * sigma[own, None] + centres[own]
            q = torch.remainder(q, BOX)
            p = torch.where(torch.rand((m, 1), generator=g, device="cuda") < 0.7, q, p)
        p[p >= BOX] = 0
        out[a:b] = p
    return out


def _fluid(a, b, g):
    nx, ny, nz = FLUID_DIMS
    h = 1.0 / nx
    idx = torch.arange(a, b, device="cuda")
    site = torch.stack([idx % nx, (idx // nx) % ny, idx // (nx * ny)], 1).double() * h
    x, y, z = site.unbind(1)
    ly, lz, w = ny * h, 0.6, 2.0 * math.pi
    flow = 0.05 * torch.stack([torch.sin(w * y / ly) * torch.cos(w * z / lz), torch.sin(w * z / lz) * torch.cos(w * x),
                               torch.sin(w * x) * torch.cos(w * y / ly)], 1)
    jitter = (torch.rand((b - a, 3), generator=g, dtype=torch.float64, device="cuda") - 0.5) * (0.6 * h)
    return site + jitter + torch.where((z >= 0.3)[:, None], flow, torch.zeros_like(flow))


# ---- what a program holds, and one call --------------------------------------


def _snapshots(case):
    """The snapshots of a batch: single-call cases."""
    ratio = case["n_hi"] / case["n_lo"]
    rows = []
    for i in range(case["count"]):
        n = int(case["n_lo"] * ratio ** ((i + 0.5) / case["count"]))
        gen = ("cosmology", "fluid")[i % 2]
        rows.append(_case("", "compress", gen, n, f64=(i // 2) % 2 == 1, eb=(1e-2, 1e-3, 1e-4)[i % 3]))
    return rows


def _mode(case):
    return pc.PC_EB_ABS if case["mode"] == "abs" else pc.PC_EB_REL


def _config(case):
    return pc.config(case["leaf"], autotune=case["autotune"], reduce=case["reduce"], reorder=case["reorder"],
                     widest=case["widest"])


def _stream(case, seed):
    """A stream as a program has it from a file: the bytes alone."""
    pos = _positions(case["gen"], case["n"], case["f64"], seed)
    dt = pc.PC_F64 if case["f64"] else pc.PC_F32
    c = pc.Compressor(case["n"], dt, _config(case), case["perm"])
    return c.out[:c.compress(pos, _mode(case), case["eb"])].clone()


def _empty_positions(case):
    return torch.empty((case["n"], 3), dtype=torch.float64 if case["f64"] else torch.float32, device="cuda")


def prepare(case, seed):
    state = {"case": case}
    kind = case["kind"]
    if kind == "compress":
        state["positions"] = _positions(case["gen"], case["n"], case["f64"], seed)
        dt = pc.PC_F64 if case["f64"] else pc.PC_F32
        state["compressor"] = pc.Compressor(case["n"], dt, _config(case), case["perm"])
        state["compressor"].out.zero_()  # so that the buffer past the stream's end is the same bytes every time
    elif kind == "decompress":
        state["stream"] = _stream(case, seed)
        state["positions"] = _empty_positions(case)
        state["workspace"] = torch.empty(pc.pc_decompress_workspace_size(case["n"]), dtype=torch.uint8, device="cuda")
    elif kind == "batch_compress":
        rows = _snapshots(case)
        state["jobs"], state["outs"], sizes = [], [], []
        for i, r in enumerate(rows):
            dt = pc.PC_F64 if r["f64"] else pc.PC_F32
            pos = _positions(r["gen"], r["n"], r["f64"], seed * 1000 + i)
            state["jobs"].append((pos, _mode(r), r["eb"], r["leaf"]))
            state["outs"].append(torch.zeros(pc.pc_compress_bound(r["n"], dt, r["leaf"]), dtype=torch.uint8,
                                             device="cuda"))
            sizes.append((r["n"], dt, r["leaf"]))
        state["workspace"] = torch.empty(pc.pc_compress_batch_workspace_size(sizes), dtype=torch.uint8, device="cuda")
    else:
        rows = _snapshots(case)
        state["streams"] = [_stream(r, seed * 1000 + i) for i, r in enumerate(rows)]
        state["outs"] = [_empty_positions(r) for r in rows]
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "compress":
        c = state["compressor"]
        size = c.compress(state["positions"], _mode(case), case["eb"])
        return [size, c.out, c.perm] if case["perm"] else [size, c.out]
    if kind == "decompress":
        pc.pc_decompress(state["stream"], state["positions"], state["workspace"])
        return [state["positions"]]
    if kind == "batch_compress":
        sizes, statuses = pc.pc_compress_batch(state["jobs"], state["outs"], state["workspace"])
        return state["outs"] + [np.array(sizes, dtype=np.int64), np.array(statuses, dtype=np.int32)]
    statuses = pc.pc_decompress_batch(state["streams"], [s.numel() for s in state["streams"]], state["outs"])
    return state["outs"] + [np.array(statuses, dtype=np.int32)]


def _is_batch(case):
    return case["kind"].startswith("batch")


def work(case):
    """Positions on one side, the stream on the other.  The stream's size depends on the data; it is put at
    what a volume of equal leaves would need: per axis the bits of a leaf's extent in lattice steps, and one."""
    if _is_batch(case):
        parts = [work(r) for r in _snapshots(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    n = case["n"]
    leaves = 2.0 ** max(0, math.ceil(math.log2(max(1.0, n / (case["leaf"] or 4096)))))
    steps = 1.0 / (2.0 * case["eb"])
    bits = 3.0 * max(1.0, math.log2(max(1.0, steps / leaves ** (1.0 / 3.0))) + 1.0)
    nbytes = 3 * (8 if case["f64"] else 4) * n + bits / 8.0 * n + 32 * leaves + 96
    return {"bytes": int(nbytes + (4 * n if case["perm"] else 0)), "flops": 6 * n}


# ---- decoded positions in 64 bits --------------------------------------------


def exact(case, seed):
    """The centre of every particle's lattice cell, o + s q, read from the stream's documented layout; streams
    themselves are bytes and have no such value."""
    if case["kind"] == "decompress":
        return [_decode(_stream(case, seed))]
    if case["kind"] == "batch_decompress":
        return [_decode(_stream(r, seed * 1000 + i)) for i, r in enumerate(_snapshots(case))] + [None]
    return None


def _decode(stream):
    head = bytes(stream[:96].cpu().numpy())
    n, = struct.unpack_from("<Q", head, 8)
    s, ox, oy, oz = struct.unpack_from("<4d", head, 32)
    leaves, words = struct.unpack_from("<2Q", head, 64)
    table = stream[96:96 + 32 * leaves].clone()
    first = table.view(torch.int64).view(leaves, 4)[:, 0].contiguous()
    word0 = table.view(torch.int64).view(leaves, 4)[:, 1].contiguous()
    ref = table.view(torch.int32).view(leaves, 8)[:, 4:7].long()
    m = table.view(leaves, 32)[:, 28:31].long()
    payload = torch.cat([stream[96 + 32 * leaves:96 + 32 * leaves + 4 * words].clone().view(torch.int32),
                         torch.zeros(2, dtype=torch.int32, device=stream.device)])
    out = torch.empty((n, 3), dtype=torch.float64, device=stream.device)
    for a in range(0, n, 1 << 23):
        i = torch.arange(a, min(n, a + (1 << 23)), device=stream.device)
        leaf = torch.searchsorted(first, i, right=True) - 1
        k = i - first[leaf]
        mm = m[leaf]
        bit = word0[leaf] * 32 + (k - 1).clamp_(min=0) * mm.sum(1)
        for d, o in enumerate((ox, oy, oz)):
            w, sh = bit >> 5, bit & 31
            lo = payload[w].long() & 0xFFFFFFFF
            hi = payload[w + 1].long() & 0x7FFFFFFF  # at most 31 + 31 bits are looked at
            code = ((lo | (hi << 32)) >> sh) & ((torch.ones_like(bit) << mm[:, d]) - 1)
            half = (torch.ones_like(bit) << (mm[:, d] - 1).clamp(min=0)) - 1
            off = torch.where((k == 0) | (mm[:, d] == 0), torch.zeros_like(code), code - half)
            out[i, d] = o + s * (ref[leaf, d] + off).double()
            bit = bit + mm[:, d]
    return out
