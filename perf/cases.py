"""Measured cases of the loop-nest executor: what its users run, through its public entry points.

A case is a dict of plain values.  ``listed()`` gives the fixed cases, ``draw(rng)`` one more
case of the same ranges, ``prepare(case, seed)`` what a program holds before the call (inputs on
the GPU, the planned nest, stencil, batch or server), ``run(state)`` one pass, ``work(case)`` the
bytes and operations a pass cannot do without, and ``exact(case, seed)`` the outputs in 64 bits.

Kinds of case:

* ``rows``     a rectangular nest whose inner levels are reduced (``Nest.run``)
* ``csr``      a ragged nest, rows of Zipf lengths, optionally with the fused histogram
* ``batch``    many uneven nests in one ``hp_nest_run_batch``
* ``serve``    a burst of requests to a server, submitted and polled
* ``stencil``  ``steps`` steps of a 2-D stencil (``Stencil.run``)
* ``ordered``  a non-commutative reduction in iteration order (``Nest.run``)
* ``narrow``   reductions and dot products of 8- and 16-bit integers (``Nest.run``)
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2309_01906_gb300 import binding as hb
from paper_2309_01906_gb300 import synth

_CHUNK = 1 << 27          # elements evaluated at once in 64 bits
_ZETA_1_5 = 2.612375348685488
_MAX_LEN = 65536          # longest CSR row


def listed():
    return [
        # a matrix-vector product of a small model layer: one short launch, latency counts
        {"name": "gemv_1k", "kind": "rows", "extents": "1024,1024", "red_level": 1, "op": "sum", "prec": "f32_comp",
         "body": "dot_bcast", "map": "auto"},
        # the 4-level nest of the benchmark under its explicit map (grid, grid, cluster, CTA); 2 GiB
        {"name": "nest4", "kind": "rows", "extents": "64,512,16,1024", "red_level": 2, "op": "sum",
         "prec": "f32_comp", "body": "dot_bcast", "map": "cluster4x4"},
        # sums over a short feature axis (100 columns), a million rows
        {"name": "rows_short", "kind": "rows", "extents": "1000000,100", "red_level": 1, "op": "sum", "prec": "f32",
         "body": "load", "map": "auto"},
        # exact integer sums of long rows whose odd length keeps them off 16-byte boundaries
        {"name": "rows_odd", "kind": "rows", "extents": "20011,8195", "red_level": 1, "op": "sum", "prec": "i64",
         "body": "load", "map": "auto"},
        # one compensated total of a whole array (a loss, a norm, a checksum)
        {"name": "total", "kind": "rows", "extents": "8192,8192", "red_level": 0, "op": "sum", "prec": "f32_comp",
         "body": "load", "map": "auto"},
        # sparse matrix-vector product with the int64 column histogram in the same sweep
        {"name": "csr_zipf", "kind": "csr", "rows": 1 << 22, "cols": 1 << 22, "prec": "f32_comp", "op": "sum",
         "hist": True},
        # 10,000 uneven nests, FP32 compensated sums and int32 maxima, in one launch per arithmetic
        {"name": "batch_uneven", "kind": "batch", "nests": 10000, "shape_seed": 9},
        # a burst of 256 requests to the default server
        {"name": "serve_burst", "kind": "serve", "requests": 256, "shape_seed": 9},
        # one time step of the 9-point diffusion stencil: bound by memory
        {"name": "stencil_step", "kind": "stencil", "ny": 16384, "nx": 16384, "radius": 1, "steps": 1},
        # four fused time steps of it
        {"name": "stencil_fused", "kind": "stencil", "ny": 16384, "nx": 16384, "radius": 1, "steps": 4},
        # gated linear recurrences: the affine maps of 64 long sequences composed in order
        {"name": "compose", "kind": "ordered", "op": "compose", "rows": 64, "len": 1 << 22},
        # int8 dot products of quantised rows
        {"name": "dot_i8", "kind": "narrow", "prec": "i8", "op": "sum", "body": "dot_bcast", "rows": 16384,
         "len": 65536},
    ]


def _log(rng, lo, hi):
    """An integer log-uniform in [2^lo, 2^hi]."""
    return int(2.0 ** rng.uniform(lo, hi))


def draw(rng):
    kind = rng.choices(["rows", "nest4", "csr", "batch", "serve", "stencil", "ordered", "narrow"],
                       [36, 8, 9, 7, 6, 14, 10, 10])[0]
    if kind == "rows":
        lt = rng.uniform(12, 29)
        lr = rng.uniform(0, lt)
        ext = [max(1, int(2.0 ** (lt - lr))), max(1, int(2.0 ** lr))]
        red = 1
        if rng.random() < 0.3 and ext[1] >= 16:      # two reduced levels
            k = rng.randint(2, 16)
            ext = [ext[0], max(1, ext[1] // k), k]
        prec = rng.choice(["f32", "f32_comp", "f32_comp", "i32", "i64"])
        return {"kind": "rows", "extents": ",".join(map(str, ext)), "red_level": red,
                "op": rng.choice(["sum", "sum", "max", "min"]), "prec": prec,
                "body": rng.choice(["load", "dot_bcast"]), "map": "auto"}
    if kind == "nest4":
        return {"kind": "rows", "extents": f"{rng.randint(1, 24)},{_log(rng, 5, 8)},{rng.randint(4, 32)},"
                                           f"{_log(rng, 7, 11)}", "red_level": 2, "op": "sum",
                "prec": rng.choice(["f32", "f32_comp"]), "body": "dot_bcast", "map": rng.choice(["cluster4x4", "cluster8x8"])}
    if kind == "csr":
        return {"kind": "csr", "rows": _log(rng, 8, 20), "cols": _log(rng, 10, 22),
                "prec": rng.choice(["f32", "f32_comp"]), "op": rng.choice(["sum", "sum", "max"]),
                "hist": rng.random() < 0.5}
    if kind == "batch":
        return {"kind": "batch", "nests": _log(rng, 5, 12), "shape_seed": rng.randint(10, 10 ** 6)}
    if kind == "serve":
        return {"kind": "serve", "requests": _log(rng, 3, 9), "shape_seed": rng.randint(10, 10 ** 6)}
    if kind == "stencil":
        radius, steps = rng.randint(1, 4), rng.choice([1, 1, 2, 3, 4, 5, 6, 7, 8])
        # at most the listed fused case's arithmetic
        top = min(13.9, 0.5 * math.log2(16384.0 ** 2 * 36 / ((2 * radius + 1) ** 2 * steps)))
        ny, nx = _log(rng, 6, top), _log(rng, 6, top)
        return {"kind": "stencil", "ny": ny, "nx": nx if rng.random() < 0.5 else (nx + 3) // 4 * 4, "radius": radius,
                "steps": steps}
    if kind == "ordered":
        lt = rng.uniform(14, 26)
        lr = rng.uniform(6, min(lt, 22))
        return {"kind": "ordered", "op": rng.choice(["compose", "mat2", "last"]),
                "rows": max(1, int(2.0 ** (lt - lr))), "len": int(2.0 ** lr)}
    prec = rng.choice(["i8", "i16"])
    op = rng.choice(["sum", "max", "min"])
    body = "dot_bcast" if prec == "i8" and op == "sum" and rng.random() < 0.6 else "load"
    lt = rng.uniform(14, 30)
    lr = rng.uniform(5, min(lt, 22))
    length = int(2.0 ** lr)
    if rng.random() < 0.5:
        length = (length + 15) // 16 * 16
    return {"kind": "narrow", "prec": prec, "op": op, "body": body, "rows": max(1, int(2.0 ** (lt - lr))),
            "len": length}


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator("cuda").manual_seed(seed)


def _normal(n, g):
    return torch.randn(n, generator=g, device="cuda", dtype=torch.float32)


def _uniform(n, lo, hi, g):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float32).mul_(hi - lo).add_(lo)


def _ints(n, lo, hi, g, dtype=torch.int32):
    return torch.randint(lo, hi + 1, (n,), generator=g, device="cuda", dtype=dtype)


def _extents(case):
    ext = [int(v) for v in case["extents"].split(",")]
    r = case["red_level"]
    return ext, math.prod(ext[:r]), math.prod(ext[r:])


def _rows_inputs(case, seed):
    _, O, R = _extents(case)
    g = _gen(seed)
    if case["prec"] in ("i32", "i64"):
        A = _ints(O * R, -1000, 1000, g)
        w = _ints(R, -1000, 1000, g)
    else:
        A = _normal(O * R, g)
        w = _uniform(R, -1.0, 1.0, g)
    return [A, w] if case["body"] == "dot_bcast" else [A]


@functools.lru_cache(maxsize=1)
def _zipf_cdf():
    k = np.arange(1, _MAX_LEN, dtype=np.float64)
    return np.append(np.cumsum(k ** -1.5) / _ZETA_1_5, 1.0)


def _mean_len():
    p = np.diff(np.concatenate([[0.0], _zipf_cdf()]))
    return float((p * np.arange(1, _MAX_LEN + 1)).sum())


def _csr_inputs(case, seed):
    """Zipf(1.5) row lengths clipped to 65536 (one draw per stratum, in random order, so that the
    number of entries hardly depends on the seed), uniform columns, normal values."""
    g = _gen(seed)
    n, m = case["rows"], case["cols"]
    u = (torch.arange(n, device="cuda", dtype=torch.float64)
         + torch.rand(n, generator=g, device="cuda", dtype=torch.float64)) / n
    cdf = torch.from_numpy(_zipf_cdf()).cuda()
    lens = (torch.searchsorted(cdf, u, right=True) + 1).clamp_(max=_MAX_LEN)
    lens = lens[torch.randperm(n, generator=g, device="cuda")]
    offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=offsets[1:])
    nnz = int(offsets[-1])
    return offsets, _ints(nnz, 0, m - 1, g), _normal(nnz, g), _normal(m, g)


_HIST_SHIFT = 10


def _bins(case):
    return ((case["cols"] - 1) >> _HIST_SHIFT) + 1


@functools.lru_cache(maxsize=4)
def _uneven(count, shape_seed, served):
    """Shapes of a batch or a burst of requests, with their places in packed buffers: for each
    (shape, buffer, first input element, first output element), and the buffers' sizes."""
    size = {"f": [0, 0], "i": [0, 0]}
    place = []
    for sh in synth.uneven_shapes(n_nests=count, seed=shape_seed):
        k = "f" if served or sh.op == "sum" else "i"
        place.append((sh, k, size[k][0], size[k][1]))
        size[k][0] += (sh.size + 3) // 4 * 4
        size[k][1] += (sh.n_out + 3) // 4 * 4
    return place, size


def _uneven_of(case):
    if case["kind"] == "batch":
        return _uneven(case["nests"], case["shape_seed"], False)
    return _uneven(case["requests"], case["shape_seed"], True)


def _uneven_inputs(case, seed):
    _, size = _uneven_of(case)
    g = _gen(seed)
    return {"f": _normal(max(size["f"][0], 4), g), "i": _ints(max(size["i"][0], 4), -(1 << 20), 1 << 20, g)}


def _stencil_coeffs(radius):
    if radius == 1:
        return list(synth.DIFFUSION9)
    k = (2 * radius + 1) ** 2
    c = np.random.Generator(np.random.PCG64(radius)).uniform(0.0, 1.0, k)
    return [float(np.float32(v)) for v in c / c.sum()]


def _stencil_input(case, seed):
    return _uniform(case["ny"] * case["nx"], -1.0, 1.0, _gen(seed)).view(case["ny"], case["nx"])


def _ordered_inputs(case, seed):
    n, g = case["rows"] * case["len"], _gen(seed)
    if case["op"] == "compose":
        return [_uniform(n, 0.9, 1.0, g), _normal(n, g)]
    if case["op"] == "mat2":
        p, q = _uniform(n, 0.0, 1.0, g), _uniform(n, 0.0, 1.0, g)
        return [torch.stack([1 - p, p, q, 1 - q], dim=-1).contiguous()]
    v = torch.where(_uniform(n, 0.0, 1.0, g) < 0.9, torch.full((n,), float("nan"), device="cuda"), _normal(n, g))
    v.view(case["rows"], case["len"])[:, 0] = 0.5      # every row has a value
    return [v]


def _narrow_inputs(case, seed):
    n, g = case["rows"] * case["len"], _gen(seed)
    dtype, half = (torch.int8, 128) if case["prec"] == "i8" else (torch.int16, 32768)
    ins = [_ints(n, -half, half - 1, g, dtype)]
    if case["body"] == "dot_bcast":
        ins.append(_ints(case["len"], -128, 127, g, torch.int8))
    return ins


# ---------------------------------------------------------------- the calls

_MAPS = {"auto": None,
         "cluster4x4": [("grid", 0, 0), ("grid", 0, 0), ("cluster", 4, 0), ("cta", 4, 0)],
         "cluster8x8": [("grid", 0, 0), ("grid", 0, 0), ("cluster", 8, 0), ("cta", 8, 0)]}


class _Server:
    """Owner of one server handle."""

    def __init__(self, budget, slots, streams):
        self.handle = hb.hp_serve_create(budget, slots, streams)

    def __del__(self):
        if self.handle:
            hb.hp_serve_destroy(self.handle)
            self.handle = None


def _out_dtype(prec):
    return {"f32": torch.float32, "f32_comp": torch.float32, "i64": torch.int64}.get(prec, torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(kind=kind)
    if kind == "rows":
        ext, O, _ = _extents(case)
        s.ins = _rows_inputs(case, seed)
        s.nest = hb.Nest(ext, case["red_level"], case["op"], case["prec"], case["body"], level_map=_MAPS[case["map"]])
        s.out = torch.empty(O, dtype=_out_dtype(case["prec"]), device="cuda")
        s.ptrs = [t.data_ptr() for t in s.ins]
    elif kind == "csr":
        s.ins = list(_csr_inputs(case, seed))
        n_bins = _bins(case)
        params = hb.hp_csr_params(s.ins[1].numel(), case["cols"], _HIST_SHIFT, int(case["hist"]), n_bins)
        s.nest = hb.Nest(csr_rows=case["rows"], red_level=1, op=case["op"], prec=case["prec"], body="csr_gather",
                         params=params)
        s.out = torch.empty(case["rows"], dtype=torch.float32, device="cuda")
        s.hist = torch.empty(n_bins, dtype=torch.int64, device="cuda") if case["hist"] else None
        s.ptrs = [t.data_ptr() for t in s.ins] + ([s.hist.data_ptr()] if case["hist"] else [])
    elif kind in ("batch", "serve"):
        place, size = _uneven_of(case)
        s.ins = _uneven_inputs(case, seed)
        s.out = {"f": torch.zeros(size["f"][1], dtype=torch.float32, device="cuda"),
                 "i": torch.zeros(size["i"][1], dtype=torch.int32, device="cuda")}
        s.nests = [hb.Nest(list(sh.extents), sh.red_level, "sum" if k == "f" else "max", "f32_comp" if k == "f" else "i32",
                           "load") for sh, k, _, _ in place]
        ins = [[s.ins[k].data_ptr() + 4 * i] for _, k, i, _ in place]
        outs = [s.out[k].data_ptr() + 4 * o for _, k, _, o in place]
        if kind == "batch":
            s.batch = hb.PreparedBatch([n.handle for n in s.nests], ins, outs)
        else:
            s.server = _Server(4 << 30, 4096, 4)
            s.requests = list(zip([n.handle for n in s.nests], ins, outs))
            torch.cuda.synchronize()      # inputs and outputs are ready before they are submitted
    elif kind == "stencil":
        s.ins = _stencil_input(case, seed)
        s.out = torch.empty_like(s.ins)
        s.stencil = hb.Stencil(case["ny"], case["nx"], case["radius"], _stencil_coeffs(case["radius"]), case["steps"])
    elif kind == "ordered":
        s.ins = _ordered_inputs(case, seed)
        s.nest = hb.Nest([case["rows"], case["len"]], 1, case["op"], "f32", "load")
        s.out = torch.empty(case["rows"], {"compose": 2, "mat2": 4, "last": 1}[case["op"]], dtype=torch.float32,
                            device="cuda")
        s.ptrs = [t.data_ptr() for t in s.ins]
    else:
        s.ins = _narrow_inputs(case, seed)
        s.nest = hb.Nest([case["rows"], case["len"]], 1, case["op"], case["prec"], case["body"])
        s.out = torch.empty(case["rows"], dtype=torch.int32, device="cuda")
        s.ptrs = [t.data_ptr() for t in s.ins]
    return s


def run(state):
    stream = torch.cuda.current_stream().cuda_stream
    if state.kind == "csr":
        state.nest.run(state.ptrs, state.out.data_ptr(), stream)
        return [state.out, state.hist] if state.hist is not None else [state.out]
    if state.kind == "batch":
        hb.hp_nest_run_batch(state.batch, stream=stream)
        return [state.out["f"], state.out["i"]]
    if state.kind == "serve":
        tickets = [hb.hp_serve_submit(state.server.handle, *req) for req in state.requests]
        for t in tickets:
            hb.hp_serve_poll(state.server.handle, t, -1)
        return state.out["f"]
    if state.kind == "stencil":
        state.stencil.run(state.ins.data_ptr(), state.out.data_ptr(), stream)
    else:
        state.nest.run(state.ptrs, state.out.data_ptr(), stream)
    return state.out


def work(case):
    kind = case["kind"]
    if kind == "rows":
        _, O, R = _extents(case)
        dot = case["body"] == "dot_bcast"
        return {"bytes": 4 * O * R + (4 * R if dot else 0) + (8 if case["prec"] == "i64" else 4) * O,
                "flops": (2 if dot else 1) * O * R}
    if kind == "csr":
        nnz = int(case["rows"] * _mean_len())
        return {"bytes": 8 * nnz + 8 * (case["rows"] + 1) + 4 * case["cols"] + 4 * case["rows"]
                + (8 * _bins(case) if case["hist"] else 0), "flops": 2 * nnz}
    if kind in ("batch", "serve"):
        place, _ = _uneven_of(case)
        n = sum(sh.size for sh, _, _, _ in place)
        return {"bytes": 4 * n + 4 * sum(sh.n_out for sh, _, _, _ in place), "flops": n}
    if kind == "stencil":
        n = case["ny"] * case["nx"]
        return {"bytes": 8 * n, "flops": 2 * (2 * case["radius"] + 1) ** 2 * case["steps"] * n}
    n = case["rows"] * case["len"]
    if kind == "ordered":
        per = {"compose": (8, 3, 2), "mat2": (16, 12, 4), "last": (4, 1, 1)}[case["op"]]
        return {"bytes": per[0] * n + 4 * per[2] * case["rows"], "flops": per[1] * n}
    dot = case["body"] == "dot_bcast"
    return {"bytes": (1 if case["prec"] == "i8" else 2) * n + (case["len"] if dot else 0) + 4 * case["rows"],
            "flops": (2 if dot else 1) * n}


# ---------------------------------------------------------------- 64-bit values

def _wrap32(v):
    return ((v + (1 << 31)) % (1 << 32) - (1 << 31)).to(torch.int32)


def _reduce(A, w, op, wide):
    """op over the rows of A (times w), elements widened to `wide`; a chunk at a time."""
    O, R = A.shape
    out = torch.empty(O, dtype=wide, device="cuda")
    rc = max(1, _CHUNK // max(R, 1))
    for i in range(0, O, rc):
        acc = None
        for j in range(0, R, _CHUNK):
            v = A[i:i + rc, j:j + _CHUNK].to(wide)
            if w is not None:
                v = v * w[j:j + _CHUNK].to(wide)
            part = v.sum(1) if op == "sum" else v.amax(1) if op == "max" else v.amin(1)
            if acc is None:
                acc = part
            else:
                acc = acc + part if op == "sum" else torch.maximum(acc, part) if op == "max" \
                    else torch.minimum(acc, part)
        out[i:i + rc] = acc
    return out


def _exact_csr(case, seed):
    offsets, col, val, x = _csr_inputs(case, seed)
    x64 = x.double()
    out = torch.empty(case["rows"], dtype=torch.float64, device="cuda")
    hist = torch.zeros(_bins(case), dtype=torch.int64, device="cuda")
    bounds = offsets.cpu().numpy()
    i = 0
    while i < case["rows"]:
        j = int(np.searchsorted(bounds, bounds[i] + _CHUNK, side="right")) - 1
        j = min(max(j, i + 1), case["rows"])
        lo, hi = int(bounds[i]), int(bounds[j])
        c = col[lo:hi].long()
        terms = val[lo:hi].double() * x64[c]
        lens = offsets[i + 1:j + 1] - offsets[i:j]
        out[i:j] = torch.segment_reduce(terms, case["op"], lengths=lens, unsafe=True)
        if case["hist"]:
            hist += torch.bincount(c >> _HIST_SHIFT, minlength=hist.numel())
        i = j
    return [out, hist] if case["hist"] else [out]


def _exact_uneven(case, seed):
    place, size = _uneven_of(case)
    ins = _uneven_inputs(case, seed)
    out = {"f": torch.zeros(size["f"][1], dtype=torch.float64, device="cuda"),
           "i": torch.zeros(size["i"][1], dtype=torch.int32, device="cuda")}
    for sh, k, i, o in place:
        A = ins[k][i:i + sh.size].view(sh.n_out, -1)
        out[k][o:o + sh.n_out] = A.double().sum(1) if k == "f" else A.amax(1)
    return out["f"] if case["kind"] == "serve" else [out["f"], out["i"]]


def _exact_stencil(case, seed):
    ny, nx, r = case["ny"], case["nx"], case["radius"]
    c = np.asarray(_stencil_coeffs(r), np.float32).astype(np.float64)
    v = torch.zeros(ny + 2 * r, nx + 2 * r, dtype=torch.float64, device="cuda")
    v[r:r + ny, r:r + nx] = _stencil_input(case, seed)
    for _ in range(case["steps"]):
        acc = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
        for dy in range(2 * r + 1):
            for dx in range(2 * r + 1):
                acc.add_(v[dy:dy + ny, dx:dx + nx], alpha=float(c[dy * (2 * r + 1) + dx]))
        v[r:r + ny, r:r + nx] = acc
    return acc


def _exact_ordered(case, seed):
    O, R = case["rows"], case["len"]
    ins = _ordered_inputs(case, seed)
    if case["op"] == "last":
        v = ins[0].view(O, R)
        idx = torch.arange(R, device="cuda").expand(O, R)
        last = torch.where(torch.isnan(v), -1, idx).amax(1)
        return v.gather(1, last[:, None]).double()
    if case["op"] == "compose":
        a, b = ins[0].view(O, R).double(), ins[1].view(O, R).double()
        while a.shape[1] > 1:
            n = a.shape[1] // 2 * 2
            a2, b2 = a[:, 1:n:2] * a[:, 0:n:2], a[:, 1:n:2] * b[:, 0:n:2] + b[:, 1:n:2]
            a, b = torch.cat([a2, a[:, n:]], 1), torch.cat([b2, b[:, n:]], 1)
        return torch.cat([a, b], 1)
    m = ins[0].view(O, R, 2, 2).double()
    while m.shape[1] > 1:
        n = m.shape[1] // 2 * 2
        e, l = m[:, 0:n:2], m[:, 1:n:2]
        p = torch.stack([l[..., 0, 0] * e[..., 0, 0] + l[..., 0, 1] * e[..., 1, 0],
                         l[..., 0, 0] * e[..., 0, 1] + l[..., 0, 1] * e[..., 1, 1],
                         l[..., 1, 0] * e[..., 0, 0] + l[..., 1, 1] * e[..., 1, 0],
                         l[..., 1, 0] * e[..., 0, 1] + l[..., 1, 1] * e[..., 1, 1]], -1)
        m = torch.cat([p.view(O, n // 2, 2, 2), m[:, n:]], 1)
    return m.reshape(O, 4)


def exact(case, seed):
    kind = case["kind"]
    if kind == "rows":
        _, O, R = _extents(case)
        ins = _rows_inputs(case, seed)
        wide = torch.int64 if case["prec"] in ("i32", "i64") else torch.float64
        v = _reduce(ins[0].view(O, R), ins[1] if len(ins) > 1 else None, case["op"], wide)
        return _wrap32(v) if case["prec"] == "i32" else v
    if kind == "csr":
        return _exact_csr(case, seed)
    if kind in ("batch", "serve"):
        return _exact_uneven(case, seed)
    if kind == "stencil":
        return _exact_stencil(case, seed)
    if kind == "ordered":
        return _exact_ordered(case, seed)
    ins = _narrow_inputs(case, seed)
    v = _reduce(ins[0].view(case["rows"], case["len"]), ins[1] if len(ins) > 1 else None, case["op"], torch.int64)
    return _wrap32(v)
