"""Workloads whose speed is tracked: what programs that use this library have it do.

Each case is one public call (or one wave of requests) at a size that comes
from the library's own workloads (bench.py, the tests), from the small calls
where launches count up to arrays that stream through the whole GPU, aligned
and ragged.  `listed()` names the fixed ones and says what each stands for;
`draw()` gives more of the same ranges.  Inputs are drawn on the device from
the seed alone; sizes and launch options come from the case alone.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2112_10034_gb300 import cox

MAX_N = 1 << 28
F32, I32 = "f32", "i32"
OPS = {"sum": cox.COX_SUM, "min": cox.COX_MIN, "max": cox.COX_MAX, "xor": cox.COX_XOR}


def listed():
    return [
        # Code 1's block sum (64 blocks x 256 threads), the smallest call: launch latency
        {"name": "block_sum_64x256", "kind": "reduce", "scope": "block", "dt": I32, "op": "sum", "n": 16384,
         "width": 32, "block": 256, "comp": False, "off": 0},
        # the shuffle scan on tiles at the width and mode that costs most
        {"name": "tile_scan_w16_comp_2p26", "kind": "tile_scan", "dt": F32, "n": 1 << 26, "width": 16, "comp": True,
         "off": 0},
        # an ordinary ragged scan: an odd length, narrow tiles
        {"name": "tile_scan_w4_1000003", "kind": "tile_scan", "dt": F32, "n": 1_000_003, "width": 4, "comp": False,
         "off": 0},
        # shfl_scan_test's first half: every 256-thread block scanned on its own
        {"name": "block_scan_b256_2p26", "kind": "scan", "scope": "block", "dt": F32, "n": 1 << 26, "block": 256,
         "comp": False, "exclusive": False, "off": 0},
        # a whole-array prefix sum of integers (offsets for a partition), the largest
        {"name": "grid_scan_i32_2p28", "kind": "scan", "scope": "grid", "dt": I32, "n": 1 << 28, "block": 256,
         "comp": False, "exclusive": False, "off": 0},
        # a cumulative sum that has to stay accurate, ragged
        {"name": "grid_scan_f32_comp_100000007", "kind": "scan", "scope": "grid", "dt": F32, "n": 100_000_007,
         "block": 256, "comp": True, "exclusive": False, "off": 0},
        # stream compaction at half density
        {"name": "compact_d50_2p28", "kind": "compact", "n": 1 << 28, "density": 0.5, "block": 256, "off": 0},
        # 256-bin histogram of Zipf keys from match_any groups
        {"name": "match_histogram_2p28", "kind": "histogram", "n": 1 << 28, "bins": 256, "width": 32, "block": 256,
         "off": 0},
        # 10,000 uneven arrays, a sum and a histogram each, one graph launch
        {"name": "batch_10000", "kind": "batch", "arrays": 10_000, "longest": 1 << 20, "lengths": 1},
        # a vector that fits on chip scaled to unit length (grid sync), as an iterative solver does each step
        {"name": "normalize_2p22", "kind": "grid_broadcast", "op": "normalize", "dt": F32, "n": 1 << 22, "off": 0},
        # integral images of a second of HD video
        {"name": "integral_u8_64x1080x1920", "kind": "integral", "dt": "u8", "batch": 64, "height": 1080,
         "width": 1920},
        # a wave of mixed requests at a server: reduce, scan and compact of 1K to 16M elements
        {"name": "serve_48_mixed", "kind": "serve", "requests": 48, "longest": 1 << 24, "lengths": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["reduce", "tile_scan", "block_scan", "grid_scan", "compact", "histogram", "batch",
                       "grid_broadcast", "integral", "serve"])
    off = rng.choice([0, 0, 0, 1])  # elements past the allocation's start: views such as x[1:]
    width = rng.choice([2, 4, 8, 16, 32])
    block = rng.choice([32, 64, 128, 256, 512, 1024, 96, 320])
    dt = rng.choice([F32, I32])
    comp = dt == F32 and rng.random() < 0.5
    if kind == "reduce":
        return {"kind": kind, "scope": rng.choice(["tile", "block", "grid"]), "dt": dt,
                "op": "sum" if comp else rng.choice(["sum", "min", "max"] + ["xor"] * (dt == I32)),
                "n": _log(rng, 1000, MAX_N), "width": width, "block": block, "comp": comp, "off": off}
    if kind == "tile_scan":
        return {"kind": kind, "dt": dt, "n": _log(rng, 1000, 1 << 26), "width": width, "comp": comp, "off": off}
    if kind in ("block_scan", "grid_scan"):
        return {"kind": "scan", "scope": kind[:-5], "dt": dt, "n": _log(rng, 1000, 1 << 27), "block": block,
                "comp": comp, "exclusive": rng.random() < 0.5, "off": off}
    if kind == "compact":
        return {"kind": kind, "n": _log(rng, 1000, MAX_N), "density": rng.choice([0.1, 0.5, 0.9]), "block": block,
                "off": off}
    if kind == "histogram":
        return {"kind": kind, "n": _log(rng, 1000, MAX_N), "bins": rng.choice([256, 256, 256, 64, 1000]),
                "width": width, "block": rng.choice([128, 256, 512]), "off": off}
    if kind == "batch":
        return {"kind": kind, "arrays": _log(rng, 100, 10_000), "longest": _log(rng, 1 << 10, 1 << 20),
                "lengths": rng.randrange(2, 1 << 20)}
    if kind == "grid_broadcast":
        op = rng.choice(["normalize", "sub_min"])
        return {"kind": kind, "op": op, "dt": F32 if op == "normalize" else dt, "n": _log(rng, 1000, 1 << 26),
                "off": off}
    if kind == "integral":
        height, width = _log(rng, 64, 2160), 4 * _log(rng, 24, 960) + rng.choice([0, 0, 0, 1])
        return {"kind": kind, "dt": rng.choice(["u8", "i32"]), "batch": rng.randint(1, max(1, min(64, (1 << 27) // (height * width)))),
                "height": height, "width": width}
    return {"kind": "serve", "requests": rng.randint(1, 60), "longest": _log(rng, 1 << 14, 1 << 24),
            "lengths": rng.randrange(2, 1 << 20)}


# ------------------------------------------------------------------ inputs
DEV = "cuda"


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _view(t, off):
    """t's values starting `off` elements past a 16-byte boundary."""
    if not off:
        return t
    b = torch.empty(t.numel() + off, dtype=t.dtype, device=t.device)
    b[off:].copy_(t)
    return b[off:]


def _values(dt, n, g, off=0):
    """N(0, 1) floats, or integers in [-1000, 1000]."""
    if dt == F32:
        return _view(torch.randn(n, generator=g, device=DEV), off)
    return _view(torch.randint(-1000, 1001, (n,), generator=g, device=DEV, dtype=torch.int32), off)


def _uniform_keys(n, g, off=0):
    return _view(torch.randint(0, (1 << 31) - 1, (n,), generator=g, device=DEV, dtype=torch.int32), off)


def _half_kept_keys(n, g):
    """Uniform keys of which exactly n - n // 2 are below half of the range, in random places."""
    k = torch.randint(0, 1 << 30, (n,), generator=g, device=DEV, dtype=torch.int32)
    k[torch.randperm(n, generator=g, device=DEV)[:n // 2]] += 1 << 30
    return k


def _zipf_keys(n, g, bins=256, off=0):
    """Keys in [0, bins), P(k) proportional to (k + 1)^-1.1."""
    w = torch.arange(1, bins + 1, dtype=torch.float64, device=DEV) ** -1.1
    cdf = torch.cumsum(w / w.sum(), 0).float()
    cdf[-1] = 1.0
    k = torch.empty(n, dtype=torch.int32, device=DEV)
    for c in range(0, n, 1 << 27):
        u = torch.rand(min(1 << 27, n - c), generator=g, device=DEV)
        torch.searchsorted(cdf, u, right=True, out_int32=True, out=k[c:c + u.numel()])
    return _view(k, off)


def _lengths(case, shortest):
    count = case["arrays"] if case["kind"] == "batch" else case["requests"]
    r = random.Random(case["lengths"])
    top = max(shortest, case["longest"])
    return [min(top, int(math.exp(r.uniform(math.log(shortest), math.log(top))))) for _ in range(count)]


def _threshold(density):
    return int(density * (1 << 31))


def _request_plan(case):
    """(what, dt, width, comp) of each request: thirds of reduces, scans, compactions."""
    r = random.Random(case["lengths"] + 1)
    plan = []
    for i in range(case["requests"]):
        what = ("reduce", "scan", "compact")[r.randrange(3)]
        dt = I32 if what == "compact" or (what == "reduce" and r.random() < 0.5) else F32
        plan.append((what, dt, r.choice([4, 8, 16, 32]), dt == F32))
    return plan


def _data(case, seed):
    """The input tensors of a case."""
    g, k = _gen(seed), case["kind"]
    if k in ("reduce", "tile_scan", "scan", "grid_broadcast"):
        return _values(case["dt"], case["n"], g, case["off"])
    if k == "compact":
        return _uniform_keys(case["n"], g, case["off"])
    if k == "histogram":
        return _zipf_keys(case["n"], g, case["bins"], case["off"])
    if k == "batch":
        lens = _lengths(case, 32)
        starts, total = [], 0
        for n in lens:
            starts.append(total)
            total += (n + 3) // 4 * 4  # every array 16-byte aligned
        vals, keys = torch.randn(total, generator=g, device=DEV), _zipf_keys(total, g)
        return [vals[s:s + n] for s, n in zip(starts, lens)], [keys[s:s + n] for s, n in zip(starts, lens)]
    if k == "integral":
        shape = (case["batch"], case["height"], case["width"])
        t = torch.randint(0, 256, shape, generator=g, device=DEV, dtype=torch.uint8)
        return t if case["dt"] == "u8" else t.int()
    assert k == "serve"
    xs = []
    for (what, dt, _, _), n in zip(_request_plan(case), _lengths(case, 1024)):
        xs.append(_half_kept_keys(n, g) if what == "compact" else _values(dt, n, g))
    return xs


# --------------------------------------------------------------- the calls
SCOPE = {"tile": cox.COX_SCOPE_TILE, "block": cox.COX_SCOPE_BLOCK, "grid": cox.COX_SCOPE_GRID}


def prepare(case, seed):
    x, k = _data(case, seed), case["kind"]
    s = {"case": case, "x": x}
    if k == "compact":  # a caller keeps its output room and scratch
        s["out"] = torch.zeros(case["n"], dtype=torch.int32, device=DEV)
        s["count"] = torch.zeros(1, dtype=torch.int64, device=DEV)
        s["ws"] = torch.empty(cox.cox_ballot_compact_workspace(case["n"], case["block"]), dtype=torch.uint8,
                              device=DEV)
    elif k == "batch":  # the prepared batch and its captured graph
        s["batch"] = cox.Batch(*x)
        s["graph"] = s["batch"].graph()
    elif k == "integral":
        s["out"] = torch.empty(x.shape, dtype=torch.int32, device=DEV)
        s["ws_bytes"] = cox.cox_integral_image_workspace(*x.shape)
        s["ws"] = torch.empty(s["ws_bytes"], dtype=torch.uint8, device=DEV)
    elif k == "serve":
        s["reqs"] = [cox.make_request({"reduce": cox.COX_REQ_REDUCE, "scan": cox.COX_REQ_SCAN,
                                       "compact": cox.COX_REQ_COMPACT}[what], t, width, comp, _threshold(0.5))
                     for (what, _, width, comp), t in zip(_request_plan(case), x)]
        torch.cuda.synchronize()  # the server reads the inputs on its own streams
        s["server"] = cox.Server(8 << 30)
    return s


def run(s):
    c, x = s["case"], s["x"]
    k = c["kind"]
    if k == "reduce":
        return cox.tile_reduce(x, OPS[c["op"]], c["width"], c["block"], SCOPE[c["scope"]], c["comp"])
    if k == "tile_scan":
        return cox.tile_scan(x, cox.COX_SUM, c["width"], 256, c["comp"])
    if k == "scan":
        return cox.scan(x, cox.COX_SUM, SCOPE[c["scope"]], c["block"], c["comp"], c["exclusive"])
    if k == "compact":
        return cox.ballot_compact(x, _threshold(c["density"]), 32, c["block"], workspace=s["ws"], out=s["out"],
                                  count=s["count"])
    if k == "histogram":
        return cox.match_histogram(x, c["bins"], c["width"], c["block"])
    if k == "batch":
        s["graph"].launch()
        b = s["batch"]
        return b.sums, b.sums64, b.hists
    if k == "grid_broadcast":
        return cox.grid_broadcast(x, cox.COX_GRID_NORMALIZE if c["op"] == "normalize" else cox.COX_GRID_SUB_MIN)
    if k == "integral":
        status = cox.cox_integral_image(cox.COX_U8 if c["dt"] == "u8" else cox.COX_I32, *x.shape, x.data_ptr(),
                                        s["out"].data_ptr(), s["ws"].data_ptr(), s["ws_bytes"],
                                        torch.cuda.current_stream().cuda_stream)
        if status != cox.COX_OK:
            raise cox.CoxError(status, "cox_integral_image")
        return s["out"]
    srv, reqs = s["server"], s["reqs"]
    tickets = srv.submit_many(reqs)
    outs = []
    for t, r in zip(tickets, reqs):
        srv.wait(t)
        outs.append(srv.result(t, r))
    torch.cuda.current_stream().synchronize()  # the copies are made before their arena memory is given back
    for t in tickets:
        srv.release(t)
    return outs


# -------------------------------------------------------- sizes and values
def work(case):
    """Every input read once and every output written once; one operation per element and combine."""
    k = case["kind"]
    if k == "reduce":
        n = case["n"]
        m = {"tile": -(-n // case["width"]), "block": -(-n // case["block"]), "grid": 1}[case["scope"]]
        return {"bytes": 4 * (n + m), "flops": n}
    if k in ("tile_scan", "scan", "grid_broadcast"):
        return {"bytes": 8 * case["n"], "flops": case["n"]}
    if k == "compact":
        return {"bytes": 4 * case["n"] * (1 + case["density"]), "flops": case["n"]}
    if k == "histogram":
        return {"bytes": 4 * (case["n"] + case["bins"]), "flops": case["n"]}
    if k == "batch":
        e = sum(_lengths(case, 32))
        return {"bytes": 8 * e + case["arrays"] * (12 + 1024), "flops": 2 * e}
    if k == "integral":
        p = case["batch"] * case["height"] * case["width"]
        return {"bytes": p * (5 if case["dt"] == "u8" else 8), "flops": 2 * p}
    per = {"reduce": 4, "scan": 8, "compact": 6}
    b = sum(per[p[0]] * n for p, n in zip(_request_plan(case), _lengths(case, 1024)))
    return {"bytes": b, "flops": b // 8}


def _segments(x, seg, fill=0):
    """x as rows of `seg` elements, the last one padded."""
    rows = -(-x.numel() // seg)
    p = torch.full((rows * seg,), fill, dtype=x.dtype, device=x.device)
    p[:x.numel()] = x
    return p.view(rows, seg)


def _wrap(t):
    return t.to(torch.int32)  # int64 sums modulo 2^32


def _scan_exact(x, seg, exclusive):
    n, whole = x.numel(), x.dtype == torch.int32
    v = _segments(x.long() if whole else x.double(), seg)
    y = v.cumsum(1)
    if exclusive:
        y -= v
    y = y.view(-1)[:n]
    return _wrap(y) if whole else y


def _reduce_exact(x, seg, op):
    whole = x.dtype == torch.int32
    if op == "xor":
        v = _segments(x, seg)
        while v.shape[1] > 1:
            if v.shape[1] % 2:
                v = torch.cat([v, torch.zeros_like(v[:, :1])], 1)
            v = v[:, 0::2] ^ v[:, 1::2]
        return v[:, 0].contiguous()
    if op == "sum":
        y = _segments(x.long() if whole else x.double(), seg).sum(1)
        return _wrap(y) if whole else y
    fill = {("min", True): (1 << 31) - 1, ("max", True): -(1 << 31), ("min", False): math.inf,
            ("max", False): -math.inf}[op, whole]
    v = _segments(x if whole else x.double(), seg, fill)
    return v.amin(1) if op == "min" else v.amax(1)


def _compact_exact(x, density):
    return x[x < _threshold(density)]


def exact(case, seed):
    x, k = _data(case, seed), case["kind"]
    if k == "reduce":
        seg = {"tile": case["width"], "block": case["block"], "grid": case["n"]}[case["scope"]]
        return _reduce_exact(x, seg, case["op"])
    if k == "tile_scan":
        return _scan_exact(x, case["width"], False)
    if k == "scan":
        return _scan_exact(x, case["block"] if case["scope"] == "block" else case["n"], case["exclusive"])
    if k == "compact":
        out = torch.zeros_like(x)
        kept = _compact_exact(x, case["density"])
        out[:kept.numel()] = kept
        return out, torch.tensor([kept.numel()], device=DEV)
    if k == "histogram":
        h = torch.zeros(case["bins"], dtype=torch.int64, device=DEV)
        for c in x.split(1 << 27):
            h += torch.bincount(c, minlength=case["bins"])
        return h.int(), torch.zeros(1, dtype=torch.int64, device=DEV)
    if k == "batch":
        vals, keys = x
        sums = torch.stack([v.double().sum() for v in vals])
        return sums, sums, torch.stack([torch.bincount(q, minlength=256) for q in keys]).int()
    if k == "grid_broadcast":
        if case["op"] == "normalize":
            d = x.double()
            return d / d.square().sum().sqrt()
        return x.double() - x.double().min() if case["dt"] == F32 else x - x.min()
    if k == "integral":
        return torch.stack([_wrap(i.long().cumsum(0).cumsum(1)) for i in x])
    outs = []
    for (what, dt, width, _), t in zip(_request_plan(case), x):
        if what == "compact":
            outs.append(_compact_exact(t, 0.5))
        elif what == "scan":
            outs.append(_scan_exact(t, width, False))
        elif dt == F32:
            total = t.double().sum()
            outs.append(torch.stack([total, total - total.float().double()]))
        else:
            outs.append(torch.stack([_wrap(t.long().sum()), torch.zeros((), dtype=torch.int32, device=DEV)]))
    return outs
