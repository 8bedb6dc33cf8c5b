"""The work that users of this library have it do, as cases that can be timed.

Each case is a dict of plain values.  ``prepare`` makes what a program has in
hand before the call (matrix, plan, handles, vectors, streams), ``run`` makes
one pass through the public entry points and returns what it computes,
``work`` counts the bytes and operations that the pass cannot do without, and
``exact`` gives the same outputs from plain 64-bit tensor arithmetic.

Paths:
  schedule  one partitioned product through ``spmv_schedule_run``: issued
            eagerly or replayed as a captured graph
  merge     the plan-free CSR product on device arrays (``spmv_csr_merge`` and
            its no-allocation form)
  batch     many independent products in one persistent launch
  single    one multi-right-hand-side serving request alone
  burst     a queue of serving requests through the serving loop
  host      a stream of products through pinned host buffers

Matrices: 5- and 7-point and 27-point stencils, the random band matrix and
random matrices with Zipf row lengths, with the recipes of
``paper_2203_02530_gb300/workloads.py`` (drawn on the GPU here, which is
faster).
"""
import itertools
import math

import numpy as np
import torch

from paper_2203_02530_gb300 import spmv

VARIANTS = {"tile": spmv.VARIANT_TILE, "vector": spmv.VARIANT_VECTOR, "merge": spmv.VARIANT_MERGE,
            "sell": spmv.VARIANT_SELL, "sell16": spmv.VARIANT_SELL16}


def listed():
    return [
        # the smallest configuration: a 64 x 64 grid, one stream, the default
        # order, replayed; a solver's inner loop on a problem that fits in L2
        {"name": "lap64_replay", "path": "schedule", "matrix": "5pt", "g": 64, "P": 2, "streams": 1,
         "granularity": "coarse", "mode": "replay", "local": "sell16:9", "remote": "sell:4"},
        # the random band matrix of the paper, 150 000 rows, four ranks, two
        # streams; replayed
        {"name": "band150k_replay", "path": "schedule", "matrix": "band", "n": 150000, "P": 4, "streams": 2,
         "granularity": "coarse", "mode": "replay", "local": "sell:8", "remote": "sell:8"},
        # a program that tunes nothing: the plan as created, issued eagerly on
        # one stream; a stencil with ragged sides
        {"name": "st27_default_eager", "path": "schedule", "matrix": "27pt", "g": 91, "P": 4, "streams": 1,
         "granularity": "coarse", "mode": "eager", "local": "tile:0", "remote": "tile:0"},
        # the 27-point stencil on 150^3 with the tuned variants and the best
        # program's streams: the largest product
        {"name": "st27_150_replay", "path": "schedule", "matrix": "27pt", "g": 150, "P": 4, "streams": 2,
         "granularity": "coarse", "mode": "replay", "local": "sell16:107", "remote": "sell:8"},
        # skewed rows, one operation per rank on four streams (a sampled
        # program of the 32-operation DAG), tuned variants
        {"name": "powerlaw_ranks_replay", "path": "schedule", "matrix": "powerlaw", "n": 2000000, "P": 8,
         "streams": 4, "granularity": "rank", "mode": "replay", "local": "sell:2105", "remote": "sell:105"},
        # the plan-free product on a caller's skewed matrix
        {"name": "merge_powerlaw", "path": "merge", "matrix": "powerlaw", "n": 700001, "noalloc": False},
        # the same inside a latency-bound loop that must not allocate: a
        # small stencil of odd size
        {"name": "merge_noalloc_small", "path": "merge", "matrix": "7pt", "g": 23, "noalloc": True},
        # 48 uneven matrices (stencils and Zipf rows), the tuner's layout
        {"name": "batch48_sliced", "path": "batch", "count": 48, "n_lo": 1000, "n_hi": 1000000, "lanes": 64},
        # a few small matrices as the batch is created, nothing tuned
        {"name": "batch12_default", "path": "batch", "count": 12, "n_lo": 1000, "n_hi": 30000, "lanes": 2},
        # one wide request alone over a skewed matrix
        {"name": "single_powerlaw_w8", "path": "single", "matrix": "zipf", "n": 600000, "width": 8},
        # a burst of 200 requests over 12 resident matrices: a server behind
        # its arrivals
        {"name": "burst200", "path": "burst", "count": 12, "n_lo": 10000, "n_hi": 1000000, "requests": 200,
         "streams": 32},
        # four products of a stream of right-hand sides that live on the host
        {"name": "host_many_st27", "path": "host", "matrix": "27pt", "g": 80, "P": 4, "products": 4,
         "local": "sell16:107", "remote": "sell:8"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["schedule"] * 5 + ["merge"] * 2 + ["batch"] * 2 + ["single"] * 2 + ["burst", "host"])
    if path == "schedule":
        matrix = rng.choice(["5pt", "7pt", "27pt", "band", "powerlaw"])
        c = {"path": path, "matrix": matrix}
        if matrix == "5pt":
            c["g"] = _log(rng, 32, 2000)
        elif matrix == "7pt":
            c["g"] = _log(rng, 12, 130)
        elif matrix == "27pt":
            c["g"] = _log(rng, 10, 130)
        else:
            c["n"] = _log(rng, 5000, 150000 if matrix == "band" else 2000000)
        c["P"] = rng.choice([1, 2, 3, 4, 8])
        c["granularity"] = rng.choice(["coarse", "coarse", "rank"])
        c["streams"] = rng.choice([1, 2, 4] if c["granularity"] == "rank" else [1, 2])
        c["mode"] = rng.choice(["replay", "replay", "eager"])
        stencil = matrix in ("5pt", "7pt", "27pt")
        tuned = ["sell16:107:8", "sell16:9:4", "sell:105:105"] if stencil else ["sell:2105:105", "sell:8:8", "sell:4:4"]
        pick = rng.choice(tuned + ["tile:0:0", "vector:2:2" if stencil else "merge:0:0"]).split(":")
        c["local"] = pick[0] + ":" + pick[1]
        c["remote"] = pick[0].replace("sell16", "sell") + ":" + pick[2]
        return c
    if path == "merge":
        if rng.random() < 0.5:
            return {"path": path, "matrix": "7pt", "g": _log(rng, 10, 110), "noalloc": rng.random() < 0.5}
        return {"path": path, "matrix": "powerlaw", "n": _log(rng, 2000, 1000000), "noalloc": rng.random() < 0.5}
    if path == "batch":
        lo = _log(rng, 500, 4000)
        return {"path": path, "count": rng.randint(3, 48), "n_lo": lo, "n_hi": _log(rng, 2 * lo, 1000000),
                "lanes": rng.choice([2, 64, 64])}
    if path == "single":
        if rng.random() < 0.5:
            return {"path": path, "matrix": "7pt", "g": _log(rng, 20, 100), "width": rng.randint(1, 8)}
        return {"path": path, "matrix": "zipf", "n": _log(rng, 10000, 800000), "width": rng.randint(1, 8)}
    if path == "burst":
        lo = _log(rng, 5000, 20000)
        return {"path": path, "count": rng.randint(2, 12), "n_lo": lo, "n_hi": _log(rng, 2 * lo, 800000),
                "requests": _log(rng, 20, 200), "streams": rng.choice([8, 32])}
    return {"path": path, "matrix": "27pt", "g": _log(rng, 20, 90), "P": rng.choice([2, 4]),
            "products": rng.randint(1, 4), "local": "sell16:107", "remote": "sell:8"}


# ---------------------------------------------------------------- matrices
# (n, row_ptr int64, col int32, val float64), all on the GPU

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(size, gen):
    return torch.rand(size, generator=gen, dtype=torch.float64, device="cuda") * 2.0 - 1.0


def _stencil(dims, box, diag, gen):
    nd = len(dims)
    n = math.prod(dims)
    if box:
        offsets = list(itertools.product((-1, 0, 1), repeat=nd))
    else:
        offsets = sorted([(0,) * nd] + [tuple(s if i == d else 0 for i in range(nd))
                                        for d in range(nd) for s in (-1, 1)])
    stride = [math.prod(dims[d + 1:]) for d in range(nd)]
    row = torch.arange(n, dtype=torch.int64, device="cuda")
    coord = [(row // stride[d]) % dims[d] for d in range(nd)]
    valid = torch.ones((n, len(offsets)), dtype=torch.bool, device="cuda")
    col = torch.empty((n, len(offsets)), dtype=torch.int32, device="cuda")
    for j, off in enumerate(offsets):
        for d in range(nd):
            if off[d] < 0:
                valid[:, j] &= coord[d] > 0
            elif off[d] > 0:
                valid[:, j] &= coord[d] < dims[d] - 1
        col[:, j] = (row + sum(o * s for o, s in zip(off, stride))).to(torch.int32)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(valid.sum(1), 0, out=ptr[1:])
    col = col[valid]
    val = _uniform(col.numel(), gen)
    centre = offsets.index((0,) * nd)
    val[ptr[:-1] + valid[:, :centre].sum(1)] = diag
    return n, ptr, col, val


def _rows(n, row, col, gen):
    """CSR of the distinct positions (row, col), columns ascending."""
    key = torch.unique(row * n + col)
    row = key // n
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(row, minlength=n), 0, out=ptr[1:])
    return n, ptr, (key - row * n).to(torch.int32), _uniform(key.numel(), gen)


def _zipf_cdf(cap):
    p = 1.0 / np.arange(1, cap + 1, dtype=np.float64) ** 2
    return np.cumsum(p / p.sum())


def _powerlaw(n, mult, cap, gen):
    """Row lengths min(cap, mult K), K ~ Zipf(2) on [1, cap]; 80 % of the
    columns within n/8 of the row, the others anywhere."""
    cdf = torch.from_numpy(_zipf_cdf(cap)).cuda()
    k = torch.searchsorted(cdf, torch.rand(n, generator=gen, dtype=torch.float64, device="cuda")) + 1
    length = torch.clamp(mult * torch.clamp(k, max=cap), max=cap)
    row = torch.repeat_interleave(torch.arange(n, dtype=torch.int64, device="cuda"), length)
    w = n // 8
    lo, hi = torch.clamp(row - w, min=0), torch.clamp(row + w, max=n - 1)
    u = torch.rand(row.numel(), generator=gen, dtype=torch.float64, device="cuda")
    near = torch.rand(row.numel(), generator=gen, dtype=torch.float64, device="cuda") < 0.8
    col = torch.where(near, lo + (u * (hi - lo + 1)).to(torch.int64), (u * n).to(torch.int64))
    return _rows(n, row, col, gen)


def _band(n, gen):
    """10 n positions uniform in the band of half width n / 4."""
    row = torch.randint(0, n, (10 * n,), generator=gen, device="cuda")
    col = row + torch.randint(-(n // 4), n // 4 + 1, (10 * n,), generator=gen, device="cuda")
    inside = (col >= 0) & (col < n)
    return _rows(n, row[inside], col[inside], gen)


def _matrix(kind, size, gen):
    if kind == "5pt":
        return _stencil((size, size), False, 5.0, gen)
    if kind == "7pt":
        return _stencil((size, size + 1, size), False, 7.0, gen)
    if kind == "27pt":
        return _stencil((size, size, size), True, 27.0, gen)
    if kind == "band":
        return _band(size, gen)
    if kind == "zipf":   # the batch's and the server's Zipf rows
        return _powerlaw(size, 2, max(1, min(4096, size // 4)), gen)
    return _powerlaw(size, 3, min(4096, size // 4), gen)


def _size(kind, size):
    """Rows and (expected) entries."""
    if kind == "5pt":
        return size * size, 5 * size * size - 4 * size
    if kind == "7pt":
        a, b = size, size + 1
        return a * a * b, 7 * a * a * b - 4 * a * b - 2 * a * a
    if kind == "27pt":
        return size ** 3, (3 * size - 2) ** 3
    if kind == "band":
        return size, int(10 * size * 0.875)
    mult, cap = (2, max(1, min(4096, size // 4))) if kind == "zipf" else (3, min(4096, size // 4))
    p = np.diff(np.concatenate([[0.0], _zipf_cdf(cap)]))
    return size, int(size * float((p * np.minimum(cap, mult * np.arange(1, cap + 1))).sum()))


def _host(m):
    n, ptr, col, val = m
    return n, ptr.cpu().numpy(), col.cpu().numpy(), val.cpu().numpy()


def _mix(case):
    """(kind, size) of every matrix of a batch: sizes spread evenly over the
    logarithm, small and large ones in turn."""
    kinds = ("5pt", "7pt", "zipf") if case["path"] == "batch" else ("7pt", "zipf")
    count, out = case["count"], []
    for i in range(count):
        at = (i * 7 % count + 0.5) / count if count % 7 else (i + 0.5) / count
        n = case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** at
        kind = kinds[i % len(kinds)]
        power = {"5pt": 1 / 2, "7pt": 1 / 3, "zipf": 1}[kind]
        out.append((kind, max(2, int(round(n ** power)))))
    return out


# ------------------------------------------------------------------ states

class _Handles:
    """Closes a state's handles with it, the last one first."""

    def __init__(self, *handles):
        self.handles = handles

    def __del__(self):
        for h in reversed(self.handles):
            h.close()


def _variant(text):
    kind, param = text.split(":")
    return VARIANTS[kind], int(param)


def _part(case, m, granularity=spmv.COARSE):
    part = spmv.Part(*_host(m), case["P"], granularity)
    for op, text in ((spmv.OP_LOCAL, case["local"]), (spmv.OP_REMOTE, case["remote"])):
        if text != "tile:0":   # a plan starts with that one
            part.set_op_variant(op, *_variant(text))
    return part


def _sell16_fits(case):
    """The 16-bit layout needs every local column within 32767 rows."""
    if case["matrix"] == "27pt":
        return case["g"] ** 2 + case["g"] + 1 <= 32767
    if case["matrix"] == "7pt":
        return case["g"] * (case["g"] + 1) <= 32767
    return True


def _program(case):
    """The order of the operations and their streams."""
    S, P = case["streams"], case["P"]
    if case["granularity"] == "coarse":   # the exchange on a stream of its own when there are two
        return [0, 1, 2, 3], [0, 0, 1 if S > 1 else 0, 0]
    order = [4 * p + k for k in range(4) for p in range(P)]
    return order, [(v // 4) % S for v in range(4 * P)]


def prepare(case, seed):
    gen = _generator(seed)
    path = case["path"]
    if path in ("schedule", "merge", "host"):
        m = _matrix(case["matrix"], case["g"] if "g" in case else case["n"], gen)
        n = m[0]
    if path == "schedule":
        if case["local"].startswith("sell16") and not _sell16_fits(case):
            case = dict(case, local=case["local"].replace("sell16", "sell"))
        gran = spmv.COARSE if case["granularity"] == "coarse" else spmv.PER_PARTITION
        part = _part(case, m, gran)
        x, y = _uniform(n, gen), torch.zeros(n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(case["streams"])]
        order, smap = _program(case)
        order, smap = np.array(order, dtype=np.int32), np.array(smap, dtype=np.int32)
        state = {"path": path, "own": _Handles(part), "part": part, "x": x, "y": y, "streams": streams,
                 "order": order, "map": smap, "flags": spmv.RUN_EAGER, "graph": 0}
        if case["mode"] == "replay":
            more = spmv.RUN_RELAXED | spmv.RUN_DEFER if case["granularity"] == "coarse" and case["streams"] > 1 else 0
            state["graph"] = part.run(order, smap, streams, x, y, spmv.RUN_CAPTURE | more)
            state["flags"] = spmv.RUN_REPLAY
        return state
    if path == "merge":
        x, y = _uniform(n, gen), torch.zeros(n, dtype=torch.float64, device="cuda")
        call = spmv.spmv_csr_merge_noalloc if case["noalloc"] else spmv.spmv_csr_merge
        return {"path": path, "call": call, "n": n, "nnz": m[2].numel(), "ptr": m[1].to(torch.int32), "col": m[2],
                "val": m[3], "x": x, "y": y, "stream": torch.cuda.current_stream()}
    if path == "host":
        part = _part(case, m)
        k = case["products"]
        x = _uniform((k, n), gen).cpu().pin_memory()
        y = torch.zeros((k, n), dtype=torch.float64).pin_memory()
        return {"path": path, "own": _Handles(part), "part": part, "x": x, "y": y, "n": n, "count": k,
                "in": torch.cuda.Stream(), "compute": torch.cuda.Stream()}
    if path == "single":
        m = _matrix(case["matrix"], case["g"] if "g" in case else case["n"], gen)
        batch = spmv.Batch([_host(m)])
        spmv.spmv_batch_set_lanes(batch.h, -1, spmv.BATCH_SLICED)
        server = spmv.Server(batch, n_streams=1)
        shape = (m[0], case["width"])
        x, y = (torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(2))
        return {"path": path, "own": _Handles(batch, server), "server": server, "x": x, "y": y,
                "width": case["width"], "seed": seed * 7919 + 1, "stream": torch.cuda.current_stream()}
    mats = [_matrix(kind, size, gen) for kind, size in _mix(case)]
    batch = spmv.Batch([_host(m) for m in mats])
    if path == "batch":
        if case["lanes"] != 2:   # a batch starts with two lanes a row
            spmv.spmv_batch_set_lanes(batch.h, -1, case["lanes"])
        rows = sum(m[0] for m in mats)
        x, y = _uniform(rows, gen), torch.zeros(rows, dtype=torch.float64, device="cuda")
        return {"path": path, "own": _Handles(batch), "batch": batch, "x": x, "y": y,
                "stream": torch.cuda.current_stream()}
    spmv.spmv_batch_set_lanes(batch.h, -1, spmv.BATCH_SLICED)
    server = spmv.Server(batch, n_streams=case["streams"])
    rng = np.random.default_rng(seed)
    k = case["requests"]
    # every request is there at the start; matrices and widths in a fixed
    # proportion, in an order of the seed
    return {"path": path, "own": _Handles(batch, server), "server": server,
            "matrix": rng.permutation(np.arange(k) % case["count"]).astype(np.int32),
            "width": rng.permutation(np.arange(k) % 8 + 1).astype(np.int32),
            "seed": rng.integers(0, 2 ** 63, size=k, dtype=np.uint64), "arrival": np.zeros(k)}


def run(state):
    path = state["path"]
    if path == "schedule":
        state["part"].run(state["order"], state["map"], state["streams"], state["x"], state["y"], state["flags"],
                          state["graph"])
        return state["y"]
    if path == "merge":
        state["call"](state["n"], state["nnz"], state["ptr"], state["col"], state["val"], state["x"], state["y"],
                      state["stream"])
        return state["y"]
    if path == "batch":
        spmv.spmv_batch_run(state["batch"].h, state["x"], state["y"], state["stream"])
        return state["y"]
    if path == "single":
        spmv.spmv_serve_single(state["server"].h, 0, state["width"], state["seed"], state["y"], state["x"],
                               state["stream"])
        return {"x": state["x"], "y": state["y"]}
    if path == "burst":   # the loop returns a hash of every request's result
        _, hashes, _ = state["server"].run(state["matrix"], state["width"], state["seed"], state["arrival"])
        return hashes.view(np.int64)
    spmv.spmv_apply_host_many(state["part"].h, state["count"], state["x"], state["n"], state["y"], state["n"],
                              spmv.HOST_Y_PARTS, state["in"], state["compute"])
    return state["y"]


def work(case):
    path = case["path"]

    def product(n, nnz, width=1):
        return {"bytes": 12 * nnz + 4 * (n + 1) + 16 * n * width, "flops": 2 * nnz * width}

    if path == "batch":
        each = [product(*_size(kind, size)) for kind, size in _mix(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    if path == "burst":
        # the matrices once, and X (drawn, then read) and Y of every request
        sizes = [_size(kind, size) for kind, size in _mix(case)]
        columns = 4.5 * case["requests"] / len(sizes)
        return {"bytes": int(sum(12 * z + 4 * n + 16 * n * columns for n, z in sizes)),
                "flops": int(sum(2 * z * columns for n, z in sizes))}
    n, nnz = _size(case["matrix"], case["g"] if "g" in case else case["n"])
    if path == "host":
        return {"bytes": case["products"] * product(n, nnz)["bytes"], "flops": case["products"] * 2 * nnz}
    return product(n, nnz, case.get("width", 1))


# ------------------------------------------------------------------- exact

def _halves(a):
    t = a * 134217729.0
    hi = t - (t - a)
    return hi, a - hi


def _sum_rows(ptr, v):
    return torch.segment_reduce(v, "sum", lengths=ptr[1:] - ptr[:-1], unsafe=True)


def _multiply(m, x):
    """A x: every product as a rounded product and its error (Dekker), the
    rounded products cut to multiples of 2^-30, whose sums carry no rounding,
    and the rests added after them."""
    n, ptr, col, val = m
    xv = x[col.long()]
    p = val * xv
    (ah, al), (bh, bl) = _halves(val), _halves(xv)
    rest = ((ah * bh - p) + ah * bl + al * bh) + al * bl
    big = 1.5 * 2.0 ** 22
    cut = (p + big) - big
    return _sum_rows(ptr, cut) + (_sum_rows(ptr, p - cut) + _sum_rows(ptr, rest))


def _splitmix(seed, t):
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (t + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def exact(case, seed):
    path = case["path"]
    if path == "burst":
        return None   # hashes
    gen = _generator(seed)
    if path == "batch":
        mats = [_matrix(kind, size, gen) for kind, size in _mix(case)]
        x = _uniform(sum(m[0] for m in mats), gen)
        at = np.concatenate([[0], np.cumsum([m[0] for m in mats])])
        return torch.cat([_multiply(m, x[at[i]:at[i + 1]]) for i, m in enumerate(mats)])
    m = _matrix(case["matrix"], case["g"] if "g" in case else case["n"], gen)
    n = m[0]
    if path == "single":
        t = np.arange(n, dtype=np.uint64)[:, None] * np.uint64(8) + np.arange(case["width"], dtype=np.uint64)[None, :]
        x = (_splitmix(seed * 7919 + 1, t) >> np.uint64(11)).astype(np.float64) * 2.0 ** -52 - 1.0
        x = torch.from_numpy(x).cuda()
        return {"x": x, "y": torch.stack([_multiply(m, x[:, j].contiguous()) for j in range(case["width"])], dim=1)}
    if path == "host":
        x = _uniform((case["products"], n), gen)
        return torch.stack([_multiply(m, x[k]) for k in range(case["products"])])
    return _multiply(m, _uniform(n, gen))
