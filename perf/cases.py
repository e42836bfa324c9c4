"""Performance cases of the library: what a program that uses it has it compute.

Every case goes through the public entry points of the package.  Vectors are
FP64 on the GPU with values U(-1, 1), coefficients U(-1, 1) or U(-2, 2), as in
the repository's tests and benchmark.  `shift` is the start offset of the
vectors, in elements past an aligned allocation: a sub-vector of a larger one.
No search runs first: the calls take the library's built-in choices.
"""
import math

import torch

import paper_1309_1894_gb300 as wx
from paper_1309_1894_gb300.binding import wxpy_batch_noalloc


def listed():
    return [
        # the smallest call: a short sub-vector, one launch, nothing but latency
        {"name": "wxpy_small", "kind": "wxpy", "n": 1027, "shift": 1, "mixed": False,
         "alias": "none", "calls": 1, "graph": False},
        # the plain call on 2^20 elements: sixteen separate sets one after another, replayed
        # from a CUDA graph so that the calls follow each other closely
        {"name": "wxpy_1m", "kind": "wxpy", "n": 1 << 20, "shift": 0, "mixed": False,
         "alias": "none", "calls": 16, "graph": True},
        # the largest call of the size sweep: ragged, 8 bytes off, in place
        {"name": "wxpy_large", "kind": "wxpy", "n": (1 << 28) + 3, "shift": 1, "mixed": False,
         "alias": "wx", "calls": 1, "graph": False},
        # 4096 uneven problems, aligned starts, one planned launch replayed from its graph
        {"name": "batch_graph", "kind": "batch", "entry": "graph", "segments": 4096,
         "n_max": 1 << 20, "packed": False},
        # a ragged batch stored back to back (starts at any element), planned on the device
        {"name": "batch_packed", "kind": "batch", "entry": "noalloc", "segments": 1024,
         "n_max": 1 << 16, "packed": True},
        # a three-vector update (two-step methods), ragged and 8 bytes off
        {"name": "axpbypcz", "kind": "axpbypcz", "n": (1 << 25) + 3, "shift": 1, "mixed": False},
        # eight basis vectors of separate allocations added to one (a restart cycle)
        {"name": "maxpy_8", "kind": "maxpy", "m": 8, "n": 1 << 24, "rows": False},
        # five rows of one basis matrix with an odd row length: every row starts elsewhere
        {"name": "maxpy_rows", "kind": "maxpy", "m": 5, "n": 1000003, "rows": True},
        # the residual update with its norm, large
        {"name": "norm2_large", "kind": "norm2", "n": (1 << 26) + 3, "shift": 0, "mixed": False},
        # an update with its inner product, an ordinary problem size
        {"name": "dot_mid", "kind": "dot", "n": 1000003, "shift": 0, "mixed": False},
        # the vector work of a stabilised bi-conjugate gradient solver, captured once in a
        # CUDA graph and replayed: many dependent calls on mid-size vectors
        {"name": "solver", "kind": "solver", "n": 131075, "iterations": 8},
        # the server: a burst of requests of mixed sizes on the caller's device data
        {"name": "served", "kind": "served", "requests": 48, "n_min": 1 << 8, "n_max": 1 << 20},
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["wxpy", "wxpy", "batch", "axpby", "axpbypcz", "maxpy", "maxpy", "pmult",
                       "norm2", "dot", "solver", "served"])
    c = {"kind": kind}
    if kind == "wxpy":
        c.update(n=_log_uniform(rng, 1 << 10, 1 << 28), shift=rng.randrange(4),
                 mixed=rng.random() < 0.3, alias=rng.choice(["none", "none", "wx", "wy", "xy"]))
        c["calls"] = 1 if c["n"] > 1 << 22 else rng.choice([1, 4, 16])
        c["graph"] = c["calls"] > 1 and rng.random() < 0.5
    elif kind == "batch":
        c.update(entry=rng.choice(["graph", "launch", "once", "noalloc"]),
                 segments=_log_uniform(rng, 64, 4096), n_max=_log_uniform(rng, 1 << 12, 1 << 20),
                 packed=rng.random() < 0.5)
    elif kind == "maxpy":
        c["m"] = rng.choice([2, 3, 4, 5, 6, 8, 10, 12, 16, 20])
        c.update(n=_log_uniform(rng, 1 << 12, (1 << 29) // (c["m"] + 2)), rows=rng.random() < 0.5)
    elif kind == "solver":
        c.update(n=_log_uniform(rng, 1 << 13, 1 << 22), iterations=rng.choice([2, 4, 8]))
    elif kind == "served":
        c.update(requests=rng.randrange(8, 49), n_min=1 << 8, n_max=_log_uniform(rng, 1 << 14, 1 << 21))
    else:
        c.update(n=_log_uniform(rng, 1 << 12, 1 << 27), shift=rng.choice([0, 0, 1, 2, 3]),
                 mixed=rng.random() < 0.25)
    return c


# ---- inputs -------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, n, scale=1.0):
    return (torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * 2 - 1) * scale


def _coefs(seed, count, scale=1.0):
    g = torch.Generator()
    g.manual_seed(seed + 77)
    return ((torch.rand(count, dtype=torch.float64, generator=g) * 2 - 1) * scale).tolist()


def _vector(g, n, shift):
    """n values starting `shift` elements past an aligned allocation."""
    t = torch.empty(n + shift, dtype=torch.float64, device="cuda")[shift:]
    t.copy_(_uniform(g, n))
    return t


def _shifts(case, count):
    """The vectors' offsets: one for all, or (mixed) each its own."""
    s = case.get("shift", 0)
    return [(s + k) % 4 if case.get("mixed") else s for k in range(count)]


def _batch_lengths(case):
    """Lengths log-uniform on [1, n_max] and start elements: the case's own, for
    every seed the same, so that its outputs keep one layout."""
    g = torch.Generator()
    g.manual_seed(20130907)
    u = torch.rand(case["segments"], dtype=torch.float64, generator=g)
    ns = torch.exp(u * math.log(case["n_max"] + 1)).long().clamp(1, case["n_max"])
    room = ns if case["packed"] else (ns + 31) // 32 * 32  # 256-byte aligned starts
    starts = torch.cumsum(room, 0) - room
    return ns.tolist(), starts.tolist(), int(room.sum())


def _request_lengths(case):
    g = torch.Generator()
    g.manual_seed(20130909)
    u = torch.rand(case["requests"], dtype=torch.float64, generator=g)
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"] + 1)
    return torch.exp(lo + u * (hi - lo)).long().clamp(case["n_min"], case["n_max"]).tolist()


def _inputs(case, seed):
    """The case's vectors and coefficients, from the seed alone."""
    g = _gen(seed)
    kind, s = case["kind"], {"case": case}
    if kind == "wxpy":
        s["alpha"] = _coefs(seed, 1, 1.0 if case["alias"] == "wx" else 2.0)[0]
        sh = _shifts(case, 3)
        s["sets"] = []
        for _ in range(case["calls"]):
            x = _vector(g, case["n"], sh[0])
            y = x if case["alias"] == "xy" else _vector(g, case["n"], sh[1])
            s["sets"].append((x, y))
    elif kind == "batch":
        s["ns"], s["starts"], total = _batch_lengths(case)
        s["alphas"] = _coefs(seed, case["segments"], 2.0)
        s["x"], s["y"] = _uniform(g, total), _uniform(g, total)
    elif kind == "maxpy":
        m, n = case["m"], case["n"]
        s["alphas"] = _coefs(seed, m)
        if case["rows"]:
            basis = _uniform(g, m * n).view(m, n)
            s["xs"] = [basis[j] for j in range(m)]
        else:
            s["xs"] = [_uniform(g, n) for _ in range(m)]
        s["y"] = _uniform(g, n)
    elif kind == "solver":
        s["vecs"] = {k: _uniform(g, case["n"]) for k in ("r", "p", "v", "s", "t", "x", "rh")}
        s["coefs"] = _coefs(seed, 3, 0.5)
    elif kind == "served":
        ns = _request_lengths(case)
        s["alphas"] = _coefs(seed, case["requests"], 2.0)
        s["xy"] = [(_uniform(g, n), _uniform(g, n)) for n in ns]
    else:
        s["coefs"] = _coefs(seed, 3, 0.5)
        s["vecs"] = [_vector(g, case["n"], sh) for sh in _shifts(case, 4)[: 4 if kind == "dot" else 3]]
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "wxpy":
        sw = _shifts(case, 3)[2]
        s["ws"] = []
        for x, y in s["sets"]:
            s["ws"].append(x if case["alias"] == "wx" else y if case["alias"] == "wy" else
                           torch.empty(case["n"] + sw, dtype=torch.float64, device="cuda")[sw:])
        if case["graph"]:
            x, y = s["sets"][0]
            wx.wxpy(s["alpha"], x, y, torch.empty_like(s["ws"][0]))  # once before the capture
            torch.cuda.synchronize()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"]):
                _wxpy_calls(s)
    elif kind == "batch":
        s["w"] = torch.zeros_like(s["x"])
        ptr = [[t.data_ptr() + 8 * b for b in s["starts"]] for t in (s["x"], s["y"], s["w"])]
        s["table"] = wx.desc_table(s["ns"], s["alphas"], *ptr)
        s["dev"] = wx.table_to_device(s["table"])
        if case["entry"] in ("graph", "launch"):
            s["plan"] = wx.wxpy_batch_plan_create(s["table"])
    elif kind in ("norm2", "dot"):
        s["result"] = torch.empty(1, dtype=torch.float64, device="cuda")
        s["workspace"] = wx.reduce_workspace(case["n"])
    elif kind == "solver":
        s["dots"] = torch.empty(2, dtype=torch.float64, device="cuda")
        s["workspace"] = wx.reduce_workspace(case["n"])
        kept = {k: t.clone() for k, t in s["vecs"].items()}
        _solver_iterations(s)  # once before the capture, as CUDA graphs want it
        for k, t in kept.items():
            s["vecs"][k].copy_(t)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _solver_iterations(s)
    elif kind == "served":
        room = sum(3 * (8 * x.numel() + 256) for x, _ in s["xy"])
        s["server"] = wx.Server(budget_bytes=2 * room + (1 << 20), max_slots=256, n_streams=2,
                                max_batch=64, max_queue=1024)
        s["tickets"] = []
    return s


def _wxpy_calls(s):
    for (x, y), w in zip(s["sets"], s["ws"]):
        wx.wxpy(s["alpha"], x, y, w)


def _solver_iterations(s):
    """The vector operations of a BiCGStab iteration with given scalars (the
    matrix products, which are not this library's, left out)."""
    d, ws = s["vecs"], s["workspace"]
    alpha, beta, omega = s["coefs"]
    n2, dot = s["dots"][0:1], s["dots"][1:2]
    for _ in range(s["case"]["iterations"]):
        wx.wxpy_axpbypcz(1.0, -omega * beta, beta, d["r"], d["v"], d["p"])    # p = r - wb v + b p
        wx.wxpy(-alpha, d["v"], d["r"], d["s"])                               # s = r - a v
        wx.wxpy_axpbypcz(alpha, omega, 0.75, d["p"], d["s"], d["x"])          # x = a p + w s + .75 x
        wx.wxpy_norm2(-omega, d["t"], d["s"], d["r"], n2, ws)                 # r = s - w t, r.r
        wx.wxpy_dot(beta, d["v"], d["r"], d["rh"], d["t"], dot, ws)           # t = b v + r, t.rh


# ---- one pass -----------------------------------------------------------------------

class _Resident:
    """A served result, resident in the server's memory until it is released."""

    def __init__(self, server, n, ptr):
        self.server = server
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<f8", "data": (ptr, False),
                                         "strides": None, "version": 2}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "wxpy":
        if case["graph"]:
            s["graph"].replay()
        else:
            _wxpy_calls(s)
        return s["ws"]
    if kind == "batch":
        if case["entry"] == "graph":
            s["plan"].graph_launch(s["dev"])
        elif case["entry"] == "launch":
            s["plan"].launch(s["dev"])
        elif case["entry"] == "once":
            wx.wxpy_batch(s["table"], s["dev"])
        else:
            wxpy_batch_noalloc(s["dev"], case["segments"])
        return s["w"]
    if kind == "maxpy":
        return wx.wxpy_maxpy(s["alphas"], s["xs"], s["y"])
    if kind == "solver":
        s["graph"].replay()
        return {**s["vecs"], "dots": s["dots"]}
    if kind == "served":
        server = s["server"]
        for t in s["tickets"]:
            server.release(t)
        s["tickets"] = [server.submit_data(a, x, y) for a, (x, y) in zip(s["alphas"], s["xy"])]
        for t in s["tickets"]:
            server.wait(t)
        out = []
        for t in s["tickets"]:
            n, _, _, w = server.result(t)
            out.append(torch.as_tensor(_Resident(server, n, w), device="cuda"))
        return out
    a, b, c = s["coefs"]
    v = s["vecs"]
    if kind == "axpby":
        return wx.wxpy_axpby(a, b, v[0], v[1])
    if kind == "axpbypcz":
        return wx.wxpy_axpbypcz(a, b, c, v[0], v[1], v[2])
    if kind == "pmult":
        return wx.wxpy_pointwise_mult(v[0], v[1], v[2])
    if kind == "norm2":
        return wx.wxpy_norm2(a, v[0], v[1], v[2], s["result"], s["workspace"])
    return wx.wxpy_dot(a, v[0], v[1], v[3], v[2], s["result"], s["workspace"])


# ---- what a pass cannot do without, and its outputs in plain torch -------------------

def work(case):
    kind = case["kind"]
    if kind == "wxpy":
        e = case["n"] * case["calls"]
        return {"bytes": (16 if case["alias"] == "xy" else 24) * e, "flops": 2 * e}
    if kind in ("batch", "served"):  # the mean of the log-uniform lengths
        lo, hi = case.get("n_min", 1), case["n_max"]
        e = case.get("segments", case.get("requests")) * (hi + 1 - lo) / math.log((hi + 1) / lo)
        # a served request's data are the caller's: read x, y and write w all the same
        return {"bytes": 24 * e, "flops": 2 * e}
    n = case["n"]
    if kind == "maxpy":
        return {"bytes": 8 * (case["m"] + 2) * n, "flops": 2 * case["m"] * n}
    if kind == "solver":  # two axpbypcz, one wxpy, one norm2, one dot
        return {"bytes": (32 + 24 + 32 + 24 + 32) * n * case["iterations"],
                "flops": (5 + 2 + 5 + 4 + 4) * n * case["iterations"]}
    b, f = {"axpby": (24, 3), "axpbypcz": (32, 5), "pmult": (24, 1), "norm2": (24, 4),
            "dot": (32, 4)}[kind]
    return {"bytes": b * n, "flops": f * n}


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "wxpy":
        return [s["alpha"] * x + y for x, y in s["sets"]]
    if kind == "batch":
        w = torch.zeros_like(s["x"])
        for n, b, a in zip(s["ns"], s["starts"], s["alphas"]):
            w[b:b + n] = a * s["x"][b:b + n] + s["y"][b:b + n]
        return w
    if kind == "maxpy":
        y = s["y"]
        for a, x in zip(s["alphas"], s["xs"]):
            y = y + a * x
        return y
    if kind == "served":
        return [a * x + y for a, (x, y) in zip(s["alphas"], s["xy"])]
    if kind == "solver":
        d = s["vecs"]
        alpha, beta, omega = s["coefs"]
        n2 = dot = None
        for _ in range(case["iterations"]):
            d["p"] = d["r"] + (-omega * beta) * d["v"] + beta * d["p"]
            d["s"] = -alpha * d["v"] + d["r"]
            d["x"] = alpha * d["p"] + omega * d["s"] + 0.75 * d["x"]
            d["r"] = -omega * d["t"] + d["s"]
            n2 = (d["r"] * d["r"]).sum()
            d["t"] = beta * d["v"] + d["r"]
            dot = (d["t"] * d["rh"]).sum()
        return {**d, "dots": torch.stack([n2, dot])}
    a, b, c = s["coefs"]
    v = s["vecs"]
    if kind == "axpby":
        return a * v[0] + b * v[1]
    if kind == "axpbypcz":
        return a * v[0] + b * v[1] + c * v[2]
    if kind == "pmult":
        return v[0] * v[1]
    w = a * v[0] + v[1]
    return w, (w * (w if kind == "norm2" else v[3])).sum().reshape(1)
