"""The framework's work as a user's program has it do, case by case: searches
from one query to ten thousand over uint8 and fp32 rows (short and long),
through each search entry point and option, the encoder on its own, an index
build and a calibration.

The indexes are the repository's own workload shapes: u8-10m, f32-10m, u8-30m
(the 1e9 workload's rows per code on 3e7 rows) and f32-1536-1m, drawn from
Gaussian mixtures of their sizes. A program keeps its index and asks it many
batches, so an index is built once a process (from logits that torch gives)
and every seed draws other queries from its mixture.
"""
import math

import numpy as np
import torch

from paper_2608_15438_gb300 import calibrate
from paper_2608_15438_gb300 import neuroute as nr
from paper_2608_15438_gb300.builder import config

DEV = "cuda:0"

# rows, dimension, type, mixture components, spread, hidden width, hidden
# widths after it, code bits, clusters a bucket, rows a cluster
SHAPES = {
    "u8-10m": (10_000_000, 128, "u8", 256, 18.0, 512, (), 20, 8, 64),
    "u8-30m": (30_000_000, 128, "u8", 512, 18.0, 512, (), 19, 16, 64),
    "f32-10m": (10_000_000, 96, "f32", 1024, 0.3, 384, (), 20, 8, 64),
    "f32-1536-1m": (1_000_000, 1536, "f32", 1024, 0.3, 512, (256, 128, 64), 16, 16, 64),
}

_KEPT = {}  # shape -> (index, centres): one a process, as a serving program holds it


def _search(name, shape, entry, nq, k, P, C, t_low, gate=-1.0, seq=0, nonempty=0):
    """gate: slope of the centroid gate M(x) = gate x (negative: off)."""
    return {"name": name, "do": "search", "shape": shape, "entry": entry, "nq": nq, "k": k, "P": P,
            "C": C, "t_low": t_low, "gate": gate, "seq": seq, "nonempty": nonempty}


def listed():
    return [
        # an interactive request: one query, the u8-10m configuration's own
        # budgets (P 64, C 128) and the default early stop
        _search("one u8 query", "u8-10m", "search", 1, 10, 64, 128, 4),
        # one request at the budgets of the 1e9 operating point
        _search("one u8 query, deep", "u8-30m", "search", 1, 10, 1024, 1024, 80, 4.0),
        # a small batch of a server that may not allocate (nr_search_static)
        _search("37 u8 queries, static", "u8-10m", "static", 37, 10, 256, 256, 0, 4.0),
        # a small fp32 batch with a long result list, budgets of the f32-10m point
        _search("16 f32 queries, top 100", "f32-10m", "search", 16, 100, 512, 256, 16),
        # embeddings of 1536 values through the four-hidden-layer encoder
        _search("4 long f32 queries", "f32-1536-1m", "search", 4, 10, 1024, 2048, 256),
        # an ordinary batch at the u8-10m operating point
        _search("1000 u8 queries", "u8-10m", "search", 1000, 10, 256, 256, 0, 4.0),
        # Algorithm 2's sequential centroid stage, logits given by the caller
        _search("333 u8 queries, sequential", "u8-30m", "logits", 333, 10, 1024, 384, 64, 4.0, seq=1),
        # the benchmark's batch, end to end from pinned host memory
        _search("10000 u8 queries, host", "u8-30m", "host", 10_000, 10, 1024, 1024, 80, 4.0),
        # the fp32 workload's batch at its operating point
        _search("10000 f32 queries", "f32-10m", "search", 10_000, 10, 512, 256, 16),
        # the encoder alone over a chunk of base rows (an index build's first pass)
        {"name": "encode 1000037 u8 rows", "do": "encode", "shape": "u8-30m", "nq": 1_000_037},
        # a whole index build of an ordinary collection
        {"name": "build 2000003 u8 rows", "do": "build", "dtype": "u8", "N": 2_000_003, "b": 16,
         "K_max": 16, "t": 64},
        # the gate and score cutoff fitted on held-out queries, after a build
        {"name": "calibrate 2000 queries", "do": "calibrate", "shape": "u8-30m", "nq": 2000, "k": 10,
         "P": 512, "C": 2048},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choice(["u8", "u8", "u8", "u8", "f32", "f32", "long", "encode", "build", "calibrate"])
    if what == "encode":
        shape = rng.choice(["u8-30m", "f32-10m", "f32-1536-1m"])
        return {"do": "encode", "shape": shape,
                "nq": _log_int(rng, 1, 100_000 if shape == "f32-1536-1m" else 1_000_000)}
    if what == "build":
        N = _log_int(rng, 20_000, 2_000_000)
        return {"do": "build", "dtype": rng.choice(["u8", "f32"]), "N": N,
                "b": max(8, int(math.log2(N)) - rng.randint(4, 6)), "K_max": rng.choice([4, 8, 16]),
                "t": rng.choice([32, 64])}
    if what == "calibrate":
        return {"do": "calibrate", "shape": rng.choice(["u8-10m", "u8-30m", "f32-10m"]),
                "nq": _log_int(rng, 100, 2000), "k": rng.choice([1, 10, 20]),
                "P": _log_int(rng, 64, 512), "C": _log_int(rng, 128, 2048)}
    k = rng.choice([1, 5, 10, 10, 10, 20, 50, 100])
    if what == "long":
        c = _search("", "f32-1536-1m", rng.choice(["search", "logits"]), _log_int(rng, 1, 60), k,
                    _log_int(rng, 8, 1024), _log_int(rng, 64, 2048), rng.choice([0, 16, 64, 256]))
    else:
        shape = "f32-10m" if what == "f32" else rng.choice(["u8-10m", "u8-30m"])
        c = _search("", shape, rng.choice(["search", "search", "logits", "static", "host"]),
                    _log_int(rng, 1, 9000), k, _log_int(rng, 4, 1024), _log_int(rng, 32, 1024),
                    rng.choice([0, 4, 16, 64, 80]), rng.choice([-1.0, 4.0]),
                    1 if rng.random() < 0.1 else 0, 1 if rng.random() < 0.1 else 0)
        if c["entry"] == "static":  # its batches fit the fixed 32 MiB
            S = 1
            while S < c["P"] * SHAPES[shape][8]:
                S *= 2
            per = 4 * SHAPES[shape][7] + 4 * c["P"] + 12 * (c["P"] + c["C"]) + 56
            per += 12 * S + 8 if S > 2048 else 0
            c["nq"] = min(c["nq"], (30 << 20) // per)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _centres(dtype, M, D):
    g = _generator(101)
    if dtype == "u8":
        return torch.rand((M, D), generator=g, device=DEV) * 215.0 + 20.0
    return torch.randn((M, D), generator=g, device=DEV)


def _rows(dtype, centres, sigma, n, g):
    """n rows of the mixture: uint8 rounded and clipped, fp32 on the unit sphere."""
    which = torch.randint(0, centres.shape[0], (n,), generator=g, device=DEV)
    x = torch.randn((n, centres.shape[1]), generator=g, device=DEV).mul_(sigma).add_(centres[which])
    if dtype == "u8":
        return x.round_().clamp_(0, 255).to(torch.uint8)
    return torch.nn.functional.normalize(x, dim=1)


def _weights(D, H, mid, b):
    """A random encoder D -> H -> mid ... -> b, weights N(0, 1 / fan_in), zero biases."""
    rng = np.random.default_rng(7)

    def layer(o, i):
        return rng.standard_normal((o, i), dtype=np.float32) / np.float32(math.sqrt(i))

    W1 = layer(H, D)
    widths = (H,) + tuple(mid)
    mids = tuple((layer(o, i), np.zeros(o, np.float32)) for i, o in zip(widths[:-1], widths[1:]))
    W2 = layer(b, widths[-1])
    out = (W1, np.zeros(H, np.float32), W2, np.zeros(b, np.float32))
    return out + (mids,) if mids else out


def _mlp(x, dtype, weights, kind):
    """The encoder's forward in torch, in `kind` precision."""
    h = x.to(kind) * (1.0 / 255.0 if dtype == "u8" else 1.0)
    mids = weights[4] if len(weights) > 4 else ()
    for W, bias in ((weights[0], weights[1]),) + tuple(mids):
        W, bias = (torch.from_numpy(a).to(DEV, kind) for a in (W, bias))
        h = torch.relu(h @ W.T + bias)
    W, bias = (torch.from_numpy(a).to(DEV, kind) for a in weights[2:4])
    return h @ W.T + bias


def _index(shape):
    if shape not in _KEPT:
        N, D, dtype, M, sigma, H, mid, b, k_max, t = SHAPES[shape]
        centres = _centres(dtype, M, D)
        weights = _weights(D, H, mid, b)
        bd = nr.Builder(config(dtype, D, H, b, k_max, t, mid=mid), N, weights)
        step = min(N, (1 << 31) // (4 * D))
        parts = [(i, min(step, N - i)) for i in range(0, N, step)]
        for i, n in parts:
            bd.set_logits(_mlp(_rows(dtype, centres, sigma, n, _generator(1000 + i)), dtype, weights,
                               torch.float32), i)
            torch.cuda.synchronize()
        bd.finish()
        for i, n in parts:
            bd.place(_rows(dtype, centres, sigma, n, _generator(1000 + i)), i)
            torch.cuda.synchronize()
        _KEPT[shape] = (bd.end(), centres, weights)
        torch.cuda.empty_cache()
    return _KEPT[shape]


def prepare(case, seed):
    g = _generator(seed)
    if case["do"] == "build":
        dtype = case["dtype"]
        D, H, sigma = (128, 512, 18.0) if dtype == "u8" else (96, 384, 0.3)
        rows = _rows(dtype, _centres(dtype, 256, D), sigma, case["N"], g)
        return {"case": case, "rows": rows, "weights": _weights(D, H, (), case["b"]),
                "cfg": config(dtype, D, H, case["b"], case["K_max"], case["t"]),
                "ids": torch.arange(case["N"], device=DEV)}
    N, D, dtype, M, sigma, H, mid, b, k_max, t = SHAPES[case["shape"]]
    ix, centres, weights = _index(case["shape"])
    q = _rows(dtype, centres, sigma, case["nq"], g)
    s = {"case": case, "ix": ix, "q": q}
    if case["do"] == "search":
        nq, k = case["nq"], case["k"]
        kw = {"t_low": case["t_low"], "nonempty_budget": case["nonempty"]}
        if case["gate"] >= 0:
            kw.update(gate_m0=0.0, gate_m1=case["gate"])
        if case["seq"]:
            kw.update(cent_mode=1, c_t_low=4)
        s["params"] = nr.params(**kw)
        # result buffers that a program keeps from call to call
        s["out"] = (torch.empty((nq, k), dtype=torch.int64, device=DEV),
                    torch.empty((nq, k), dtype=torch.float32, device=DEV))
        if case["entry"] == "logits":
            s["logits"] = _mlp(q, dtype, weights, torch.float32)
        if case["entry"] == "host":
            s["q"] = q.cpu().pin_memory()
            s["out"] = tuple(o.cpu().pin_memory() for o in s["out"])
    return s


# ---------------------------------------------------------------- one pass


def run(state):
    case = state["case"]
    if case["do"] == "build":
        bd = nr.Builder(state["cfg"], case["N"], state["weights"])
        bd.encode(state["rows"], 0)
        info = bd.finish()
        bd.place(state["rows"], 0)
        ix = bd.end()
        loc = ix.locate(state["ids"])  # where every row was stored
        tau = ix.thresholds()
        ix.close()
        return {"buckets": info["n_buckets"], "tau": tau, "code": loc[:, 1],
                "cluster": loc[:, 0] - loc[:, 2], "clusters": loc[:, 3]}
    ix = state["ix"]
    if case["do"] == "encode":
        return ix.encode(state["q"])
    if case["do"] == "calibrate":
        c = calibrate.calibrate(ix, state["q"], k=case["k"], P=case["P"], C=case["C"])
        return {"scores": c["scores"], "x": c["x"], "y": c["y"],
                "s_max": float(c["s_max"]) if c["s_max"] is not None else 0.0,
                "curve": [list(v) for v in c["gate_curve"]] if c["gate_curve"] else []}
    ix.set_params(state["params"])
    args = (case["k"], case["P"], case["C"])
    if case["entry"] == "search":
        return ix.search(state["q"], *args, out=state["out"])
    if case["entry"] == "logits":
        return ix.search_logits(state["q"], state["logits"], *args, out=state["out"])
    if case["entry"] == "static":
        return ix.search_static(state["q"], *args, out=state["out"])
    return ix.search_host(state["q"], *args, out=state["out"])


# ---------------------------------------------------------------- what it takes


def _encoder_flops(D, H, mid, b, n):
    widths = (D, H) + tuple(mid) + (b,)
    return 2.0 * n * sum(i * o for i, o in zip(widths[:-1], widths[1:]))


def work(case):
    """Search: the candidate rows the method gives a distance (the statistics
    of one pass; no row more than once), the centroids scored, queries and
    results; three operations a coordinate. Build: rows in and stored, ids,
    logits out and in; the encoder and five passes of k-means."""
    if case["do"] == "build":
        N, b = case["N"], case["b"]
        D, H, esz = (128, 512, 1) if case["dtype"] == "u8" else (96, 384, 4)
        K = min(case["K_max"], max(1.0, N / 2.0 ** b / case["t"]))
        return {"bytes": N * (2.0 * D * esz + 2 * 4 * b + 8 + 16),
                "flops": _encoder_flops(D, H, (), b, N) + 5.0 * 3 * N * K * b}
    N, D, dtype, M, sigma, H, mid, b, k_max, t = SHAPES[case["shape"]]
    rb, nq = D * (1 if dtype == "u8" else 4), case["nq"]
    enc = _encoder_flops(D, H, mid, b, nq)
    if case["do"] == "encode":
        weights = D * H + sum(a * c for a, c in zip((H,) + mid, mid + (b,)))
        return {"bytes": float(nq * (rb + 4 * b) + 4 * weights), "flops": enc}
    run(prepare(case, 1))
    torch.cuda.synchronize()
    st = _index(case["shape"])[0].last_stats()
    n_cl = _index(case["shape"])[0].n_clusters
    bytes_ = (min(st.candidates, N) * rb + min(st.scored, n_cl) * 4 * b + nq * (rb + 12 * case["k"]))
    if case["do"] == "calibrate":
        bytes_ += 4 * N  # the stored ids that the targets are looked for in
    return {"bytes": float(bytes_), "flops": 3.0 * (st.candidates * D + st.scored * b) + enc}


def tolerance(case):
    """Every step after the encoder has one fixed order of fp32 operations or
    is in whole numbers: exact where the logits are given. The encoder's sums
    are fp32 over fp16 operands: against the same operands summed in another
    order, its logits differ by up to 6e-5 of their norm (2.3e-4 with four
    hidden layers: hidden values on an fp16 rounding boundary go either way)
    and 7e-4 at most, and no result of the listed searches changes."""
    if case["do"] == "encode":
        deep = bool(SHAPES[case["shape"]][6])
        return {"rel": 1e-3 if deep else 2.5e-4, "max": 3e-3}
    if case["do"] == "search" and case["entry"] == "logits":
        return "exact"
    if case["do"] == "search":  # a result at the edge of two probes or of a gate
        return {"rel": 1e-4, "max": 0.05, "differ": 1e-3}
    # a row or target on a threshold; y is a difference of two distances
    return {"rel": 1e-3, "max": 0.05, "differ": 5e-3}


def exact(case, seed):
    """The encoder in 64 bits. A search's, build's or calibration's answer
    follows from the index's k-means, which has no statement outside the
    repository."""
    if case["do"] != "encode":
        return None
    dtype = SHAPES[case["shape"]][2]
    q = prepare(case, seed)["q"]
    weights = _index(case["shape"])[2]
    return torch.cat([_mlp(x, dtype, weights, torch.float64) for x in q.split(1 << 17)])
