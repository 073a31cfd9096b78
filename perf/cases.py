"""Timed cases of the Parallel-l0 framework: the work its users have it do.

A user draws a left d-regular expander A (``make_expander``), measures a
k-sparse signal (``measure``), and recovers it from y (``decode_parallel_l0``
and its asynchronous form); sweeps and services do so for many problems of
uneven sizes (``ccs_decode_batch_async``, ``Server``).  The sizes are the
workloads of ``paper_1508_01256_gb300/inputs.py``, of bench.py and of the
recovery protocols in ``paper_1508_01256_gb300/phase.py``.

Kinds of case:

- ``decode``    one problem, A and y on the device; ``call`` says whether the
                host waits for the result (``blocking``) or enqueues decode
                after decode (``async``)
- ``scaled``    a +-1 signal through the column-scaled matrix: measure with
                scales, decode, unscale (Sec. 4.3.3)
- ``expander``  drawing A and its transpose
- ``measure``   y = A x for a matrix the caller brought
- ``batch``     many problems of mixed sizes in one call
- ``serve``     seeded requests through the continuous-batching server

Signals follow the package's value models: ``gauss-grid`` (N(0,1) on a 2^-32
grid, where binary64 sums are exact), ``gauss-raw`` (literal N(0,1), where
the decoder keeps the residual by ordered sums) and +-1.
"""
import math

import numpy as np
import torch

from paper_1508_01256_gb300 import ccs, inputs

GRID = 2.0 ** -32


def _decode(name, n, m, d, k, values="gauss-grid", score="l0", alpha=2, shifted=False,
            call="async"):
    return {"name": name, "kind": "decode", "n": n, "m": m, "d": d, "k": k, "values": values,
            "score": score, "alpha": alpha, "shifted": shifted, "call": call}


def listed():
    return [
        # the smallest instance of the benchmark suite, decoded on demand: the
        # caller waits for each result, so launches and latency are what counts
        _decode("decode_small", 4096, 410, 7, 41, call="blocking"),
        # integer-valued signals (not dissociated) at an odd size: measured with
        # the column-scaled matrix, decoded, unscaled
        {"name": "scaled_pm1", "kind": "scaled", "n": 200003, "m": 20011, "d": 9, "k": 2001},
        # the at-scale benchmark (n = 2^20, m/n = 1/8, rho = 0.2), decode after
        # decode: A stays in L2
        _decode("decode_at_scale", 2 ** 20, 2 ** 17, 7, 26214),
        # the same with literal Gaussian values, as measured data has them: the
        # residual is kept by ordered sums
        _decode("decode_at_scale_raw", 2 ** 20, 2 ** 17, 7, 26214, values="gauss-raw"),
        # extreme undersampling (n/m ~ 10^3, rho = 0.05), the headline benchmark:
        # A streams from HBM
        _decode("decode_extreme", 2 ** 24, 16777, 9, 839),
        # the same beyond its phase transition (rho = 0.15): a sweep pays for the
        # decodes that do not converge too, and they are most of its time
        _decode("decode_extreme_dense", 2 ** 24, 16777, 9, 2517),
        # the largest size of the paper's table of timings (delta = 10^-3, d = 7)
        _decode("decode_table3_large", 2 ** 26, 67109, 7, 3355),
        # drawing A at scale (rows of ~56 columns) and at extreme undersampling
        # (rows of ~9000 columns): every problem of a sweep begins with it
        {"name": "expander_at_scale", "kind": "expander", "n": 2 ** 20, "m": 2 ** 17, "d": 7},
        {"name": "expander_extreme", "kind": "expander", "n": 2 ** 24, "m": 16777, "d": 9},
        # measuring a sparse signal at extreme undersampling
        {"name": "measure_extreme", "kind": "measure", "n": 2 ** 24, "m": 16777, "d": 9,
         "k": 839},
        # a mixed batch as the recovery sweeps hand it over: n log-uniform over
        # 2^12 .. 2^20, four delta, three rho, four d; some never converge
        {"name": "batch_mixed", "kind": "batch", "count": 64, "shapes": 4242, "lo": 12.0,
         "hi": 20.0},
        # a burst of requests to the decode server: A drawn from each request's
        # seed, y from the host, x_hat's nonzeros back to the host
        {"name": "serve_burst", "kind": "serve", "count": 24, "shapes": 777, "lo": 12.0,
         "hi": 19.0},
    ]


def draw(rng):
    def log2size(lo, hi):
        return int(round(2.0 ** rng.uniform(lo, hi)))

    kind = rng.choice(["decode", "decode", "decode", "decode", "scaled", "expander", "expander",
                       "measure", "measure", "batch", "serve"])
    if kind in ("batch", "serve"):
        lo = rng.uniform(12.0, 16.0)
        return {"kind": kind, "count": rng.randint(2, 64 if kind == "batch" else 24),
                "shapes": rng.randrange(1 << 20), "lo": lo,
                "hi": rng.uniform(lo + 1.0, 20.0 if kind == "batch" else 19.0)}
    n = log2size(12.0, 24.0)
    deltas = [0.01, 0.02, 0.05, 0.1, 0.241, 0.5] if n < 2 ** 20 else [0.001, 0.01, 0.1, 0.125]
    d = rng.choice([5, 7, 7, 7, 9, 9, 11, 15])
    m = max(2 * d, inputs.round_half_up(rng.choice(deltas) * n))
    k = max(1, inputs.round_half_up(rng.choice([0.01, 0.05, 0.1, 0.2]) * m))
    if kind == "expander":
        return {"kind": kind, "n": n, "m": m, "d": d}
    if kind == "measure":
        return {"kind": kind, "n": n, "m": m, "d": d, "k": k}
    if kind == "scaled":
        return {"kind": kind, "n": n, "m": m, "d": d, "k": k}
    score, alpha = rng.choice([("l0", 2), ("l0", 2), ("l0", 3), ("count", ccs.lddsr_alpha(d))])
    c = _decode("", n, m, d, k, rng.choice(["gauss-grid", "gauss-grid", "gauss-raw"]), score,
                alpha, rng.random() < 0.15, rng.choice(["async", "blocking"]))
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------

def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + stream) % (2 ** 62))
    return g


def _signal(n, k, values, seed):
    """A k-sparse x on a uniform support, dense on the device."""
    at = torch.randperm(n, generator=_generator(seed, 1), device="cuda")[:k]
    g = _generator(seed, 2)
    if values == "pm1":
        v = torch.randint(0, 2, (k,), generator=g, device="cuda").double() * 2.0 - 1.0
    else:
        v = torch.randn(k, generator=g, device="cuda", dtype=torch.float64)
        if values == "gauss-grid":
            v = torch.round(v / GRID) * GRID
            v[v == 0.0] = GRID
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    x[at] = v
    return x


def _own_matrix(n, m, d, seed):
    """A matrix a caller brings: d distinct rows a column by torch, ascending
    (CSC), and its transpose (CSR), without the library."""
    g = _generator(seed, 3)
    rows = torch.randint(0, m, (n, d), generator=g, device="cuda", dtype=torch.int32)
    rows = rows.sort(dim=1).values
    while True:
        bad = (rows[:, 1:] == rows[:, :-1]).any(dim=1).nonzero().flatten()
        if bad.numel() == 0:
            break
        rows[bad] = torch.randint(0, m, (bad.numel(), d), generator=g, device="cuda",
                                  dtype=torch.int32).sort(dim=1).values
    by_row, at = torch.sort(rows.flatten(), stable=True)
    cols = (at // d).to(torch.int32)
    ptr = torch.searchsorted(by_row, torch.arange(m + 1, device="cuda", dtype=torch.int32))
    return rows, ptr.to(torch.int64), cols


def _problem_set(case, seed):
    """(n, m, d, k, problem seed) of a batch or a burst."""
    ds = inputs.BATCH_DS if case["kind"] == "batch" else (7, 9)
    shapes = inputs.batch_shapes(case["count"], case["shapes"], case["lo"], case["hi"], ds)
    return [(n, m, d, k, seed * 4099 + q) for q, (n, m, d, k) in enumerate(shapes)]


def prepare(case, seed):
    return {"decode": _prepare_decode, "scaled": _prepare_scaled, "expander": _prepare_expander,
            "measure": _prepare_measure, "batch": _prepare_batch,
            "serve": _prepare_serve}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


# ---- one decode ----------------------------------------------------------------

def _prepare_decode(case, seed):
    n, m, d = case["n"], case["m"], case["d"]
    csc, ptr, cols = ccs.make_expander(n, m, d, inputs.expander_seed(seed))
    x = _signal(n, case["k"], case["values"], seed)
    y = ccs.measure(ptr, cols, x, m, d)
    mode = ccs.SCORE_COUNT if case["score"] == "count" else ccs.SCORE_L0_DECREASE
    return {"run": _run_blocking if case["call"] == "blocking" else _run_async,
            "n": n, "m": m, "d": d, "csc": csc, "ptr": ptr, "cols": cols, "y": y,
            "alpha": case["alpha"], "mode": mode, "shifted": case["shifted"],
            "params": ccs.params(alpha=case["alpha"], score_mode=mode, shifted=case["shifted"]),
            "x_hat": torch.empty(n, dtype=torch.float64, device="cuda"),
            "r": torch.empty(m, dtype=torch.float64, device="cuda"),
            "result": ccs.result_buffer(1),
            "ws": ccs.workspace(ccs.ccs_workspace_size(ccs.OP_DECODE, n, m, d))}


def _run_blocking(s):
    o = ccs.decode_parallel_l0(s["csc"], s["ptr"], s["cols"], s["y"], alpha=s["alpha"],
                               score_mode=s["mode"], shifted=s["shifted"], ws=s["ws"],
                               out=(s["x_hat"], s["r"], None))
    return {"x_hat": o.x_hat, "r": o.r, "outcome": [o.status, o.iterations, o.r0_final]}


def _run_async(s):
    ccs.ccs_decode_parallel_l0_async(s["n"], s["m"], s["d"], s["csc"], s["ptr"], s["cols"],
                                     s["y"], s["x_hat"], s["r"], None, s["params"], s["result"],
                                     s["ws"])
    # the outcome: status, iterations and the two halves of ||r||_0; the fields
    # after it count how the decode went about it
    return {"x_hat": s["x_hat"], "r": s["r"], "outcome": s["result"].view(torch.int32)[:4]}


# ---- column-scaled measurement, decode, unscale -----------------------------------

def _prepare_scaled(case, seed):
    n, m, d = case["n"], case["m"], case["d"]
    csc, ptr, cols = ccs.make_expander(n, m, d, inputs.expander_seed(seed))
    return {"run": _run_scaled, "n": n, "m": m, "d": d, "csc": csc, "ptr": ptr, "cols": cols,
            "x": _signal(n, case["k"], "pm1", seed), "scales": ccs.column_scales(n, seed + 1),
            "z": torch.empty(n, dtype=torch.float64, device="cuda"),
            "r": torch.empty(m, dtype=torch.float64, device="cuda"),
            "params": ccs.params(), "result": ccs.result_buffer(1),
            "ws": ccs.workspace(ccs.ccs_workspace_size(ccs.OP_DECODE, n, m, d))}


def _run_scaled(s):
    y = ccs.measure_scaled(s["ptr"], s["cols"], s["scales"], s["x"], s["m"], s["d"])
    ccs.ccs_decode_parallel_l0_async(s["n"], s["m"], s["d"], s["csc"], s["ptr"], s["cols"], y,
                                     s["z"], s["r"], None, s["params"], s["result"], s["ws"])
    return {"y": y, "x": ccs.unscale(s["scales"], s["z"]), "r": s["r"]}


# ---- drawing A, measuring ---------------------------------------------------------

def _prepare_expander(case, seed):
    n, m, d = case["n"], case["m"], case["d"]
    return {"run": _run_expander, "n": n, "m": m, "d": d, "seed": inputs.expander_seed(seed),
            "csc": torch.empty((n, d), dtype=torch.int32, device="cuda"),
            "ptr": torch.empty(m + 1, dtype=torch.int64, device="cuda"),
            "cols": torch.empty(n * d, dtype=torch.int32, device="cuda"),
            "ws": ccs.workspace(ccs.ccs_workspace_size(ccs.OP_MAKE_EXPANDER, n, m, d))}


def _run_expander(s):
    ccs.ccs_make_expander(s["n"], s["m"], s["d"], s["seed"], s["csc"], s["ptr"], s["cols"],
                          s["ws"])
    return {"csc": s["csc"], "ptr": s["ptr"], "cols": s["cols"]}


def _prepare_measure(case, seed):
    n, m, d = case["n"], case["m"], case["d"]
    _, ptr, cols = _own_matrix(n, m, d, seed)
    return {"run": _run_measure, "m": m, "d": d, "ptr": ptr, "cols": cols,
            "x": _signal(n, case["k"], "gauss-grid", seed)}


def _run_measure(s):
    return ccs.measure(s["ptr"], s["cols"], s["x"], s["m"], s["d"])


# ---- many problems ------------------------------------------------------------------

def _prepare_batch(case, seed):
    shapes = _problem_set(case, seed)
    x_hat = torch.empty(sum(q[0] for q in shapes), dtype=torch.float64, device="cuda")
    r = torch.empty(sum(q[1] for q in shapes), dtype=torch.float64, device="cuda")
    keep, probs, at_n, at_m = [], [], 0, 0
    for n, m, d, k, sd in shapes:
        csc, ptr, cols = ccs.make_expander(n, m, d, inputs.expander_seed(sd))
        y = ccs.measure(ptr, cols, _signal(n, k, "gauss-grid", sd), m, d)
        keep.append((csc, ptr, cols, y))
        probs.append(ccs.problem(csc, ptr, cols, y, x_hat[at_n:at_n + n], r[at_m:at_m + m]))
        at_n, at_m = at_n + n, at_m + m
    return {"run": _run_batch, "keep": keep, "probs": probs, "x_hat": x_hat, "r": r,
            "params": ccs.params(), "results": ccs.result_buffer(len(probs)),
            "ws": ccs.workspace(ccs.ccs_batch_workspace_size(probs))}


def _run_batch(s):
    ccs.ccs_decode_batch_async(s["probs"], s["params"], s["results"], s["ws"])
    return {"x_hat": s["x_hat"], "r": s["r"], "results": s["results"]}


class _Burst:
    """A server and the host buffers of one burst; the server stops with it."""

    def __init__(self, case, seed):
        shapes = _problem_set(case, seed)
        total = sum(n for n, *_ in shapes)
        self.idx = np.zeros(total, dtype=np.int64)
        self.val = np.zeros(total, dtype=np.float64)
        self.nnz = np.zeros(len(shapes), dtype=np.int64)
        self.requests, pool, at = [], 16 << 20, 0
        for q, (n, m, d, k, sd) in enumerate(shapes):
            a_seed = inputs.expander_seed(sd)
            _, ptr, cols = ccs.make_expander(n, m, d, a_seed)
            y = ccs.measure(ptr, cols, _signal(n, k, "gauss-grid", sd), m, d).cpu().numpy()
            out = (self.idx[at:at + n], self.val[at:at + n], self.nnz[q:q + 1])
            self.requests.append((n, m, d, a_seed, y, out))
            pool += ccs.ccs_seeded_request_bytes(n, m, d, 100, n) + 256
            at += n
        self.server = ccs.Server(pool, max_batch=64)

    def __del__(self):
        if hasattr(self, "server"):
            self.server.close()


def _prepare_serve(case, seed):
    return {"run": _run_serve, "burst": _Burst(case, seed)}


def _run_serve(s):
    b = s["burst"]
    tickets = [b.server.submit_seeded(n, m, d, a_seed, y, nonzeros=out)
               for n, m, d, a_seed, y, out in b.requests]
    infos = [b.server.wait(t) for t in tickets]
    return {"idx": b.idx, "val": b.val, "nnz": b.nnz,
            "iterations": np.array([i.result.iterations for i in infos]),
            "status": np.array([i.result.status for i in infos])}


# ---- what a pass cannot do without, and its exact outputs ------------------------------

def _decode_bytes(n, m, d):
    """A's columns and y read, x_hat and r written."""
    return 4 * d * n + 8 * m + 8 * n + 8 * m


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        shapes = _problem_set(case, 0)
        if kind == "batch":
            total = sum(_decode_bytes(n, m, d) for n, m, d, _, _ in shapes)
        else:  # y in, the nonzeros out, A's columns made and read on the way
            total = sum(8 * d * n + 8 * m + 16 * k for n, m, d, k, _ in shapes)
        return {"bytes": total, "flops": 0}
    n, m, d = case["n"], case["m"], case["d"]
    transpose = 4 * d * n + 8 * (m + 1)
    return {"bytes": {"decode": _decode_bytes(n, m, d),
                      "scaled": transpose + 16 * n + 8 * m + _decode_bytes(n, m, d),
                      "expander": 4 * d * n + transpose,
                      "measure": transpose + 8 * n + 8 * m}[kind],
            "flops": 0}


def exact(case, seed):
    """A decode that recovers returns the signal itself and r = 0; that is
    taken for granted well inside the recovery region only.  On the grid
    y = A x is an exact sum in any order."""
    kind = case["kind"]
    if kind == "measure":
        n, m, d = case["n"], case["m"], case["d"]
        rows, _, _ = _own_matrix(n, m, d, seed)
        x = _signal(n, case["k"], "gauss-grid", seed)
        y = torch.zeros(m, dtype=torch.float64, device="cuda")
        at = x.nonzero().flatten()
        return y.index_add_(0, rows[at].flatten().long(), x[at].repeat_interleave(d))
    if kind not in ("decode", "scaled"):
        return None
    n, m, d, k = case["n"], case["m"], case["d"], case["k"]
    # columns sharing two rows with a given column compete with it
    collisions = n * math.comb(d, 2) ** 2 * 2 / m ** 2
    inside = (m >= 4000 and k <= 0.2 * m and collisions < 1 or
              m >= 16000 and k <= 0.11 * m and collisions < 20 or
              m >= 16000 and k <= 0.051 * m)
    if not 7 <= d <= 9 or not inside:
        return None
    if kind == "scaled":
        return {"y": None, "x": _signal(n, k, "pm1", seed),
                "r": torch.zeros(m, dtype=torch.float64, device="cuda")}
    if case["values"] != "gauss-grid" or case["score"] != "l0" or case["alpha"] != 2:
        return None
    return {"x_hat": _signal(n, k, case["values"], seed),
            "r": torch.zeros(m, dtype=torch.float64, device="cuda"), "outcome": None}
