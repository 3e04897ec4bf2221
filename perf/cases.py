"""What this framework is timed on: its public calls over the sizes they are used at.

A case is a dict of plain values with a "kind" (the call) and its sizes:

  round    ubqp.solve: one multi-start round, starts to best solution
  steps    the same round made of its separate calls, every result handed back
  rounds   ubqp.solve_rounds: several independent rounds of one instance together
  search   ubqp.search: the whole multi-round loop around an incumbent
  batch    Batch.run: one round for many instances of uneven size, tuned and captured
  serve    Server: host instances submitted together, then waited for
  eval     ubqp.eval: xQx of a batch of given solutions
  relink   ubqp.relink: path relinking between pairs of local optima
  load     Instance(...) into an arena from device coefficients, and a first evaluation

Instances are symmetric int8 matrices with coefficients uniform on [-100, 100],
an off-diagonal pair or diagonal element being nonzero with the given density.
"""
import math

import numpy as np
import torch

from paper_1706_00037_gb300 import ubqp

MODES = {"random": ubqp.RANDOM, "diversify": ubqp.DIVERSIFY}


def listed():
    return [
        # the smallest use: a sparse 100-variable problem, where launches and latency count
        {"name": "round_n100", "kind": "round", "n": 100, "density": 0.1, "starts": 1000,
         "mode": "diversify", "lam": 0.5},
        # a small dense problem just past a power of two (ragged tiles and rows)
        {"name": "round_n1025", "kind": "round", "n": 1025, "density": 1.0, "starts": 1000,
         "mode": "diversify", "lam": 0.5},
        # the shape of the ORLIB bqp2500 problems: 2500 variables at 10% density
        {"name": "round_n2500", "kind": "round", "n": 2500, "density": 0.1, "starts": 1000,
         "mode": "diversify", "lam": 0.5},
        # the benchmark's round: the largest Palubeckis size, dense, random starts
        {"name": "round_n7000", "kind": "round", "n": 7000, "density": 1.0, "starts": 1000,
         "mode": "random", "lam": 0.5},
        # a large batch of which half passes the screen, call by call, as a program that
        # keeps every intermediate result runs it
        {"name": "steps_n5000", "kind": "steps", "n": 5000, "density": 0.1, "starts": 8192,
         "mode": "diversify", "lam": 0.5},
        # four restarts of the benchmark's round with fresh seeds in one call
        {"name": "rounds_n7000", "kind": "rounds", "n": 7000, "density": 1.0, "starts": 1000,
         "mode": "random", "lam": 0.5, "rounds": 4},
        # the method end to end: a search of ten rounds around its incumbent
        {"name": "search_n2500", "kind": "search", "n": 2500, "density": 0.1, "starts": 1000,
         "lam": 0.5, "rounds": 10, "samples": 1000},
        # a portfolio of instances solved together
        {"name": "batch_32", "kind": "batch", "instances": 32, "n_min": 200, "n_max": 2500,
         "starts": 1024, "mode": "diversify", "lam": 0.5},
        # requests that arrive together from host memory
        {"name": "serve_8", "kind": "serve", "instances": 8, "n_min": 500, "n_max": 4000,
         "starts": 1024, "mode": "diversify", "lam": 0.5},
        # scoring of given solutions at the largest Table 1 size
        {"name": "eval_n7000", "kind": "eval", "n": 7000, "density": 1.0, "starts": 1000},
        # the polishing phase: 256 elite pairs
        {"name": "relink_n5000", "kind": "relink", "n": 5000, "density": 1.0, "pairs": 256},
        # a new instance taken in and looked at once; rows of odd length (not 4-byte aligned)
        {"name": "load_n6001", "kind": "load", "n": 6001, "density": 1.0, "starts": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["round", "round", "round", "steps", "rounds", "search", "batch", "serve",
                           "eval", "relink", "load"])
        c = {"kind": kind}
        if kind in ("batch", "serve"):
            c["instances"] = rng.randint(4, 32) if kind == "batch" else rng.randint(2, 16)
            c["n_min"], c["n_max"] = (200, 2500) if kind == "batch" else (500, 4000)
        else:
            c["n"] = _log_int(rng, 64, 7000)
            c["density"] = rng.choice([0.1, 0.5, 1.0])
        if kind == "relink":
            c["pairs"] = _log_int(rng, 16, 512)
        elif kind == "load":
            c["starts"] = _log_int(rng, 1, 256)
        else:
            c["starts"] = _log_int(rng, 100, 8192)
        if kind not in ("eval", "relink", "load"):
            c["lam"] = rng.choice([0.25, 0.5, 0.75])
            if kind != "search":
                c["mode"] = rng.choice(["random", "diversify"])
        if kind == "rounds":
            c["rounds"] = rng.randint(2, 4)
        if kind == "search":
            c["rounds"], c["samples"] = rng.randint(2, 10), _log_int(rng, 100, 1000)
        if _cost(c) <= most:
            return c


# ------------------------------------------------------------------ inputs
def _instance(n, density, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    v = torch.randint(-100, 101, (n, n), dtype=torch.int8, device="cuda", generator=g)
    if density < 1.0:
        v *= torch.rand((n, n), device="cuda", generator=g) < density
    up = torch.triu(v)
    return up + torch.triu(v, 1).T


def _sizes(case):
    """(n, density) of a batch's instances: the case's own, whatever the seed, so that passes
    on other inputs are the same work."""
    r = np.random.default_rng(case["instances"])
    lo, hi, k = case["n_min"], case["n_max"], case["instances"]
    if case["kind"] == "serve":  # requests: log-uniform
        ns = np.exp(r.uniform(math.log(lo), math.log(hi), k)).astype(int)
    else:
        ns = r.integers(lo, hi + 1, k)
    return [(int(n), float(d)) for n, d in zip(ns, r.choice([0.1, 0.5, 1.0], k))]


def _instances(case, seed):
    return [_instance(n, d, seed * 1000 + i) for i, (n, d) in enumerate(_sizes(case))]


def _solutions(n, S, seed):
    g = torch.Generator("cuda").manual_seed(seed + 7)
    W = (n + 63) // 64
    X = torch.randint(-2**63, 2**63 - 1, (S, W), dtype=torch.int64, device="cuda", generator=g)
    if n % 64:
        X[:, -1] &= (1 << (n % 64)) - 1
    return X


def _bytes(nbytes):
    return torch.empty(max(int(nbytes), 16), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        Qs = _instances(case, seed)
        p = ubqp.make_params(case["starts"], case["lam"], mode=MODES[case["mode"]], seed=seed)
        if kind == "serve":
            return {"kind": kind, "seed": seed, "Qs": [Q.cpu().pin_memory() for Q in Qs],
                    "server": ubqp.Server(4, case["n_max"], p)}
        plan = ubqp.Batch([ubqp.Instance(Q) for Q in Qs], p)
        plan.tune()
        plan.capture()
        return {"kind": kind, "seed": seed, "plan": plan}
    n = case["n"]
    Q = _instance(n, case["density"], seed)
    if kind == "load":
        return {"kind": kind, "Q": Q, "X": _solutions(n, case["starts"], seed),
                "arena": _bytes(ubqp.arena_size(n))}
    inst = ubqp.Instance(Q)
    st = {"kind": kind, "inst": inst, "seed": seed}
    S = case.get("starts")
    if kind == "eval":
        st["X"] = _solutions(n, S, seed)
        st["ws"] = _bytes(ubqp.eval_workspace_size(inst, S))
    elif kind == "relink":  # elite pairs: local optima, each toward the next
        P = case["pairs"]
        X = ubqp.diversify(inst, P, mode=ubqp.RANDOM, seed=seed)
        f = ubqp.eval(inst, X)
        every = torch.arange(P, dtype=torch.int32, device="cuda")
        ubqp.ascent(inst, X, f, every, torch.tensor([P], device="cuda"))
        st.update(X=X, f=f, G=X.roll(-1, 0).contiguous(),
                  ws=_bytes(ubqp.relink_workspace_size(inst, P)))
    elif kind == "search":
        st.update(args=(case["samples"], S, case["rounds"], case["lam"]))
    elif kind == "steps":
        st.update(S=S, lam=case["lam"], mode=MODES[case["mode"]],
                  ws=_bytes(max(ubqp.eval_workspace_size(inst, S),
                                ubqp.ascent_workspace_size(inst, S))))
    else:
        p = ubqp.make_params(S, case["lam"], mode=MODES[case["mode"]], seed=seed)
        st["p"] = p
        if kind == "rounds":
            st["R"] = case["rounds"]
            st["ws"] = _bytes(ubqp.solve_rounds_workspace_size(inst, p, case["rounds"]))
        else:
            st["ws"] = _bytes(ubqp.solve_workspace_size(inst, p))
    return st


def run(state):
    kind = state["kind"]
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(Q, seed=state["seed"] + i) for i, Q in enumerate(state["Qs"])]
        done = [server.wait(t) for t in tickets]
        return {"f": [np.array(bf, np.int64) for bf, _, _ in done],
                "x": [bx.view(np.int64) for _, bx, _ in done]}
    if kind == "batch":
        plan = state["plan"]
        plan.run(state["seed"])
        got = [plan.result(i) for i in range(len(plan.instances))]
        return {"x": torch.cat([bx for bx, _ in got]), "f": torch.stack([bf for _, bf in got])}
    if kind == "load":
        inst = ubqp.Instance(state["Q"], arena=state["arena"])
        return {"x0": ubqp.first_derivative(inst), "max_abs": inst.max_abs,
                "f": ubqp.eval(inst, state["X"])}
    inst = state["inst"]
    if kind == "eval":
        return ubqp.eval(inst, state["X"], ws=state["ws"])
    if kind == "relink":
        x, f, dist = ubqp.relink(inst, state["X"], state["f"], state["G"], ws=state["ws"])
        return {"x": x, "f": f, "dist": dist}
    if kind == "search":
        return ubqp.search(inst, *state["args"], seed=state["seed"])
    if kind == "rounds":
        x, f = ubqp.solve_rounds(inst, state["p"], state["R"], ws=state["ws"])
        return {"x": x, "f": f}
    if kind == "round":
        x, f, _ = ubqp.solve(inst, state["p"], ws=state["ws"], want_stats=False)
        return {"x": x, "f": f}
    S, ws = state["S"], state["ws"]
    X = ubqp.diversify(inst, S, mode=state["mode"], seed=state["seed"])
    f = ubqp.eval(inst, X, ws=ws)
    f0 = f.clone()
    sc = ubqp.screen(f, state["lam"])
    flips = torch.full((S,), -1, dtype=torch.int32, device="cuda")  # -1: did not pass
    ubqp.ascent(inst, X, f, sc["idx"], sc["count"], flips=flips, ws=ws)
    x, best = ubqp.best(f, X)
    return {"f0": f0, "count": sc["count"], "Tm": sc["Tm"], "stats": sc["stats"], "X": X, "f": f,
            "flips": flips, "best_x": x, "best_f": best}


# ------------------------------------------------------------------ work
# How many starts pass the screen and how many moves a climb takes, as shares of S and of n
# (rough means of measured rounds): random starts climb far, diversified ones start near the
# first-derivative solution.
_PASS = {("random", 0.25): 0.2, ("random", 0.5): 0.045, ("random", 0.75): 0.008,
         ("diversify", 0.25): 0.64, ("diversify", 0.5): 0.52, ("diversify", 0.75): 0.22}
_MOVES = {"random": 0.54, "diversify": 0.24}


def _round_work(n, S, mode, lam, rounds=1):
    W8 = (n + 63) // 64 * 8
    climbs = _PASS[mode, lam] * S * _MOVES[mode] * n
    return {"bytes": n * n + rounds * (S * W8 + 8 * S),
            "flops": rounds * (n * (n + 1) * S + 3.0 * n * climbs)}


def _moves_work(n, S, mode, lam, rounds=1):
    return rounds * 3.0 * n * _PASS[mode, lam] * S * _MOVES[mode] * n


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        each = [_round_work(n, case["starts"], case["mode"], case["lam"])
                for n, _ in _sizes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n = case["n"]
    W8 = (n + 63) // 64 * 8
    if kind == "eval":
        S = case["starts"]
        return {"bytes": n * (n + 1) // 2 + S * (W8 + 8), "flops": n * (n + 1) * S}
    if kind == "load":  # the coefficients read, the int8 copy and two bf16 triangles written
        S = case["starts"]
        return {"bytes": 2 * n * n + 2 * n * (n + 1), "flops": n * (n + 1) * S}
    if kind == "relink":  # y = Qx of each pair, then a walk of about 0.13 n steps
        P = case["pairs"]
        return {"bytes": n * n + 3 * P * W8 + 20 * P, "flops": 2.0 * n * n * P + 3.0 * n * P * 0.13 * n}
    mode = case.get("mode", "diversify")
    w = _round_work(n, case["starts"], mode, case["lam"], case.get("rounds", 1))
    if kind == "search":
        w["flops"] += n * (n + 1) * case["samples"]
    return w


def _cost(case):
    """Rough microseconds of a pass at the rates seen: products, moves (in chains) and bytes."""
    w = work(case)
    kind = case["kind"]
    if kind in ("eval", "load"):
        moves = 0.0
    elif kind == "relink":
        moves = 3.0 * case["n"] * case["pairs"] * 0.13 * case["n"]
    elif kind in ("batch", "serve"):
        moves = sum(_moves_work(n, case["starts"], case["mode"], case["lam"])
                    for n, _ in _sizes(case))
    else:
        moves = _moves_work(case["n"], case["starts"], case.get("mode", "diversify"), case["lam"],
                            case.get("rounds", 1))
    return (w["flops"] - moves) / 1e9 + moves / 6e6 + w["bytes"] / 3e6


# ------------------------------------------------------------------ plain versions
_M = (1 << 64) - 1
_GOLDEN = 0x9E3779B97F4A7C15


def _splitmix(z):
    with np.errstate(over="ignore"):
        z = z + np.uint64(_GOLDEN)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _rand(seed, stream, ctr):
    with np.errstate(over="ignore"):
        return _splitmix(np.uint64(seed & _M) ^ (np.asarray(stream, np.uint64) * np.uint64(_GOLDEN))
                         ^ np.asarray(ctr, np.uint64))


def _bits(X, n):
    """(S, W) words -> (S, n) 0/1 on the GPU."""
    X = torch.as_tensor(np.ascontiguousarray(X).view(np.int64)) if isinstance(X, np.ndarray) else X
    j = torch.arange(n, device="cuda")
    return (X.cuda()[:, j // 64] >> (j % 64)) & 1


def _words(x):
    S, n = x.shape
    W = (n + 63) // 64
    pad = torch.zeros((S, W * 64), dtype=torch.int64, device=x.device)
    pad[:, :n] = x
    return (pad.view(S, W, 64) << torch.arange(64, device=x.device)).sum(-1)


def _value(Q, x):
    """xQx of every row (S, n), exact in double."""
    Qd, out = Q.double(), []
    for part in x.split(1024):
        d = part.double()
        out.append(((d @ Qd) * d).sum(1))
    return torch.cat(out).round().to(torch.int64)


def _first_derivative(Q):
    return (Q.to(torch.int64).sum(1) > 0).to(torch.int64)


def _starts(inc, n, S, mode, seed, rnd, div_h=64):
    """The start rule: uniform words, or h-patterns and blends around the incumbent."""
    W = (n + 63) // 64
    w = np.arange(W, dtype=np.uint64)[None, :]
    if mode == "random":
        return _bits(_rand(seed, np.arange(S, dtype=np.uint64)[:, None], w), n)
    x = inc.expand(S, n).clone()
    i = rnd * S + np.arange(S, dtype=np.int64)
    j = torch.arange(n, device="cuda")
    even = np.nonzero((i % 2 == 0) & (i > 0))[0]
    if even.size:
        jp, H = i[even] // 2, min(n, div_h)
        h = 1 + (jp - 1) % H
        o = ((jp - 1) // H) % h
        rows = torch.as_tensor(even, device="cuda")
        h, o = (torch.as_tensor(v, device="cuda")[:, None] for v in (h, o))
        x[rows] = x[rows] ^ (j % h == o).to(torch.int64)
    odd = np.nonzero(i % 2 == 1)[0]
    if odd.size:
        c = i[odd].astype(np.uint64)[:, None]
        partner = _rand(seed, np.uint64(1 << 63) | c, w)
        m = 1 + ((i[odd] - 1) // 2) % 6
        mask = np.full(partner.shape, _M, np.uint64)
        for k in range(6):
            word = _rand(seed, np.uint64(1 << 62) | (np.uint64(8) * c + np.uint64(k)), w)
            mask = np.where((k < m)[:, None], mask & word, mask)
        rows = torch.as_tensor(odd, device="cuda")
        mk = _bits(mask, n)
        x[rows] = (x[rows] & (1 - mk)) | (_bits(partner, n) & mk)
    return x


def _screen(f, lam, mean_of=None, top=None):
    total, count = (int(f.sum()), f.numel()) if mean_of is None else mean_of
    mean = float(total) / float(count)
    top = int(f.max()) if top is None else top
    return mean + lam * (float(top) - mean), mean


def _walk(Q, x, f, guide=None):
    """Steepest 1-flip moves of every row, lowest index on ties: uphill while a gain is positive,
    or with a guide through the variables where the two differ.  (x, f, moves), and with a guide
    the best strictly between the ends."""
    P, n = x.shape
    x, f = x.clone(), f.clone()
    diag = Q.diagonal().to(torch.int64)
    y = torch.cat([part.double() @ Q.double() for part in x.split(1024)]).round().to(torch.int64)
    Q16 = Q.to(torch.int16)
    order = torch.arange(n - 1, -1, -1, device="cuda")
    moves = torch.zeros(P, dtype=torch.int64, device="cuda")
    rows = torch.arange(P, device="cuda")
    live = rows
    if guide is not None:
        todo = (x ^ guide).bool()
        dist = todo.sum(1)
        best_x, best_f = x.clone(), f.clone()
        live = rows[dist >= 2]
    step = 0
    ax, ay = x[live], y[live]
    while live.numel():
        gain = diag + 2 * (1 - 2 * ax) * ay
        if guide is not None:
            gain = torch.where(todo[live], gain, -(1 << 40))
        top = (gain * 16384 + order).amax(1)
        k = n - 1 - (top & 16383)
        g = top >> 14
        go = g > 0 if guide is None else torch.ones_like(g, dtype=torch.bool)
        r = torch.arange(live.numel(), device="cuda")
        d = torch.where(go, 1 - 2 * ax[r, k], 0)
        ax[r, k] += d
        ay += d[:, None] * Q16[k]
        f[live] += torch.where(go, g, 0)
        moves[live] += go
        step += 1
        if guide is not None:
            todo[live, k] = False
            inner = moves[live] < dist[live]
            up = inner & ((moves[live] == 1) | (f[live] > best_f[live]))
            best_f[live[up]] = f[live[up]]
            best_x[live[up]] = ax[up]
            keep = moves[live] < dist[live] - 1
        else:
            keep = go
        if step % 32 == 0 or guide is not None:
            if not bool(keep.all()):
                x[live] = ax
                live, ax, ay = live[keep], ax[keep], ay[keep]
    if guide is not None:
        return best_x, best_f, dist
    return x, f, moves


def _round(Q, S, mode, lam, seed, rnd=0):
    n = Q.shape[0]
    X = _starts(_first_derivative(Q), n, S, mode, seed, rnd)
    f0 = _value(Q, X)
    T, mean = _screen(f0, lam)
    idx = torch.nonzero(f0.double() > T).flatten()
    f, flips = f0.clone(), torch.full((S,), -1, dtype=torch.int32, device="cuda")
    if idx.numel():
        x, g, m = _walk(Q, X[idx], f0[idx])
        X[idx], f[idx], flips[idx] = x, g, m.to(torch.int32)
    return X, f0, f, flips, idx, T, mean


def _first_max(f):
    return int(torch.nonzero(f == f.max())[0])


def _best(X, f):
    b = _first_max(f)
    return _words(X[b:b + 1])[0], torch.tensor([int(f[b]), b])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        got = []
        for i, Q in enumerate(_instances(case, seed)):
            s = seed + i if kind == "serve" else seed
            X, _, f, *_ = _round(Q, case["starts"], case["mode"], case["lam"], s)
            got.append(_best(X, f))
        if kind == "serve":
            return {"f": [b for _, b in got], "x": [x for x, _ in got]}
        return {"x": torch.cat([x for x, _ in got]), "f": torch.stack([b for _, b in got])}
    n = case["n"]
    Q = _instance(n, case["density"], seed)
    if kind in ("eval", "load"):
        f = _value(Q, _bits(_solutions(n, case["starts"], seed), n))
        if kind == "eval":
            return f
        return {"x0": _words(_first_derivative(Q)[None])[0],
                "max_abs": int(Q.to(torch.int64).abs().max()), "f": f}
    if kind == "relink":
        x = _starts(None, n, case["pairs"], "random", seed, 0)
        x, f, _ = _walk(Q, x, _value(Q, x))
        bx, bf, dist = _walk(Q, x, f, guide=x.roll(-1, 0))
        return {"x": _words(bx), "f": bf, "dist": dist.to(torch.int32)}
    if kind == "rounds":
        got = []
        for k in range(case["rounds"]):
            X, _, f, *_ = _round(Q, case["starts"], case["mode"], case["lam"], seed + k, k)
            got.append(_best(X, f))
        return {"x": torch.stack([x for x, _ in got]), "f": torch.stack([b for _, b in got])}
    if kind == "search":
        S, NS = case["starts"], case["samples"]
        total = int(_value(Q, _starts(None, n, NS, "random", seed, 0)).sum())
        inc = _first_derivative(Q)
        top, hist, passed, moved = int(_value(Q, inc[None])[0]), [], 0, 0
        for r in range(case["rounds"]):
            X = _starts(inc, n, S, "diversify", seed, r)
            f = _value(Q, X)
            T, _ = _screen(f, case["lam"], (total, NS), top)
            idx = torch.nonzero(f.double() > T).flatten()
            if idx.numel():
                X[idx], f[idx], m = _walk(Q, X[idx], f[idx])
                passed, moved = passed + idx.numel(), moved + int(m.sum())
            b = _first_max(f)
            if int(f[b]) > top:
                top, inc = int(f[b]), X[b].clone()
            hist.append(top)
        return {"best_x": _words(inc[None])[0], "best_f": torch.tensor([top]),
                "history": torch.tensor(hist), "stats": torch.tensor([passed, moved, total])}
    X, f0, f, flips, idx, T, mean = _round(Q, case["starts"], case["mode"], case["lam"], seed)
    x, b = _best(X, f)
    if kind == "round":
        return {"x": x, "f": b}
    return {"f0": f0, "count": torch.tensor([idx.numel()]),
            "Tm": torch.tensor([T, mean], dtype=torch.float64),
            "stats": torch.tensor([int(f0.sum()), int(f0.max()), _first_max(f0)]),
            "X": _words(X), "f": f, "flips": flips, "best_x": x, "best_f": b}
