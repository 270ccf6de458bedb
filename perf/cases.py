"""What this framework is timed on: calls of its public entry points as a
user's program makes them, over the sizes its workloads have (synth.py) --
kernel sets of 5 to 12 kernels whose whole permutation space is scored, sets
of up to 24 kernels scored by lists of orders and searched, simulated GPUs of
13, 15 and 148 SMs, and the surrogate network's own calls.

A case is a dict of plain values; ``prepare`` builds what the program holds
before the call, ``run`` is one pass.  Every makespan, count and histogram is
a whole number; the network's outputs are floating point.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1511_07983_gb300 import ko, synth

IN, HID = 192, 256           # the surrogate's encoded width and hidden width
SLOTS, SLOT_FEATURES = 24, 7
OPS_PER_PLACEMENT = 27       # integer operations of one placement: fit test, usage, sums, duration, release


def listed() -> list[dict]:
    return [
        # a handful of hand-picked orders compared (the smallest call; host buffers in and out)
        {"name": "orders16_n8_13sm", "kind": "orders", "workload": "single8", "n": 8, "count": 16,
         "source": "rows", "where": "host"},
        # one 8-kernel set ranked in its whole space, tuned on itself (40,320 orders)
        {"name": "rank_n8_13sm", "kind": "rank", "workload": "single8", "n": 8, "tune": "self"},
        # one ten-kernel set of the 64-set study ranked, with the batch tuner's choice (3.6M orders)
        {"name": "rank_n10_15sm", "kind": "rank", "workload": "sets10", "n": 10, "tune": "class"},
        # the headline's 148-SM sets, one kernel fewer: 39.9M orders ranked with a 4096-bin histogram
        {"name": "rank_n11_148sm", "kind": "rank", "workload": "single12", "n": 11, "tune": "class"},
        # every makespan of a nine-kernel set on the large GPU, options left alone (the study's call)
        {"name": "all_n9_148sm", "kind": "all", "workload": "single12", "n": 9},
        # a population of mixed sets (N 5..10 on 13, 15 and 148 SMs) in one captured graph
        {"name": "batch_48_mixed", "kind": "batch", "sets": 48, "nbins": 0},
        # a sample of a twelve-kernel space by Lehmer index, device buffers (an odd count)
        {"name": "indices_n12_148sm", "kind": "orders", "workload": "single12", "n": 12, "count": 100003,
         "source": "idx", "where": "device"},
        # exact steepest descent from Algorithm 1's order of a set too large to enumerate
        {"name": "descent_n20", "kind": "descent", "workload": "large", "n": 20},
        # guided search with the benchmark's settings: screening, rounds of rescored neighbours, descent
        {"name": "search_n20", "kind": "search", "workload": "large", "n": 20, "candidates": 1 << 18, "rounds": 6},
        # the network's forward pass over encoded orders held by the host
        {"name": "predict_65536", "kind": "predict", "rows": 65536},
        # loss and gradients of one minibatch
        {"name": "grad_4096", "kind": "grad", "rows": 4096},
        # a training run: exact labels for every set, then minibatch steps; returns curve and weights
        {"name": "train_32x4096", "kind": "train", "sets": 32, "pairs": 4096, "steps": 96, "batch": 4096},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    """One more case; sizes spread over their logarithm, odd ones included."""
    kind = rng.choice(["orders", "orders", "rank", "rank", "all", "batch", "descent", "search", "predict", "grad",
                       "train"])
    if kind == "orders":
        n = rng.randint(5, 24)
        return {"kind": kind, "workload": rng.choice(["single8", "sets10", "single12"]), "n": n,
                "count": _log_int(rng, 5, 100003), "source": "rows" if n > 20 else rng.choice(["rows", "idx"]),
                "where": rng.choice(["host", "device"])}
    if kind == "rank":
        return {"kind": kind, "workload": rng.choice(["single8", "sets10", "single12"]), "n": rng.randint(5, 10),
                "tune": "class"}
    if kind == "all":
        return {"kind": kind, "workload": rng.choice(["single8", "sets10", "single12"]), "n": rng.randint(5, 9)}
    if kind == "batch":
        return {"kind": kind, "sets": _log_int(rng, 2, 24), "nbins": rng.choice([0, 1000, 4096])}
    if kind == "descent":
        return {"kind": kind, "workload": "large", "n": rng.randint(8, 24)}
    if kind == "search":
        return {"kind": kind, "workload": "large", "n": rng.randint(16, 24),
                "candidates": _log_int(rng, 5000, 1 << 20), "rounds": rng.randint(0, 8)}
    if kind == "predict":
        return {"kind": kind, "rows": 64 * _log_int(rng, 1, 1024)}
    if kind == "grad":
        return {"kind": kind, "rows": 64 * _log_int(rng, 1, 128)}
    return {"kind": kind, "sets": _log_int(rng, 4, 32), "pairs": _log_int(rng, 500, 4096),
            "steps": _log_int(rng, 16, 96), "batch": 64 * _log_int(rng, 4, 64)}


# ------------------------------------------------------------------- inputs

def _set(case: dict, seed: int):
    return synth.gen_set(case["workload"], 10_000 + seed, n=case["n"])


def _batch_sets(case: dict, seed: int):
    return [synth.gen_set("batched", 100_000 + 1000 * seed + i) for i in range(case["sets"])]


def _rows(n: int, count: int, seed: int) -> np.ndarray:
    """`count` uniform orders of n kernels, int8."""
    rng = np.random.default_rng([seed, n, 1])
    return np.argsort(rng.random((count, n)), axis=1).astype(np.int8)


def _indices(n: int, count: int, seed: int) -> np.ndarray:
    rng = np.random.default_rng([seed, n, 2])
    return rng.integers(0, math.factorial(n), size=count, dtype=np.uint64)


def _class_options(n_sm: int, n: int) -> dict:
    """The tuner's choices per (N_SM class, N), fixed so that a prepared handle
    is the same every time; the library's defaults where a class is too small
    for the tuner to time."""
    if n_sm <= 16:
        return {7: dict(lanes=1, levels=1, lane_state=2), 8: dict(lanes=1, levels=2, lane_state=2),
                9: dict(lanes=1, levels=2, lane_state=2)}.get(n, dict(lanes=1, levels=3, lane_state=1) if n > 9 else {})
    return {8: dict(lanes=1, levels=2, lane_state=1), 9: dict(lanes=1, levels=2, lane_state=1),
            10: dict(lanes=1, levels=3, lane_state=1)}.get(n, dict(lanes=1, levels=4, lane_state=0) if n > 10 else {})


def _features(rows: int, seed: int):
    """Encoded orders as the encoder lays them out (slots of kernel descriptors
    in launch order, then globals), rounded to bfloat16, and log2 targets."""
    rng = np.random.default_rng([seed, rows, 3])
    sets, n = 16, int(rng.integers(6, 25))
    feat = np.empty((sets, n, SLOT_FEATURES))
    feat[..., 0] = rng.integers(16, 64, (sets, n)) * rng.choice([128, 256, 512], (sets, n)) / 65536
    feat[..., 1] = rng.integers(0, 7, (sets, n)) * 4096 / 49152
    feat[..., 2] = rng.choice([4, 8, 16], (sets, n)) / 64
    feat[..., 3] = rng.integers(1, 10, (sets, n)) / 16
    feat[..., 4] = np.log2(rng.integers(1000, 50001, (sets, n))) / 16
    feat[..., 5] = feat[..., 4] + rng.uniform(-3.3, 3.3, (sets, n)) / 16
    feat[..., 6] = 1.0
    which = rng.integers(0, sets, rows)
    order = np.argsort(rng.random((rows, n)), axis=1)
    slot = np.round(23 * np.arange(n) / (n - 1)).astype(int)
    x = np.zeros((rows, SLOTS, SLOT_FEATURES), dtype=np.float32)
    x[:, slot] = feat[which[:, None], order]
    glob = np.array([n / 24, 13 / 148, 16 / 24, 15.6 / 24, 6 / 24, 4 / 24, 0.55, 1.0], dtype=np.float32)
    x = np.concatenate([x.reshape(rows, -1), np.tile(glob, (rows, 1)),
                        np.zeros((rows, IN - SLOTS * SLOT_FEATURES - 8), np.float32)], axis=1)
    x = torch.from_numpy(x).to(torch.bfloat16).to(torch.float32).numpy()
    return np.ascontiguousarray(x), rng.uniform(0.0, 3.0, rows).astype(np.float32)


def _weights(seed: int) -> np.ndarray:
    """He-normal weights in the model's order: W1, b1, W2, b2, W3, b3, w4, b4."""
    rng = np.random.default_rng([seed, 4])
    live = SLOTS * SLOT_FEATURES + 8
    w1 = rng.normal(0, math.sqrt(2 / live), (IN, HID))
    w1[live:] = 0.0
    parts = [w1, rng.normal(0, 0.05, HID)]
    for _ in range(2):
        parts += [rng.normal(0, math.sqrt(2 / HID), (HID, HID)), rng.normal(0, 0.05, HID)]
    parts += [rng.normal(0, math.sqrt(1 / HID), HID), rng.normal(0, 0.05, 1)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


# --------------------------------------------------------------------- cases

def prepare(case: dict, seed: int) -> dict:
    torch.cuda.init()
    kind = case["kind"]
    st: dict = {"case": case}
    if kind in ("orders", "rank", "all", "descent", "search"):
        s = _set(case, seed)
        g = ko.Gpu.from_set(s)
        st["gpu"] = g
        if kind == "orders":
            rows = case["source"] == "rows"
            data = _rows(s.n, case["count"], seed) if rows else _indices(s.n, case["count"], seed)
            if case["where"] == "device":
                data = torch.from_numpy(data if rows else data.view(np.int64)).cuda()
                st["out"] = torch.empty(case["count"], dtype=torch.int64, device="cuda")
            st["rows" if rows else "idx"] = data
        elif kind == "rank":
            if case["tune"] == "self":
                g.autotune()
            else:
                g.configure(**_class_options(s.gpu[0], s.n))
        elif kind == "all":
            st["out"] = torch.empty(math.factorial(s.n), dtype=torch.int64, device="cuda")
        elif kind == "search":
            st["model"] = ko.Model(seed=seed)
            st["model"].set_params(_weights(seed))
            st["seed"] = seed
    elif kind == "batch":
        sets = _batch_sets(case, seed)
        st["gpus"] = [ko.Gpu.from_set(s).configure(**_class_options(s.gpu[0], s.n)) for s in sets]
        st["batch"] = ko.Batch(st["gpus"], nbins=case["nbins"])
    elif kind == "train":
        st["gpus"] = [ko.Gpu.from_set(synth.gen_set("train", 100_000 + 1000 * seed + i))
                      for i in range(case["sets"])]
        st["model"], st["params"], st["seed"] = ko.Model(seed=seed), _weights(seed), seed
    else:
        st["x"], st["t"] = _features(case["rows"], seed)
        st["model"] = ko.Model(seed=seed)
        st["model"].set_params(_weights(seed))
    return st


def run(st: dict):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "orders":
        return st["gpu"].eval_orders(idx=st.get("idx"), orders=st.get("rows"), out=st.get("out"))
    if kind == "rank":
        rank, hist = st["gpu"].rank_order(None, nbins=4096)
        return {**rank, "hist": hist}
    if kind == "all":
        st["gpu"].eval_all(st["out"])
        return st["out"]
    if kind == "batch":
        ranks, hists = st["batch"].run()
        table = {f: np.array([r[f] for r in ranks]) for f in ranks[0]}  # one column per statistic
        return table if hists is None else {**table, "hist": hists}
    if kind == "descent":
        order, makespan, steps, simulated, _ = st["gpu"].local_search()
        return {"order": order, "makespan": makespan, "steps": steps, "simulated": simulated}
    if kind == "search":
        order, makespan, _ = st["model"].search(st["gpu"], n_cand=case["candidates"], rounds=case["rounds"],
                                                seed=st["seed"])
        return {"order": order, "makespan": makespan}
    if kind == "predict":
        return st["model"].predict(st["x"])
    if kind == "grad":
        grad, loss = st["model"].grad(st["x"], st["t"])
        return {"grad": grad, "loss": loss}
    st["model"].set_params(st["params"])  # every pass trains from the same weights
    curve = st["model"].train(st["gpus"], pairs_per_set=case["pairs"], steps=case["steps"], batch=case["batch"],
                              seed=st["seed"])
    return {"curve": curve, "params": st["model"].get_params()}


def _nodes(n: int) -> int:
    """Kernel placements of a space whose orders share their prefixes."""
    return sum(math.factorial(n) // math.factorial(n - d) for d in range(1, n + 1))


def work(case: dict) -> dict:
    """Bytes in and out, and operations: for the simulator the integer
    operations of one placement per kernel placed (a kernel starts at least one
    group of blocks; orders of a whole space share their prefixes), for the
    network its multiply-adds."""
    kind = case["kind"]
    fwd = 2 * (IN * HID + 2 * HID * HID + HID)
    params = 4 * ko.KO_MODEL_PARAMS
    if kind == "orders":
        n, count = case["n"], case["count"]
        return {"bytes": count * ((n if case["source"] == "rows" else 8) + 8) + 28 * n,
                "flops": count * n * OPS_PER_PLACEMENT}
    if kind == "rank":
        return {"bytes": 28 * case["n"] + 8 * 4096 + 88, "flops": _nodes(case["n"]) * OPS_PER_PLACEMENT}
    if kind == "all":
        return {"bytes": 28 * case["n"] + 8 * math.factorial(case["n"]),
                "flops": _nodes(case["n"]) * OPS_PER_PLACEMENT}
    if kind == "batch":  # N uniform in 5..10
        mean = sum(_nodes(n) for n in range(5, 11)) / 6
        return {"bytes": case["sets"] * (28 * 8 + 88 + 8 * case["nbins"]),
                "flops": int(case["sets"] * mean) * OPS_PER_PLACEMENT}
    if kind == "descent":  # the first neighbourhood at least
        n = case["n"]
        return {"bytes": 28 * n + 4 * n + 8, "flops": 3 * n * (n - 1) // 2 * n * OPS_PER_PLACEMENT}
    if kind == "search":
        n = case["n"]
        return {"bytes": 28 * n + 4 * n + 8 + params,
                "flops": case["candidates"] * fwd + (1024 + 256 * case["rounds"]) * n * OPS_PER_PLACEMENT}
    if kind == "predict":
        return {"bytes": case["rows"] * (4 * IN + 4) + params, "flops": case["rows"] * fwd}
    if kind == "grad":
        return {"bytes": case["rows"] * (4 * IN + 4) + 2 * params, "flops": 3 * case["rows"] * fwd}
    return {"bytes": case["sets"] * 28 * 9 + 2 * params + 4 * case["steps"],
            "flops": case["sets"] * case["pairs"] * 9 * OPS_PER_PLACEMENT + 3 * case["steps"] * case["batch"] * fwd}


# ----------------------------------------------------------------- exactness

def _makespan(gpu, kernels, order) -> int:
    """One order block by block: strict first-in-first-out dispatch, round-robin
    first fit, durations fixed at the end of each burst."""
    n_sm, limit, cap = gpu[0], np.array(gpu[1:5]), gpu[5:7]
    need = [np.array([r, s, w, 1]) for r, s, w, *_ in kernels]
    used, demand = np.zeros((n_sm, 4), int), np.zeros((n_sm, 2), int)
    queue = [k for k in order for _ in range(kernels[k][3])]
    head, pointer, now, running = 0, 0, 0, []
    while True:
        started = []
        while head < len(queue):
            k = queue[head]
            fits = np.flatnonzero(np.all(used + need[k] <= limit, axis=1))
            if fits.size == 0:
                break
            sm = int(fits[np.argmin((fits - pointer) % n_sm)])
            used[sm] += need[k]
            demand[sm] += kernels[k][4:6]
            started.append((sm, k))
            pointer, head = (sm + 1) % n_sm, head + 1
        for sm, k in started:
            running.append((now + max(-(-int(kernels[k][4 + i]) * max(int(demand[sm, i]), cap[i]) // cap[i])
                                      for i in range(2)), sm, k))
        if not running:
            return now
        now = min(e for e, _, _ in running)
        for end, sm, k in [r for r in running if r[0] == now]:
            used[sm] -= need[k]
            demand[sm] -= kernels[k][4:6]
        running = [r for r in running if r[0] != now]


def _unrank(index: int, n: int) -> list[int]:
    rest, order = list(range(n)), []
    for d in range(n - 1, -1, -1):
        q, index = divmod(index, math.factorial(d))
        order.append(rest.pop(q))
    return order


def _split(flat: np.ndarray):
    out, at = [], 0
    for shape in ((IN, HID), (HID,), (HID, HID), (HID,), (HID, HID), (HID,), (HID, 1), (1,)):
        size = math.prod(shape)
        out.append(torch.from_numpy(flat[at:at + size].astype(np.float64)).reshape(shape))
        at += size
    return out


def exact(case: dict, seed: int):
    """Short order lists block by block, the network in 64 bits; None where a
    whole space or a long list would have to be simulated."""
    kind = case["kind"]
    if kind == "orders" and case["count"] * case["n"] <= 256 and case["workload"] != "single12":
        s = _set(case, seed)
        rows = (_rows(s.n, case["count"], seed).tolist() if case["source"] == "rows" else
                [_unrank(int(i), s.n) for i in _indices(s.n, case["count"], seed)])
        return np.array([_makespan(s.gpu, s.kernels.tolist(), r) for r in rows], dtype=np.int64)
    if kind not in ("predict", "grad"):
        return None
    x, t = _features(case["rows"], seed)
    w = _split(_weights(seed))
    a = [torch.from_numpy(x).double()]
    for i in (0, 2, 4):
        a.append(torch.relu(a[-1] @ w[i] + w[i + 1]))
    y = (a[3] @ w[6] + w[7])[:, 0]
    if kind == "predict":
        return y.numpy()
    d = y - torch.from_numpy(t).double()
    dz = (2.0 / len(d)) * d[:, None]
    grads = []
    for i, act in ((6, a[3]), (4, a[2]), (2, a[1]), (0, a[0])):
        grads = [act.T @ dz, dz.sum(0)] + grads
        if i:
            dz = (dz @ w[i].T) * (act > 0)
    return {"grad": torch.cat([g.reshape(-1) for g in grads]).numpy(), "loss": float((d * d).mean())}
