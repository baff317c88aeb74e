"""Measured cases of the relational hot path: what a program that uses this
library runs, through its public entry points, from calls of a few thousand
rows to columns of 2e8 rows.

A case is a dict of plain values.  Kinds:

  kv        group-by of one int64 / int32 key column and one int64 value
            column.  plan "exact": the exact distinct count and the sample
            sketch, then the run (the plain form); "learned": one
            groupby_auto call with the trained planner network; "hint": the
            caller knows the number of groups.
  lineitem  the fused filter + packed-key group-by with product expressions.
  report    a filtered group-by no specialised kernel covers: two range
            filters, a (uint8, int32) key, sums of products, min and max.
  join      hash build, then probe with pair emission and payload gather;
            "unique" build keys (a key column) or several rows per key.
  batch     many uneven group-bys and join partitions prepared once and
            replayed from a CUDA graph.
  train     one training step of the planner network.

Group order and pair order are unspecified, so run() ends as a program that
wants a definite order does: groups sorted by key (ORDER BY) into result
columns that it keeps, pairs of a unique-key join scattered to their probe
rows, other pairs sorted.  Result columns have room for every possible group
or pair; what is past the count is zero.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_13696_gb300 import planner, rel, workloads

OPS4 = ("sum", "count", "min", "max")
OPS2 = ("sum", "count")


def listed():
    return [
        # the smallest calls: a dashboard query over a few thousand rows, all latency
        {"name": "kv_small", "kind": "kv", "rows": 4001, "key": "int64", "aggs": 4,
         "family": "uniform", "s": 0.0, "domain": 37, "plan": "exact"},
        # the fused filter + aggregation at 1e6 rows (the benchmark's size)
        {"name": "lineitem_1e6", "kind": "lineitem", "rows": 1_000_000, "date_hi": 2430},
        # ... and over a full fact table, bound by its columns; ragged row count
        {"name": "lineitem_1e8", "kind": "lineitem", "rows": 100_000_007, "date_hi": 2430},
        # the large skewed group-by of the benchmark: millions of groups
        {"name": "zipf_2e8", "kind": "kv", "rows": 200_000_000, "key": "int64", "aggs": 4,
         "family": "zipf", "s": 1.1, "domain": 10_000_000, "plan": "exact"},
        # the large group-by with a handful of groups (the benchmark's)
        {"name": "fourkeys_2e8", "kind": "kv", "rows": 200_000_000, "key": "int64", "aggs": 4,
         "family": "uniform", "s": 0.0, "domain": 4, "plan": "exact"},
        # a mid-size group-by planned by the network, keys without skew
        {"name": "uniform_learned", "kind": "kv", "rows": 23_456_789, "key": "int64", "aggs": 4,
         "family": "uniform", "s": 0.0, "domain": 1_500_000, "plan": "learned"},
        # int32 keys in runs (a column clustered on load), group count known
        {"name": "clustered_i32", "kind": "kv", "rows": 6_000_001, "key": "int32", "aggs": 2,
         "family": "clustered", "s": 0.0, "domain": 20_000, "plan": "hint"},
        # a report query outside the specialised shapes
        {"name": "report_1e7", "kind": "report", "rows": 10_000_019, "stores": 700},
        # the benchmark's join: fact rows against a dimension's key column
        {"name": "join_1e6_16e6", "kind": "join", "build": 1_000_000, "probe": 16_000_000,
         "per_key": 1, "hit": 0.9},
        # a small join whose build keys repeat (several matches per row), sized by a count
        {"name": "join_dups", "kind": "join", "build": 60_013, "probe": 400_009, "per_key": 3,
         "hit": 0.8},
        # hundreds of uneven group-bys and joins in one prepared batch
        {"name": "batch_512_64", "kind": "batch", "groupbys": 512, "joins": 64},
        # training of the planner network at its batch size
        {"name": "train_256", "kind": "train", "batch": 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["kv", "kv", "kv", "kv", "lineitem", "report", "join", "join", "batch",
                       "train"])
    if kind == "kv":
        family, s = rng.choice([("uniform", 0.0), ("zipf", 0.5), ("zipf", 1.0), ("zipf", 1.1),
                                ("zipf", 1.5), ("clustered", 0.0)])
        return {"kind": "kv", "rows": _log(rng, 1_000, 150_000_000),
                "key": rng.choice(["int64", "int64", "int32"]), "aggs": rng.choice([4, 4, 2]),
                "family": family, "s": s, "domain": _log(rng, 2, 5_000_000),
                "plan": rng.choice(["exact", "exact", "learned", "hint"])}
    if kind == "lineitem":
        return {"kind": "lineitem", "rows": _log(rng, 10_000, 100_000_000),
                "date_hi": rng.randint(100, 2526)}
    if kind == "report":
        return {"kind": "report", "rows": _log(rng, 10_000, 10_000_000),
                "stores": _log(rng, 4, 5_000)}
    if kind == "join":
        if rng.random() < 0.6:
            return {"kind": "join", "build": _log(rng, 1_000, 1_000_000),
                    "probe": _log(rng, 8_000, 16_000_000), "per_key": 1,
                    "hit": rng.choice([0.3, 0.9, 0.9, 1.0])}
        return {"kind": "join", "build": _log(rng, 1_000, 200_000),
                "probe": _log(rng, 8_000, 1_000_000), "per_key": rng.randint(2, 5),
                "hit": rng.choice([0.5, 0.8])}
    if kind == "batch":
        return {"kind": "batch", "groupbys": _log(rng, 16, 500), "joins": _log(rng, 2, 60)}
    return {"kind": "train", "batch": _log(rng, 32, 1024)}


# ----------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _i64(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _mix64(x):
    """splitmix64 of an int64 tensor: a bijective scramble over all of int64."""
    z = x + _i64(0x9E3779B97F4A7C15)
    z ^= (z >> 30) & ((1 << 34) - 1)
    z *= _i64(0xBF58476D1CE4E5B9)
    z ^= (z >> 27) & ((1 << 37) - 1)
    z *= _i64(0x94D049BB133111EB)
    z ^= (z >> 31) & ((1 << 33) - 1)
    return z


def _ranks(g, family, s, n, domain):
    """n ranks in [1, domain]: uniform, Zipf(s) by the inverse of the
    integrated density, or uniform in runs of 64 rows."""
    if family == "zipf":
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        lo, hi = 0.5, domain + 0.5
        if s == 1.0:
            x = (u * math.log(hi / lo) + math.log(lo)).exp_()
        else:
            a, b = lo ** (1.0 - s), hi ** (1.0 - s)
            x = (u.mul_(b - a).add_(a)).pow_(1.0 / (1.0 - s))
        return x.add_(0.5).to(torch.int64).clamp_(1, domain)
    if family == "clustered":
        r = torch.randint(1, domain + 1, (n // 64 + 1,), generator=g, device="cuda")
        return r.repeat_interleave(64)[:n]
    return torch.randint(1, domain + 1, (n,), generator=g, device="cuda")


def _kv(g, family, s, n, domain, key):
    k = _mix64(_ranks(g, family, s, n, domain))
    if key == "int32":
        k = k.to(torch.int32)
    v = torch.randint(-1_000_000, 1_000_001, (n,), generator=g, device="cuda")
    return k.contiguous(), v


def _groups(family, s, n, domain):
    """Expected number of distinct keys of n draws."""
    if family == "zipf":
        x = np.geomspace(1.0, domain + 1.0, 20_001)
        mid, cnt = np.sqrt(x[1:] * x[:-1]), np.diff(x)
        p = mid ** -s
        p = p / float((p * cnt).sum())
        return float((cnt * -np.expm1(n * np.log1p(-np.minimum(p, 0.999)))).sum())
    draws = n / 64 if family == "clustered" else n
    return domain * -math.expm1(draws * math.log1p(-1.0 / domain)) if domain > 1 else 1.0


def _randint(g, lo, hi, n, dtype=torch.int64):
    return torch.randint(lo, hi + 1, (n,), generator=g, device="cuda", dtype=dtype)


def _join_sides(g, n_build, n_probe, per_key, hit):
    """Build keys scrambled over int64 (each key per_key times, shuffled),
    payloads, and probe keys of which the share `hit` is present."""
    n_keys = -(-n_build // per_key)
    ids = torch.arange(n_build, device="cuda") % n_keys
    if per_key > 1:
        ids = ids[torch.randperm(n_build, generator=g, device="cuda")]
    salt = int(torch.randint(0, 1 << 40, (1,), generator=g, device="cuda").item()) << 22
    bk = _mix64(ids + salt)
    bp = torch.randint(0, 1 << 62, (n_build,), generator=g, device="cuda")
    pick = torch.randint(0, n_keys, (n_probe,), generator=g, device="cuda")
    present = torch.rand(n_probe, generator=g, device="cuda") < hit
    pk = _mix64(torch.where(present, pick, pick + n_keys) + salt)
    return bk.contiguous(), bp, pk.contiguous()


def _batch_shapes(case):
    rng = np.random.default_rng([case["groupbys"], case["joins"]])
    lu = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    gb = [(lu(1e3, 4e6), lu(1, 1e5), "int32" if i % 2 == 0 else "int64")
          for i in range(case["groupbys"])]
    jn = [(lu(1e3, 2.56e5), lu(8e3, 2e6)) for _ in range(case["joins"])]
    return gb, jn


def _columns(n, count):
    return [torch.zeros(n, dtype=torch.int64, device="cuda") for _ in range(count)]


_registered = False


def _planner():
    global _registered
    if not _registered:
        planner.use_default()
        _registered = True


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "kv":
        n, d = case["rows"], case["domain"]
        k, v = _kv(g, case["family"], case["s"], n, d, case["key"])
        q = workloads.kv_query(k, v, OPS4 if case["aggs"] == 4 else OPS2)
        state = {"case": case, "q": q, "out": _columns(min(n, d), 1 + case["aggs"])}
        if case["plan"] == "learned":
            _planner()
            state["ws"] = torch.empty(rel.auto_ws_bytes(q), dtype=torch.uint8, device="cuda")
        return state
    if kind == "lineitem":
        n = case["rows"]
        li = {"flag": _randint(g, 0, 2, n, torch.uint8), "status": _randint(g, 0, 1, n, torch.uint8),
              "qty": _randint(g, 1, 50, n), "price": _randint(g, 90_000, 10_500_000, n),
              "disc": _randint(g, 0, 10, n), "tax": _randint(g, 0, 8, n),
              "date": _randint(g, 0, 2526, n, torch.int32)}
        return {"case": case, "q": workloads.lineitem_query(li, case["date_hi"]),
                "out": _columns(6, 6)}
    if kind == "report":
        n = case["rows"]
        cols = [_randint(g, 0, 4, n, torch.uint8), _randint(g, 1, case["stores"], n, torch.int32),
                _randint(g, 0, 364, n, torch.int32), _randint(g, 1, 500_000, n),
                _randint(g, 0, 30, n)]
        q = {"cols": cols, "keys": [0, 1], "preds": [(2, 30, 329), (3, 1_000, 499_000)],
             "aggs": [("sum", 3, [(4, 100, -1)]), ("min", 3, []), ("max", 3, []), ("count", 3, [])]}
        return {"case": case, "q": q, "out": _columns(5 * case["stores"], 5)}
    if kind == "join":
        sides = _join_sides(g, case["build"], case["probe"], case["per_key"], case["hit"])
        pairs = case["probe"] * case["per_key"] if case["per_key"] > 1 else 0
        return {"case": case, "sides": sides, "out": _columns(pairs, 2)}
    if kind == "batch":
        return _prepare_batch(case, g)
    b = case["batch"]
    x = torch.rand((b, rel.MLP_IN), generator=g, device="cuda")
    x[:, 256] = 10.0 + 16.0 * x[:, 256]  # log2 rows
    x[:, 258] *= 64.0                    # log2 key range
    x[:, 262] = 1.0 + 63.0 * x[:, 262]   # run length
    parts = []
    for fo, fi in ((rel.MLP_HIDDEN, rel.MLP_IN), (rel.MLP_HIDDEN, rel.MLP_HIDDEN),
                   (rel.MLP_OUT, rel.MLP_HIDDEN)):
        lim = 1.0 / math.sqrt(fi)
        parts.append((torch.rand(fo * fi, generator=g, device="cuda") * 2.0 - 1.0) * lim)
        parts.append((torch.rand(fo, generator=g, device="cuda") * 2.0 - 1.0) * 0.1)
    p = torch.cat(parts)
    p[-rel.MLP_OUT] = 10.0
    bf = torch.empty(rel.MLP_PARAMS, dtype=torch.bfloat16, device="cuda")
    rel.mlp_round(p, bf)
    ws = torch.empty(int(rel.load().rel_mlp_ws_bytes(b)), dtype=torch.uint8, device="cuda")
    return {"case": case, "x": x, "t": torch.rand(b, generator=g, device="cuda") * 24.0,
            "var": torch.randint(0, 3, (b,), generator=g, device="cuda", dtype=torch.int32),
            "p": p, "bf": bf, "m": torch.zeros_like(p), "v": torch.zeros_like(p),
            "acts": torch.empty((b, 2 * rel.MLP_HIDDEN), device="cuda"),
            "grad": torch.empty_like(p), "loss": torch.empty(1, device="cuda"), "ws": ws,
            "step": 0}


def _prepare_batch(case, g):
    gb, jn = _batch_shapes(case)
    gs = []
    for n, groups, key in gb:
        k, v = _kv(g, "uniform", 0.0, n, groups, key)
        est = min(n, groups)
        slots = 1 << max(4, (2 * est - 1).bit_length())
        # the planner's variant rule: per-CTA tables for few groups
        gs.append({"keys": k, "vals": v, "ops": list(OPS2), "slots": slots,
                   "est_groups": est if est <= 512 else 1 << 40, "capacity": min(n, slots)})
    js = []
    for nb, npr in jn:
        bk, bp, pk = _join_sides(g, nb, npr, 1, 0.9)
        js.append({"build_keys": bk, "build_payload": bp, "probe_keys": pk, "capacity": npr})
    b = rel.Batch(gs, js).prepare((512, 4, 1, 512))
    graph = b.capture()
    # flat positions of the outputs: instance and index inside it
    dev = "cuda"
    cap = torch.tensor(np.diff(b.gk_off), device=dev)
    inst = torch.repeat_interleave(torch.arange(len(gs), device=dev), cap)
    koff = torch.tensor(b.gk_off[:-1].copy(), device=dev)
    at = torch.arange(int(b.gk_off[-1]), device=dev) - koff[inst]
    agg0 = torch.tensor(b.ga_off[:-1].copy(), device=dev)[inst] + at
    jinst = torch.repeat_interleave(torch.arange(len(js), device=dev),
                                    torch.tensor(np.diff(b.j_off), device=dev))
    joff = torch.tensor(b.j_off[:-1].copy(), device=dev)
    jat = torch.arange(int(b.j_off[-1]), device=dev) - joff[jinst]
    return {"case": case, "batch": b, "graph": graph, "cap": cap, "inst": inst.to(torch.int16),
            "at": at.to(torch.int32), "agg0": agg0, "jinst": jinst.to(torch.int16),
            "jbase": joff[jinst], "jat": jat.to(torch.int32),
            "out": _columns(sum(min(n, groups) for n, groups, _ in gb), 3),
            "out_inst": torch.zeros(sum(min(n, groups) for n, groups, _ in gb), dtype=torch.int16,
                                    device=dev)}


# -------------------------------------------------------------------- runs

def _place(out, columns, order):
    """columns[i][order] into the leading rows of out[i], the rest zero."""
    n = order.numel()
    for o, c in zip(out, columns):
        torch.index_select(c, 0, order, out=o[:n])
        o[n:].zero_()
    return out


def _ordered(out, keys, aggs):
    return [keys.numel()] + _place(out, [keys] + list(aggs), torch.argsort(keys))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("kv", "lineitem", "report"):
        q = state["q"]
        mode = case.get("plan", "exact")
        if mode == "learned":
            keys, aggs, _ = rel.groupby_auto(q, flags=rel.PLAN_LEARNED | rel.PLAN_SKETCH,
                                             ws=state["ws"])
        elif mode == "hint":
            keys, aggs = rel.groupby(q, flags=rel.PLAN_SKETCH,
                                     groups_hint=max(1, min(case["domain"], case["rows"])))
        else:
            plan = rel.plan_groupby(q, flags=rel.PLAN_EXACT | rel.PLAN_SKETCH)
            keys, aggs = rel.groupby(q, plan=plan)
        return _ordered(state["out"], keys, aggs)
    if kind == "join":
        bk, bp, pk = state["sides"]
        table = rel.JoinTable(bk, bp)
        if case["per_key"] == 1:
            pi, bi, pay = table.probe(pk, capacity=pk.numel())
            # the build row and payload of every probe row, -1 / 0 without a match
            row = torch.full((pk.numel(),), -1, dtype=torch.int32, device="cuda")
            val = torch.zeros(pk.numel(), dtype=torch.int64, device="cuda")
            at = pi.to(torch.int64)
            return [row.scatter_(0, at, bi), val.scatter_(0, at, pay)]
        n = table.count(pk)
        pi, bi, pay = table.probe(pk, capacity=max(1, n))
        code = pi.to(torch.int64) * bk.numel() + bi
        return [n] + _place(state["out"], [code, pay], torch.argsort(code))
    if kind == "batch":
        return _run_batch(state)
    s = state
    y = rel.mlp_forward(s["bf"], s["p"], s["x"], s["acts"])
    rel.mlp_backward(s["bf"], s["x"], s["acts"], y, s["t"], s["var"], s["grad"], s["loss"],
                     ws=s["ws"])
    s["step"] += 1
    rel.mlp_adamw(s["p"], s["bf"], s["m"], s["v"], s["grad"], s["step"])
    return [y, s["loss"], s["grad"], s["p"], s["m"], s["v"]]


def _run_batch(s):
    b = s["batch"]
    s["graph"].replay()
    counts, flags = b.results()
    if any(flags):
        raise RuntimeError("an instance of the batch overflowed")
    ng = len(b.gspec)
    n = torch.tensor(counts, device="cuda")
    # group-bys as one table (instance, key, sum, count) in that order
    i = (s["at"] < n[:ng][s["inst"].to(torch.int64)]).nonzero().squeeze(1)
    i = i[torch.argsort(b.gkeys[i])]
    inst, o = torch.sort(s["inst"][i], stable=True)
    i = i[o]
    s["out_inst"][:i.numel()] = inst
    s["out_inst"][i.numel():].zero_()
    a0 = s["agg0"][i]
    second = a0 + s["cap"][inst.to(torch.int64)]
    for o, c, at in zip(s["out"], (b.gkeys, b.gaggs, b.gaggs), (i, a0, second)):
        _place([o], [c], at)
    # joins: build row and payload per probe row, -1 / 0 without a match
    j = (s["jat"] < n[ng:][s["jinst"].to(torch.int64)]).nonzero().squeeze(1)
    to = s["jbase"][j] + b.jpi[j]
    row = torch.full((s["jat"].numel(),), -1, dtype=torch.int32, device="cuda")
    val = torch.zeros(s["jat"].numel(), dtype=torch.int64, device="cuda")
    return [n, s["out_inst"], *s["out"], row.scatter_(0, to, b.jbi[j]),
            val.scatter_(0, to, b.jpay[j])]


# -------------------------------------------------------------------- work

def work(case):
    kind = case["kind"]
    if kind == "kv":
        n = case["rows"]
        row = (8 if case["key"] == "int64" else 4) + 8
        groups = _groups(case["family"], case["s"], n, case["domain"])
        return {"bytes": n * row + groups * 8 * (1 + case["aggs"]), "flops": 0}
    if kind == "lineitem":
        return {"bytes": case["rows"] * 38 + 6 * 48, "flops": 0}
    if kind == "report":
        return {"bytes": case["rows"] * 25 + 5 * case["stores"] * 40, "flops": 0}
    if kind == "join":
        pairs = case["probe"] * case["hit"] * case["per_key"]
        return {"bytes": case["build"] * 16 + case["probe"] * 8 + pairs * 16, "flops": 0}
    if kind == "batch":
        # means of the log-uniform rows, groups, build and probe sides
        mean = lambda lo, hi: (hi - lo) / math.log(hi / lo)  # noqa: E731
        gb = case["groupbys"] * (mean(1e3, 4e6) * 14 + 0.8 * mean(1, 1e5) * 24)
        jn = case["joins"] * (mean(1e3, 2.56e5) * 16 + mean(8e3, 2e6) * (8 + 0.9 * 16))
        return {"bytes": gb + jn, "flops": 0}
    b, p = case["batch"], rel.MLP_PARAMS
    return {"bytes": 4 * b * (rel.MLP_IN + 128 + 4 + 2) + p * (4 * 7 + 2), "flops": 6 * b * p}


# ------------------------------------------------------------------- exact

def exact(case, seed):
    """The training step in 64 bits (BF16 weights, inputs and hidden
    activations as the network defines them); every other output is whole
    numbers, which have no nearer value."""
    if case["kind"] != "train":
        return None
    s = prepare(case, seed)
    d = lambda t: t.to(torch.float64)  # noqa: E731
    bf = lambda t: d(t.to(torch.float32).to(torch.bfloat16))  # noqa: E731
    H, I, O, b = rel.MLP_HIDDEN, rel.MLP_IN, rel.MLP_OUT, case["batch"]
    sizes = [H * I, H, H * H, H, O * H, O]
    w1, _, w2, _, w3, _ = torch.split(d(s["bf"]), sizes)
    _, b1, _, b2, _, b3 = torch.split(d(s["p"]), sizes)
    w1, w2, w3 = w1.view(H, I), w2.view(H, H), w3.view(O, H)
    x = bf(s["x"])
    z1 = x @ w1.T + b1
    h1 = bf(z1.clamp_min(0))
    z2 = h1 @ w2.T + b2
    h2 = bf(z2.clamp_min(0))
    y = h2 @ w3.T + b3
    lab = s["var"].to(torch.int64)
    prob = torch.softmax(y[:, 1:], dim=1)
    err = y[:, 0] - d(s["t"])
    ce = -torch.log_softmax(y[:, 1:], dim=1).gather(1, lab[:, None]).squeeze(1)
    loss = ((err * err + ce).sum() / b).reshape(1)
    one = torch.nn.functional.one_hot(lab, 3).to(torch.float64)
    dy = torch.cat([2 * err[:, None], prob - one], dim=1) / b
    d2 = (dy @ w3) * (z2 > 0)
    d1 = (d2 @ w2) * (z1 > 0)
    grad = torch.cat([(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0),
                      (dy.T @ h2).reshape(-1), dy.sum(0)])
    lr, b1_, b2_, eps, wd = 1e-3, 0.9, 0.999, 1e-8, 1e-4
    m, v = (1 - b1_) * grad, (1 - b2_) * grad * grad
    decay = torch.cat([torch.full((n,), wd if k % 2 == 0 else 0.0, dtype=torch.float64,
                                  device="cuda") for k, n in enumerate(sizes)])
    p = d(s["p"])
    p = p - lr * decay * p
    p = p - lr * (m / (1 - b1_)) / ((v / (1 - b2_)).sqrt() + eps)
    return [y, loss, grad, p, m, v]
