"""The work that users of the scan library have it do, as timed cases.

Every case goes through the package's Python entry points with the built-in
launch shapes (nothing tuned beforehand) on synthetic columns: uniform values,
or the sorted multiset with a fraction `swapped` of its positions displaced.
Sizes follow the repository's own workloads: single scans of 1e5 to 2^28
values, zone-mapped columns, selects, conjunctions, column loading, batches of
columns with log-uniform lengths, a burst of queries on a server, and the
planner's network.

  listed()            the listed cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) inputs and handles a program has before the call, on the GPU
  run(state)          one pass
  work(case)          bytes the pass cannot do without (inputs once, outputs once) and operations
  exact(case, seed)   what run returns, from plain torch on 64-bit integers (or float64)
"""
import math
import random

import numpy as np
import torch

from paper_2606_22423_gb300 import gbscan

SERVE_WIDTHS = (4, 8, 12, 16, 24, 32)   # the serving table's widths


def listed():
    return [
        # a point lookup on a small dimension column, result on the host: latency is all
        dict(name="point_scan", kind="scan", n=100_003, b=11, base=1000, sigma=0.01, order="uniform",
             layout="lanes", strategy="branchfree", host=True),
        # the plain single-column scan: 2^24 values of 8 bits, a tenth selected
        dict(name="plain_scan_b8", kind="scan", n=1 << 24, b=8, base=0, sigma=0.1, order="uniform",
             layout="lanes", strategy="branchfree", host=False),
        # the width sweep at full size: a narrow width (decoding against bandwidth)
        dict(name="sweep_b5", kind="scan", n=1 << 28, b=5, base=0, sigma=0.5, order="uniform",
             layout="lanes", strategy="branchfree", host=False),
        # a middle width with the branchy kernel, a ragged tail and a frame of reference
        dict(name="sweep_b12_branchy", kind="scan", n=(1 << 28) - 12_345, b=12, base=1 << 20, sigma=0.1,
             order="uniform", layout="lanes", strategy="branchy", host=False),
        # a column another system packed: one row-major bit stream
        dict(name="rowmajor_b18", kind="scan", n=(1 << 27) + 77, b=18, base=0, sigma=0.1, order="uniform",
             layout="rowmajor", strategy="branchfree", host=False),
        # a clustered (time-ordered) column with a zone map, the library picking the strategy
        dict(name="zone_sorted_auto", kind="scan", n=1 << 28, b=16, base=0, sigma=0.1, order="sorted",
             swapped=0.0, layout="lanes", strategy="auto", host=False),
        # positions of the matching rows, for a later gather or join
        dict(name="select_b16", kind="select", n=1 << 27, b=16, base=0, sigma=0.1, strategy="branchfree"),
        # WHERE a AND b AND c, SUM of d, over one table
        dict(name="conj_3_of_2e26", kind="conj", n=(1 << 26) + 5, widths="8,12,16", agg=24, sigma=0.5),
        # loading a column: encode on the GPU, wrap, build its zone map
        dict(name="load_b13", kind="load", n=1 << 27, b=13, base=0, order="uniform"),
        # a thousand columns of uneven lengths and widths in one planned launch
        dict(name="batch_1024", kind="batch", ncols=1024, total=1 << 29),
        # a burst of 1-8 column queries on a resident table of mixed widths and orders
        dict(name="serve_burst_48", kind="serve", columns=12, n=1 << 24, queries=48),
        # planning a batch of columns and one training pass of the planner's network
        dict(name="planner", kind="planner", plan_rows=4096, train_rows=160),
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(["scan"] * 6 + ["select", "conj", "load", "batch", "serve", "planner"])
    sigma = math.exp(rng.uniform(math.log(1e-4), 0.0))
    b = rng.randint(1, 32)
    base = rng.choice([0, rng.randint(1, 1 << 20)]) if b < 31 else 0
    order = rng.choice(["uniform", "sorted"])
    if kind == "scan":
        layout = rng.choice(["lanes", "lanes", "lanes", "rowmajor"] + (["bytes"] if b in (8, 16, 32) else []))
        strategies = ["branchfree", "branchy"]
        if layout == "lanes" and order == "sorted":
            strategies += ["auto", "zone_bf", "zone_br", "zone_agg_bf"]
        case = dict(kind=kind, n=_log_int(rng, 1000, 1 << 28), b=b, base=base, sigma=sigma, order=order,
                    layout=layout, strategy=rng.choice(strategies), host=rng.random() < 0.3)
        if order == "sorted":
            case["swapped"] = rng.choice([0.0, 0.01, 0.1])
        return case
    if kind == "select":
        return dict(kind=kind, n=_log_int(rng, 1000, 1 << 27), b=b, base=base, sigma=sigma,
                    strategy=rng.choice(["branchfree", "branchy"]))
    if kind == "conj":
        widths = [rng.randint(1, 24) for _ in range(rng.randint(1, 3))]
        return dict(kind=kind, n=_log_int(rng, 1000, 1 << 26), widths=",".join(map(str, widths)),
                    agg=rng.choice([0, rng.randint(1, 24)]), sigma=rng.uniform(0.05, 0.9))
    if kind == "load":
        return dict(kind=kind, n=_log_int(rng, 1000, 1 << 27), b=b, base=base, order=order)
    if kind == "batch":
        ncols = _log_int(rng, 8, 1024)
        return dict(kind=kind, ncols=ncols, total=ncols * _log_int(rng, 1 << 13, 1 << 19))
    if kind == "serve":
        return dict(kind=kind, columns=rng.randint(6, 12), n=_log_int(rng, 1 << 18, 1 << 23),
                    queries=rng.randint(1, 48))
    return dict(kind=kind, plan_rows=_log_int(rng, 64, 4096), train_rows=_log_int(rng, 32, 512))


# ------------------------------------------------------------------ inputs
def _values(seed, n, b, base, order="uniform", swapped=0.0):
    """n column values on the GPU as int32 tensors of uint32 bits."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if b < 32:
        v = torch.randint(0, 1 << b, (n,), generator=g, device="cuda", dtype=torch.int32 if b < 31 else torch.int64)
    else:
        v = torch.randint(-(1 << 31), 1 << 31, (n,), generator=g, device="cuda", dtype=torch.int64)
        if order == "sorted":
            v += 1 << 31
    if order == "sorted":
        v = torch.sort(v).values
        if swapped > 0.0:
            idx = torch.nonzero(torch.rand(n, generator=g, device="cuda") < swapped).squeeze(1)
            v[idx] = v[idx[torch.randperm(idx.numel(), generator=g, device="cuda")]]
    if base:
        v = v + base
    if v.dtype == torch.int64:
        v = torch.where(v >= (1 << 31), v - (1 << 32), v).to(torch.int32)
    return v


def _wide(v):
    return v.to(torch.int64) & 0xFFFFFFFF


def _range(rng, b, sigma, base):
    """[lo, hi) with target selectivity sigma on uniform values."""
    d = 1 << b
    w = max(1, min(d, round(sigma * d)))
    lo = rng.randint(0, d - w)
    return base + lo, base + lo + w


def _share(b, sigma):
    """The part of the domain that _range selects."""
    return max(1, min(1 << b, round(sigma * (1 << b)))) / (1 << b)


def _select_room(case):
    """Positions a program makes room for: the expected matches and some more."""
    return min(case["n"], int(1.05 * case["n"] * _share(case["b"], case["sigma"])) + 4096)


def _column(values, n, b, base, layout="lanes", zones=False):
    col = gbscan.Column.from_device(values, n, b, base, layout=layout)
    if zones:
        col.zonemap_build()
    return col


def _is_zoned(case):
    return case["strategy"] not in ("branchfree", "branchy")


def _scan_inputs(case, seed):
    rng = random.Random(seed)
    v = _values(seed, case["n"], case["b"], case["base"], case["order"], case.get("swapped", 0.0))
    return v, _range(rng, case["b"], case["sigma"], case["base"])


def _conj_inputs(case, seed):
    rng = random.Random(seed)
    widths = [int(x) for x in case["widths"].split(",")]
    vals = [_values(seed * 31 + i, case["n"], b, 0) for i, b in enumerate(widths)]
    preds = [_range(rng, b, case["sigma"], 0) for b in widths]
    agg = _values(seed * 31 + 30, case["n"], case["agg"], 0) if case["agg"] else None
    return widths, vals, preds, agg


def _batch_spec(case, seed):
    """Lengths log-uniform over [2^10, 2^26], scaled to `total` values in all; b uniform in
    1..32; half the columns sorted with 0, 1% or 10% of the positions displaced."""
    rng = random.Random(seed)
    lens = [math.exp(rng.uniform(math.log(1 << 10), math.log(1 << 26))) for _ in range(case["ncols"])]
    scale = case["total"] / sum(lens)
    spec = []
    for i, x in enumerate(lens):
        b = rng.randint(1, 32)
        is_sorted = rng.random() < 0.5
        swapped = rng.choice([0.0, 0.01, 0.1])
        sigma = math.exp(rng.uniform(math.log(1e-4), 0.0))
        spec.append((max(1, int(x * scale)), b, is_sorted, swapped, _range(rng, b, sigma, 0)))
    return spec


def _serve_inputs(case, seed):
    rng = random.Random(seed)
    table = []
    for c in range(case["columns"]):
        b = SERVE_WIDTHS[c % len(SERVE_WIDTHS)]
        table.append((b, "sorted" if c % 2 == 0 else "uniform", seed * 31 + c))
    sizes = random.Random(case["queries"])
    queries = []
    for _ in range(case["queries"]):
        ids = rng.sample(range(case["columns"]), sizes.randint(1, min(8, case["columns"])))
        preds = [_range(rng, table[c][0], math.exp(rng.uniform(math.log(1e-4), 0.0)), 0) for c in ids]
        queries.append((ids, preds))
    return table, queries


def _planner_inputs(case, seed):
    rng = np.random.default_rng(seed)
    fan = [(4, 64), (64, 64), (64, 4)]
    params = []
    for fi, fo in fan:
        lim = math.sqrt(6.0 / fi)
        params.append(rng.uniform(-lim, lim, fi * fo).astype(np.float32))
        params.append(rng.uniform(-0.1, 0.1, fo).astype(np.float32))
    plan = rng.uniform(0.0, 1.0, (case["plan_rows"], 4)).astype(np.float32)
    x = rng.uniform(0.0, 1.0, (case["train_rows"], 4)).astype(np.float32)
    t = rng.normal(-2.0, 2.0, (case["train_rows"], 4)).astype(np.float32)   # log milliseconds
    return np.concatenate(params), plan, x, t


class _DeviceArray:
    """Device memory of a column as a tensor source; holds the column while a tensor uses it."""

    def __init__(self, column, ptr, shape, typestr):
        self.column = column
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "typestr": typestr, "version": 2}


# ----------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind, "case": case}
    if kind == "scan":
        v, (lo, hi) = _scan_inputs(case, seed)
        state["column"] = _column(v, case["n"], case["b"], case["base"], case["layout"], _is_zoned(case))
        state.update(lo=lo, hi=hi, strategy=case["strategy"], host=case["host"])
        if case["strategy"] == "auto":   # the first such call copies the zone map to the host, once per column
            state["column"].run(lo, hi, "auto")
        if not case["host"]:
            state["out"] = torch.zeros(4, dtype=torch.int64, device="cuda")
    elif kind == "select":
        v, (lo, hi) = _scan_inputs(dict(case, order="uniform"), seed)
        state["column"] = _column(v, case["n"], case["b"], case["base"])
        state.update(lo=lo, hi=hi, strategy=case["strategy"],
                     positions=torch.zeros(_select_room(case), dtype=torch.int32, device="cuda"),
                     count=torch.zeros(1, dtype=torch.int64, device="cuda"))
    elif kind == "conj":
        widths, vals, preds, agg = _conj_inputs(case, seed)
        cols = [_column(v, case["n"], b, 0) for v, b in zip(vals, widths)]
        agg_col = _column(agg, case["n"], case["agg"], 0) if agg is not None else None
        state["query"] = gbscan.Conj(cols, preds, agg_col)
        state["out"] = torch.zeros(4, dtype=torch.int64, device="cuda")
    elif kind == "load":
        state["values"] = _values(seed, case["n"], case["b"], case["base"], case["order"])
        state["packed"] = torch.zeros(gbscan.scan_packed_words(case["n"], case["b"]), dtype=torch.int32, device="cuda")
    elif kind == "batch":
        cols, strategies, preds = [], [], []
        for i, (n, b, is_sorted, swapped, pred) in enumerate(_batch_spec(case, seed)):
            v = _values(seed * 4099 + i, n, b, 0, "sorted" if is_sorted else "uniform", swapped)
            cols.append(_column(v, n, b, 0, zones=is_sorted))
            strategies.append("zone_bf" if is_sorted else "branchfree")
            preds.append(pred)
        state["batch"] = gbscan.Batch(cols, strategies)
        state["preds"] = gbscan.Batch.pred_array(preds)
        state["out"] = torch.zeros((len(cols), 4), dtype=torch.int64, device="cuda")
        state["batch"].run(state["preds"], dev_out=state["out"], host=False)   # records the plan's graph
    elif kind == "serve":
        table, queries = _serve_inputs(case, seed)
        cols = [_column(_values(s, case["n"], b, 0, order), case["n"], b, 0, zones=True) for b, order, s in table]
        state["server"] = gbscan.Server(cols, slots=4, device_bytes_per_slot=112 * 512)
        state["queries"] = queries
    elif kind == "planner":
        params, plan, x, t = _planner_inputs(case, seed)
        state["net"] = gbscan.Planner(4, seed=1)
        state["net"].set_params(params)
        state["plan"], state["x"], state["t"] = (torch.from_numpy(a).cuda() for a in (plan, x, t))
        state["y"] = torch.zeros((case["plan_rows"], 4), dtype=torch.float32, device="cuda")
        state["grads"] = torch.zeros(params.size, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    return state


# --------------------------------------------------------------------- run
def run(state):
    kind = state["kind"]
    if kind == "scan":
        if state["host"]:
            r = state["column"].run(state["lo"], state["hi"], state["strategy"])
            return [int(r.count), int(r.sum), int(r.blocks_scanned)]
        state["column"].run_async(state["lo"], state["hi"], state["out"], state["strategy"])
        return state["out"]
    if kind == "select":
        state["column"].select_async(state["lo"], state["hi"], state["positions"], state["count"], state["strategy"])
        return [state["count"], state["positions"]]
    if kind == "conj":
        state["query"].run_async(state["out"])
        return state["out"]
    if kind == "load":
        case = state["case"]
        gbscan.scan_encode_device(state["values"], case["n"], case["b"], case["base"], state["packed"])
        col = gbscan.Column.from_packed(state["packed"], case["n"], case["b"], case["base"])
        col.zonemap_build()
        blocks = (case["n"] + 1023) // 1024
        zones = torch.as_tensor(_DeviceArray(col, col.zonemap_ptr(), (blocks, 2), "<i4"), device="cuda")
        sums = torch.as_tensor(_DeviceArray(col, col.dev_blocksums, (blocks,), "<i8"), device="cuda")
        return [state["packed"], zones, sums]
    if kind == "batch":
        state["batch"].run(state["preds"], dev_out=state["out"], host=False)
        return state["out"]
    if kind == "serve":
        server, queries = state["server"], state["queries"]
        results = []
        for query_id, (ids, _) in zip(server.submit_many(queries), queries):
            _, rows, _ = server.poll(query_id, len(ids), wait=True)
            results += [(r.count, r.sum, r.blocks_scanned) for r in rows]
        return np.array(results, dtype=np.int64)
    net = state["net"]
    net.forward(state["plan"], state["plan"].shape[0], state["y"])
    loss = net.gradients(state["x"], state["t"], state["x"].shape[0], state["grads"])
    return {"y": state["y"], "loss": np.float32(loss), "grads": state["grads"]}


# -------------------------------------------------------------------- work
def _blocks(n):
    return (n + 1023) // 1024


def work(case):
    kind = case["kind"]
    if kind == "scan":
        data = _blocks(case["n"]) * 128 * case["b"]
        if _is_zoned(case) and not case.get("swapped"):   # sorted: the zone map and the blocks in the range
            data = min(data, _blocks(case["n"]) * 8 + int(data * case["sigma"]))
        return {"bytes": data + 32, "flops": 0}
    if kind == "select":
        return {"bytes": _blocks(case["n"]) * 128 * case["b"] + 4 * int(case["n"] * _share(case["b"], case["sigma"])) + 8, "flops": 0}
    if kind == "conj":
        widths = [int(x) for x in case["widths"].split(",")] + ([case["agg"]] if case["agg"] else [])
        return {"bytes": _blocks(case["n"]) * 128 * sum(widths) + 32, "flops": 0}
    if kind == "load":   # values in; packed words, (min, max) and sum of every block out
        return {"bytes": 4 * case["n"] + _blocks(case["n"]) * (128 * case["b"] + 16), "flops": 0}
    if kind == "batch":
        total = 0
        for n, b, is_sorted, _, _ in _batch_spec(case, 0):
            total += _blocks(n) * (128 * b // (2 if is_sorted else 1)) + 32
        return {"bytes": total, "flops": 0}
    if kind == "serve":
        table, queries = _serve_inputs(case, 0)
        total = 0
        for ids, preds in queries:
            for c, (lo, hi) in zip(ids, preds):
                b, order, _ = table[c]
                part = (hi - lo) / (1 << b) if order == "sorted" else 1.0
                total += int(_blocks(case["n"]) * 128 * b * part) + 32
        return {"bytes": total, "flops": 0}
    weights = 4 * 64 + 64 * 64 + 64 * 4
    rows = case["plan_rows"] + 3 * case["train_rows"]
    floats = 8 * case["plan_rows"] + 8 * case["train_rows"] + 2 * (weights + 132)
    return {"bytes": 4 * floats, "flops": 2 * weights * rows}


# ------------------------------------------------------------------- exact
def _count_sum(wide, lo, hi):
    hit = wide[(wide >= lo) & (wide < hi)]
    return int(hit.numel()), int(hit.sum())


def _zones(wide):
    """Per-block minima, maxima and sums."""
    n = wide.numel()
    full = n // 1024 * 1024
    parts = [wide[:full].view(-1, 1024)] if full else []
    mins, maxs, sums = ([f(p) for p in parts] for f in (lambda p: p.amin(1), lambda p: p.amax(1), lambda p: p.sum(1)))
    if n > full:
        tail = wide[full:]
        mins.append(tail.min().view(1))
        maxs.append(tail.max().view(1))
        sums.append(tail.sum().view(1))
    return torch.cat(mins), torch.cat(maxs), torch.cat(sums)


def _scan_row(wide, lo, hi, b, strategy):
    """(count, sum, blocks read) of one scan by the documented rules of its strategy."""
    blocks = _blocks(wide.numel())
    if strategy not in ("branchfree", "branchy"):
        mins, maxs, _ = _zones(wide)
        keep = (maxs >= lo) & (mins < hi)
        if strategy.startswith("zone_agg"):
            keep &= ~((mins >= lo) & (maxs < hi))
        kept = int(keep.sum())
        dense = math.ceil(min(0.9, (128.0 * b - 8.0) / (128.0 * b + 8.0)) * blocks)
        if strategy != "auto" or kept < dense:
            blocks = kept
    return [*_count_sum(wide, lo, hi), blocks]


def exact(case, seed):
    kind = case["kind"]
    if kind == "scan":
        v, (lo, hi) = _scan_inputs(case, seed)
        row = _scan_row(_wide(v), lo, hi, case["b"], case["strategy"])
        return row if case["host"] else torch.tensor(row + [0])
    if kind == "select":
        v, (lo, hi) = _scan_inputs(dict(case, order="uniform"), seed)
        wide = _wide(v)
        hits = torch.nonzero((wide >= lo) & (wide < hi)).squeeze(1).to(torch.int32)
        pos = torch.zeros(_select_room(case), dtype=torch.int32, device="cuda")   # the rest stays as it was
        pos[:hits.numel()] = hits[:pos.numel()]
        return [torch.tensor([hits.numel()]), pos]
    if kind == "conj":
        _, vals, preds, agg = _conj_inputs(case, seed)
        hit = torch.ones(case["n"], dtype=torch.bool, device="cuda")
        for v, (lo, hi) in zip(vals, preds):
            wide = _wide(v)
            hit &= (wide >= lo) & (wide < hi)
        total = int(_wide(agg)[hit].sum()) if agg is not None else 0
        full = case["n"] // 1024 * 1024
        # blocks read of the summed column: those with a selected row (none without such a column)
        used = int(hit[:full].view(-1, 1024).any(1).sum()) + int(hit[full:].any()) if agg is not None else 0
        return torch.tensor([int(hit.sum()), total, used, 0])
    if kind == "load":
        mins, maxs, sums = _zones(_wide(_values(seed, case["n"], case["b"], case["base"], case["order"])))
        zones = torch.stack([mins, maxs], 1)
        zones = torch.where(zones >= (1 << 31), zones - (1 << 32), zones).to(torch.int32)
        return [None, zones, sums]
    if kind == "batch":
        rows = []
        for i, (n, b, is_sorted, swapped, (lo, hi)) in enumerate(_batch_spec(case, seed)):
            v = _values(seed * 4099 + i, n, b, 0, "sorted" if is_sorted else "uniform", swapped)
            rows.append(_scan_row(_wide(v), lo, hi, b, "zone_bf" if is_sorted else "branchfree") + [0])
        return torch.tensor(rows)
    if kind == "serve":
        table, queries = _serve_inputs(case, seed)
        wide = [_wide(_values(s, case["n"], b, 0, order)) for b, order, s in table]
        rows = [_scan_row(wide[c], lo, hi, table[c][0], "zone_bf") for ids, preds in queries
                for c, (lo, hi) in zip(ids, preds)]
        return np.array(rows, dtype=np.int64)
    params, plan, x, t = _planner_inputs(case, seed)
    p = torch.from_numpy(params).double().requires_grad_(True)
    parts, at = [], 0
    for fi, fo in [(4, 64), (64, 64), (64, 4)]:
        parts.append((p[at:at + fi * fo].view(fi, fo), p[at + fi * fo:at + fi * fo + fo]))
        at += fi * fo + fo

    def net(rows):
        h = rows
        for i, (w, c) in enumerate(parts):
            h = h @ w + c
            h = torch.relu(h) if i < 2 else h
        return h

    y = net(torch.from_numpy(plan).double())
    loss = ((net(torch.from_numpy(x).double()) - torch.from_numpy(t).double()) ** 2).mean()
    loss.backward()
    return {"y": y.detach(), "loss": np.float64(loss.item()), "grads": p.grad}
