"""What is measured: batches of design points simulated through the public binding.

A user of this framework builds a tile graph, uploads it and a table of hardware rows, and simulates the table,
call after call: one row while a model is being set up, a few dozen to a few thousand in a sweep, makespans alone
for a search, busy cycles for a utilisation study, the whole trace for a timeline.  Every case below is one such
call (or, for the last, the upload that comes before it).  The graphs are the shapes this repository generates
(its workloads, profiling-size cases and studies); the rows are drawn over the axes those workloads sweep.
"""
import functools

import numpy as np
import torch

from paper_2607_11262_gb300 import clusters, gts, l2gemm, pipelines
from paper_2607_11262_gb300 import workloads as W

TRACE, DIGEST, CTA_SM, BUSY = gts.GTS_FULL_TRACE, gts.GTS_WANT_DIGEST, gts.GTS_WANT_CTA_SM, gts.GTS_WANT_BUSY
ALL = TRACE | DIGEST | CTA_SM | BUSY

AX_MMA_LAT = (W.P_MMA_LAT, 16, 64)
AXES = {
    "gemm": [W.AX_SMS, W.AX_HBM, AX_MMA_LAT],
    "ws_gemm": [W.AX_SMS, W.AX_HBM, W.AX_TMA_LAT, W.AX_MMA_RATE],
    "attention": [W.AX_SMS, W.AX_HBM, W.AX_TMA_LAT, W.AX_MMA_RATE, W.AX_ALU_RATE],
    "decoder": [W.AX_SMS, W.AX_HBM, W.AX_TMA_LAT, W.AX_MMA_RATE, W.AX_ALU_RATE],
}


def listed():
    return [
        # one row of the smallest workload, makespan only, buffers allocated by the call: a model being set up, or
        # one step of a search that looks at a single candidate
        {"name": "gemm_one_row", "graph": "gemm", "tiles": 16, "ksteps": 8, "points": 1, "flags": 0, "fresh": True},
        # the whole small sweep with every output, as the named workload and the tests run it
        {"name": "gemm_sweep", "graph": "gemm", "tiles": 16, "ksteps": 8, "points": 64, "flags": ALL, "fresh": False},
        # the benchmark's kernel shape at its profiling size, a ragged number of rows, whole trace
        {"name": "ws_gemm_trace", "graph": "ws_gemm", "m": 2048, "n": 2048, "k": 1024, "points": 1500,
         "flags": TRACE, "fresh": False},
        # a larger GEMM, makespan and utilisation only: the widest sweep, more rows than fit the GPU at once
        {"name": "ws_gemm_wide", "graph": "ws_gemm", "m": 4096, "n": 4096, "k": 2048, "points": 3000,
         "flags": BUSY, "fresh": False},
        # attention forward with the ping-pong ordering edges, whole trace: a timeline of each row
        {"name": "attention_trace", "graph": "attention", "heads": 16, "seq": 2048, "points": 257,
         "flags": TRACE | DIGEST, "fresh": False},
        # nine gated kernels of a decoder layer, CTA placement and busy cycles
        {"name": "decoder_layer", "graph": "decoder", "hidden": 1024, "ffn": 2816, "tokens": 2048, "points": 300,
         "flags": CTA_SM | BUSY, "fresh": False},
        # random layered DAGs, one row each: edges between CTAs, nodes in no CTA order
        {"name": "random_dags", "graph": "dags", "instances": 48, "nodes": 9000, "points": 48, "flags": TRACE | DIGEST,
         "fresh": False},
        # issue-policy study: the same rows under lowest-id, greedy-then-oldest and round-robin with 1, 2 and 4
        # schedulers per SM, makespans only
        {"name": "issue_policies", "graph": "ws_gemm", "m": 2048, "n": 1024, "k": 1024, "points": 448, "flags": 0,
         "policies": True, "fresh": False},
        # on-chip network against DRAM exchanges, clusters of 2-16 CTAs, busy cycles and the schedules' digests
        {"name": "noc_fusion", "graph": "clusters", "points": 64, "flags": BUSY | DIGEST, "fresh": False},
        # L2 capacity study: two tile orders, six capacities, busy cycles (which hold the hit counts) and digests
        {"name": "l2_capacity", "graph": "l2", "m": 2048, "n": 2048, "k": 2048, "points": 96, "flags": BUSY | DIGEST,
         "fresh": False},
        # software-pipelining study: 96 single-SM graphs in one stack, several rows per graph
        {"name": "pipelines_one_sm", "graph": "pipelines", "points": 1536, "flags": BUSY | DIGEST, "fresh": False},
        # a graph and a table of rows taken from host memory to the device, checked and packed: paid once per graph
        {"name": "load_graph", "graph": "attention", "heads": 16, "seq": 4096, "points": 1000, "flags": 0,
         "load": True, "fresh": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(2 ** rng.uniform(np.log2(lo), np.log2(hi))))


def draw(rng):
    kind = rng.choice(["gemm", "ws_gemm", "ws_gemm", "attention", "decoder", "dags", "clusters", "l2", "pipelines"])
    flags = rng.choice([0, BUSY, TRACE, TRACE | DIGEST, ALL])
    if kind in ("clusters", "pipelines"):  # graphs of several sizes in one stack: trace rows of the smaller ones end early
        flags = rng.choice([0, BUSY, BUSY | DIGEST])
    c = {"graph": kind, "flags": flags, "fresh": rng.random() < 0.3}
    if kind == "gemm":
        c.update(tiles=_log_int(rng, 4, 200), ksteps=_log_int(rng, 2, 24), points=_log_int(rng, 1, 900))
    elif kind == "ws_gemm":
        c.update(m=128 * _log_int(rng, 4, 24), n=256 * _log_int(rng, 2, 12), k=64 * _log_int(rng, 4, 24),
                 points=_log_int(rng, 1, 2500), policies=rng.random() < 0.25)
        if c["policies"]:
            c["points"] = 7 * max(1, c["points"] // 21)
    elif kind == "attention":
        c.update(heads=_log_int(rng, 2, 16), seq=128 * _log_int(rng, 2, 16), points=_log_int(rng, 1, 500),
                 load=rng.random() < 0.2)
    elif kind == "decoder":
        c.update(hidden=256 * rng.randint(1, 4), ffn=256 * rng.randint(2, 11), tokens=512 * rng.randint(1, 4),
                 points=_log_int(rng, 1, 300))
    elif kind == "dags":
        k = _log_int(rng, 1, 48)
        c.update(instances=k, nodes=_log_int(rng, 500, 9000), points=k)
    elif kind == "clusters":
        c.update(points=8 * _log_int(rng, 1, 12))
    elif kind == "l2":
        c.update(m=1024 * rng.randint(1, 2), n=1024 * rng.randint(1, 2), k=64 * rng.randint(4, 32),
                 points=12 * _log_int(rng, 1, 8))
    else:
        c.update(points=96 * _log_int(rng, 1, 20))
    return c


@functools.lru_cache(maxsize=4)
def _fixed_graph(key):
    """Host-side graphs that do not depend on the seed (the graph of a sweep is the model, not the data)."""
    c = dict(key)
    if c["graph"] == "gemm":
        tpl = W.gemm_2stage_cta(ksteps=c["ksteps"])
        return W.assemble("gemm", 4, [tpl], np.zeros(c["tiles"], np.int64), np.zeros(c["tiles"], np.uint32))
    if c["graph"] == "ws_gemm":
        return W.ws_gemm(c["m"], c["n"], c["k"], 132, "ws_gemm")
    if c["graph"] == "attention":
        return W.fa_fwd(batch=1, heads=c["heads"], seq=c["seq"])
    if c["graph"] == "decoder":
        return W.decoder_layer(hidden=c["hidden"], heads=c["hidden"] // 128, ffn=c["ffn"], tokens=c["tokens"], seq=512)
    if c["graph"] == "clusters":
        return clusters.study_set()[0]
    if c["graph"] == "l2":
        return l2gemm.study_set(M=c["m"], N=c["n"], K=c["k"])[0]
    return pipelines.study_set()[0]


SIZES = ("graph", "tiles", "ksteps", "m", "n", "k", "heads", "seq", "hidden", "ffn", "tokens")


def _graph(case, seed):
    if case["graph"] == "dags":
        return W.stress_set(case["instances"], n_nodes=case["nodes"], seed0=26_000_000 + 1000 * (seed % 1_000_000))
    return _fixed_graph(tuple((k, case[k]) for k in SIZES if k in case))


def _rows(case, graph, seed):
    """The design points: every axis the workload sweeps is drawn anew from the seed."""
    kind, n = case["graph"], case["points"]
    if kind == "dags":
        return W.stress_params(n)
    if kind in ("clusters", "l2", "pipelines"):  # the studies' first row of a group is their fixed default: drawn ones only
        groups = {"clusters": 8, "l2": 12, "pipelines": 96}[kind]
        if kind == "clusters":
            rows = clusters.study_params(clusters.study_cases(), points_per_graph=n // groups + 1, seed=seed)
        elif kind == "l2":
            rows = l2gemm.study_params(2, points_per_capacity=n // groups + 1, seed=seed)
        else:
            rows = pipelines.study_params(graph.n_graphs, n // groups + 1, seed=seed)
        return np.ascontiguousarray(rows.reshape(groups, -1, W.NPARAM)[:, 1:].reshape(-1, W.NPARAM))
    if not case.get("policies"):
        return W.sweep_params(seed, n, AXES[kind], 2 if kind == "gemm" else 1)
    base = W.sweep_params(seed, n // 7, AXES[kind], 1)
    variants = [base]
    for policy in (W.POLICY_GTO, W.POLICY_RR):
        for schedulers in (1, 2, 4):
            p = base.copy()
            p[:, W.P_ISSUE_POLICY], p[:, W.P_SUBPARTITIONS] = policy, schedulers
            variants.append(p)
    return np.ascontiguousarray(np.concatenate(variants))


def prepare(case, seed):
    graph = _graph(case, seed)
    rows = _rows(case, graph, seed)
    state = {"case": case, "graph": graph, "rows": rows}
    if case.get("load"):  # host data is what such a call starts from
        return state
    state["dg"] = gts.DeviceGraph(graph)
    state["dp"] = gts.DeviceParams(state["dg"], rows)
    if not case["fresh"]:  # a sweep keeps its buffers between calls
        state["out"] = gts.alloc_outputs(state["dg"], case["points"], case["flags"])
        state["scratch"] = gts.alloc_scratch(state["dg"], state["dp"], case["flags"])
    return state


def _present(out):
    named = (("makespan", out.makespan), ("status", out.status), ("start", out.start), ("finish", out.finish),
             ("digest", out.digest), ("cta_sm", out.cta_sm), ("busy", out.busy))
    return {k: v for k, v in named if v is not None}


def run(state):
    case = state["case"]
    if case.get("load"):
        dg = gts.DeviceGraph(state["graph"])
        dp = gts.DeviceParams(dg, state["rows"])
        return {"packed": dg.workspace, "order": dp.order}
    if case["fresh"]:
        return _present(gts.simulate(state["dg"], state["dp"], flags=case["flags"]))
    return _present(gts.simulate(state["dg"], state["dp"], flags=case["flags"] | gts.GTS_SCRATCH_CLEAN,
                                 out=state["out"], scratch=state["scratch"]))


@functools.lru_cache(maxsize=32)
def _sizes(key):
    c = dict(key)
    if c["graph"] == "dags":
        return None
    g = _fixed_graph(tuple((k, c[k]) for k in SIZES if k in c))
    return g.n_nodes, g.n_edges, g.n_ctas, np.diff(g.node_off.astype(np.int64)).tolist()


def work(case):
    points = case["points"]
    if case["graph"] == "dags":
        n = case["instances"] * case["nodes"]
        m, ctas, node_points = 5 * n // 2, 8, n
    else:
        n, m, ctas, each = _sizes(tuple((k, case[k]) for k in SIZES if k in case))
        node_points = sum(each) * points // len(each)
    graph_bytes = n * 17 + (n + 1) * 4 + m * 5
    if case.get("load"):  # the logical graph in, the packed graph and the row order out
        return {"bytes": graph_bytes + 32 * n + 8 * m + 132 * points, "flops": 0}
    b = graph_bytes + 128 * points + 8 * points
    if case["flags"] & TRACE:
        b += 8 * node_points
    if case["flags"] & DIGEST:
        b += 8 * points
    if case["flags"] & CTA_SM:
        b += 4 * ctas * points
    if case["flags"] & BUSY:
        b += 8 * gts.GTS_BUSY_CLASSES * points
    # each node-point costs at least one selection, its latency and the release of its successors: some 16 integer
    # operations and 4 per edge
    return {"bytes": b, "flops": 16 * node_points + 4 * node_points * m // max(n, 1)}


def tolerance(case):
    return "exact"  # integer cycles, ids and counts


# ---------------------------------------------------------------- the model in plain Python
_UNIT = {W.LOAD: (1, 4), W.SMEM: (2, 6), W.MMA: (0, 8), W.EW: (3, 10), W.STORE: (1, 4), W.BAR: (4, None)}  # class, rate
_BASE = {W.LOAD: (5, 3), W.SMEM: (7,), W.MMA: (9,), W.EW: (11,), W.STORE: (5,), W.BAR: (12,), W.NOP: ()}


def _simulate_one(g, row):
    """One row under the lowest-id order: at each cycle CTAs launch, then the lowest issuable head issues, one at a
    time, until none is left; then time moves to the next release, free server or retirement."""
    row = [int(x) for x in row]
    n, wpc, ncta = g.n_nodes, g.warps_per_cta, g.n_ctas
    typ, wrk, ext, cta, warp = (getattr(g, k).tolist() for k in ("type", "work", "lat_extra", "cta", "warp"))
    ptr, col, kind, kern = g.row_ptr.tolist(), g.col.tolist(), g.ekind.tolist(), g.cta_kernel.tolist()
    streams = {}
    for v in range(n):
        streams.setdefault((cta[v], warp[v]), []).append(v)
    pend = [0] * n
    for w in col:
        pend[w] += 1
    ready, start, finish = [0] * n, [0] * n, [0] * n
    left = [0] * ncta
    for c in cta:
        left[c] += 1
    end = [0] * ncta
    slots = [None] * min(row[0] * row[1], ncta)
    free = [[[0] * row[13 + r] for r in range(5)] for _ in range(row[0])]
    hbm = [0] * row[18]
    busy = [0] * 9
    place = [-1] * ncta
    at = {}
    t = issued = nxt = 0
    ceil = lambda a, b: -(-a // b)  # noqa: E731
    while True:
        while True:  # retire, launch
            for j, c in enumerate(slots):
                if c is not None and left[c] == 0 and end[c] <= t:
                    slots[j] = None
            gaps = [j for j, c in enumerate(slots) if c is None]
            if nxt >= ncta or not gaps or any(c is not None and kern[c] < kern[nxt] for c in slots):
                break
            slots[gaps[0]] = nxt
            place[nxt] = gaps[0] // row[1]
            for w in range(wpc):
                if (nxt, w) in streams:
                    at[(nxt, w)] = 0
            nxt += 1
        if issued == n:
            break
        best, later = None, []
        for key, i in at.items():
            v = streams[key][i]
            if pend[v]:
                continue
            need = ready[v]
            if typ[v] in _UNIT:
                need = max(need, min(free[place[key[0]]][_UNIT[typ[v]][0]]))
            if typ[v] in (W.LOAD, W.STORE):
                need = max(need, min(hbm))
            if need > t:
                later.append(need)
            elif best is None or v < best[0]:
                best = (v, key)
        if best is None:
            later += [end[c] for c in slots if c is not None and left[c] == 0]
            t = min(later)
            continue
        v, key = best
        lat = sum(row[i] for i in _BASE[typ[v]]) + ext[v]
        held = 0
        if typ[v] in _UNIT:
            cls, rate = _UNIT[typ[v]]
            held = ceil(wrk[v], row[rate]) if rate is not None else 1
            pool = free[place[key[0]]][cls]
            pool[pool.index(min(pool))] = t + held
            busy[cls] += held
        if typ[v] in (W.LOAD, W.STORE):
            over = ceil(wrk[v], row[2])
            hbm[hbm.index(min(hbm))] = t + over
            busy[5] += over
            held = max(held, over)
        start[v], finish[v] = t, t + lat + held
        for e in range(ptr[v], ptr[v + 1]):
            pend[col[e]] -= 1
            ready[col[e]] = max(ready[col[e]], t if kind[e] else finish[v])
        at[key] += 1
        if at[key] == len(streams[key]):
            del at[key]
        left[key[0]] -= 1
        end[key[0]] = max(end[key[0]], finish[v])
        issued += 1
    return start, finish, place, busy


def _mix(z):
    m = (1 << 64) - 1
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9 & m
    z = (z ^ (z >> 27)) * 0x94D049BB133111EB & m
    return z ^ (z >> 31)


def exact(case, seed):
    """The same outputs from the plain model; None where it would take too long or the rows use an extension."""
    if case["graph"] != "gemm" or case.get("policies"):
        return None
    if case["tiles"] * case["ksteps"] * 17 * case["points"] * min(case["tiles"], 264) > 2.5e6:
        return None
    g = _graph(case, seed)
    rows = _rows(case, g, seed)
    cols = {k: [] for k in ("makespan", "status", "start", "finish", "digest", "cta_sm", "busy")}
    for row in rows:
        start, finish, place, busy = _simulate_one(g, row)
        total = sum(_mix((v << 32 | s) ^ (f * 0x9E3779B97F4A7C15 & ((1 << 64) - 1)))
                    for v, (s, f) in enumerate(zip(start, finish))) & ((1 << 64) - 1)
        for k, x in zip(cols, (max(finish), 0, start, finish, total - (1 << 64) if total >> 63 else total, place, busy)):
            cols[k].append(x)
    keep = ["makespan", "status"] + [k for k, f in (("start", TRACE), ("finish", TRACE), ("digest", DIGEST),
                                                    ("cta_sm", CTA_SM), ("busy", BUSY)) if case["flags"] & f]
    wide = ("digest", "busy")
    return {k: torch.tensor(cols[k], dtype=torch.int64 if k in wide else torch.int32) for k in keep}
