"""What a scheduler has this library do: evaluate candidate placements of an
operator graph, by full simulation or as moves against a base placement, with
pure-latency or arbitrated transfers; run a scheduling round; refit the
estimators.

A case of the simulation paths is a graph (prefill or decode requests with the
layer structure of ``paper_2608_15762_gb300.workloads``), a set of accelerators
and a number of candidates; one pass evaluates every candidate and selects the
best.  All its results are whole numbers (microseconds, bytes, counts) and are
compared bit for bit.  The estimator cases return fitted coefficients in 64
bits and the whole numbers derived from them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_15762_gb300 import gmgsim as G
from paper_2608_15762_gb300 import workloads as W

MiB = W.MiB
# Gaps of an online request between its segments (idle slices: median 2.55 s,
# p90 10.9 s, between 10 ms and 20 s).
GAP_SIGMA = math.log(10.9 / 2.55) / 1.2815515655446004
ACCELERATORS_PER_NODE = 8
KINDS = 14        # template operators: embed, twelve per layer, lm_head
FEATURES = 5      # operator estimator features (the last one constant)
SIM = dict(steps=1, types=1, links="uniform", arrivals_s=0.0, online=False, placement="random", moves=0,
           arbitrated=False, base="none", traced=0, score_mode=0)


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    def sim(name, path, requests, layers, accelerators, candidates, **kw):
        return dict(SIM, name=name, path=path, requests=requests, layers=layers, accelerators=accelerators,
                    candidates=candidates, **kw)
    return [
        # the smallest call: one short request on two accelerators, where
        # launches and one simulation's latency count
        sim("tiny", "batch", 1, 4, 2, 256),
        # a round of incremental scheduling: collect a batch, evaluate it on
        # every accelerator partition, commit the best
        sim("round", "round", 8, 32, 8, 14),
        # the ordinary call: a batch of prefill requests on one node
        sim("prefill", "batch", 8, 32, 8, 4096),
        # contiguous per-request stages on two nodes of two accelerator
        # generations, odd sizes, per-operator schedules of a few candidates
        # kept, deadlines before completion times
        sim("stages_two_types", "batch", 7, 27, 16, 1501, types=2, links="nodes", placement="stages", traced=3,
            score_mode=1),
        # decode with growing KV tensors and a capacity that binds
        sim("decode", "batch", 8, 32, 8, 2048, steps=16),
        # offline work moved into the idle slices of online requests, from a
        # base taken for this decision
        sim("moves", "moves", 32, 32, 16, 4096, online=True, moves=16, base="new"),
        # many tenants of mixed depth on 256 accelerators, the largest call
        sim("wide", "batch", 128, 0, 256, 4096, arrivals_s=0.75),
        # the same service, moves against its base
        sim("wide_moves", "moves", 128, 0, 256, 2048, arrivals_s=0.75, moves=64, base="new"),
        # transfers that wait for endpoints and links
        sim("arbitrated", "batch", 8, 32, 8, 2048, arbitrated=True),
        # the same for moves, resumed from an arbitrated base
        sim("arbitrated_moves", "moves", 16, 32, 16, 2048, online=True, moves=16, base="new", arbitrated=True),
        # arbitrated transfers across eight nodes
        sim("arbitrated_wide", "batch", 32, 16, 64, 1024, links="nodes", arbitrated=True),
        # feedback of the executors into every estimator, then the durations
        # and link tables of the next simulations
        dict(name="estimators", path="estimators", types=2, samples=16384, accelerators=8, link_samples=4096,
             ops=197632),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(["batch"] * 4 + ["moves"] * 3 + ["arbitrated"] * 2 + ["round", "estimators"])
    if path == "estimators":
        return dict(path="estimators", types=rng.randint(1, 2), samples=spread(48, 16384),
                    accelerators=rng.randint(2, 8), link_samples=spread(16, 4096), ops=spread(50, 197632))
    c = dict(SIM, path=path)
    c["arbitrated"] = path == "arbitrated"
    if c["arbitrated"]:
        c["path"] = rng.choice(["batch", "moves"])
    c["accelerators"] = spread(8, 32) if path == "round" else spread(2, 256)
    narrow = c["accelerators"] <= 32
    # operators of the graph and operators over all candidates
    most_ops = 13000 if c["arbitrated"] and narrow else 6500 if c["arbitrated"] or path == "round" else 50000
    most_work = 6e6 if c["arbitrated"] and not narrow else 1.2e7 if c["arbitrated"] else 8e7
    if path != "round" and rng.random() < 0.3:
        c["steps"] = rng.randint(2, 16)
    c["layers"] = rng.randint(2, 80)
    c["requests"] = max(1, min(spread(1, 128), most_ops // (c["steps"] * (12 * c["layers"] + 2))))
    c["steps"] = max(1, min(c["steps"], most_ops // (c["requests"] * (12 * c["layers"] + 2))))
    c["layers"] = max(1, min(c["layers"], (most_ops // (c["requests"] * c["steps"]) - 2) // 12))
    n = c["requests"] * c["steps"] * (12 * c["layers"] + 2)
    c["candidates"] = spread(1, max(1, min(4096, int(most_work / n))))
    if path == "round":
        c["candidates"] = _partitions(c["accelerators"])[0].size - 1
    else:
        c["types"] = 2 if rng.random() < 0.25 else 1
        c["placement"] = rng.choice(["random", "random", "stages"])
        c["traced"] = rng.choice([0, 0, 1])
    c["links"] = rng.choice(["uniform", "uniform", "nodes"])
    # an hour of arrivals needs times beyond 32 bits
    c["arrivals_s"] = rng.choice([0.0, 0.0, 0.75, 3600.0])
    c["score_mode"] = rng.randint(0, 1)
    if c["path"] == "moves":
        c["moves"] = spread(1, 64)
        c["base"] = rng.choice(["new", "kept"])
        c["online"] = c["steps"] == 1 and c["layers"] >= 8 and rng.random() < 0.5
    return c


# ---------------------------------------------------------------------------
# Graphs, placements, moves
# ---------------------------------------------------------------------------

def _templates(case):
    if case["steps"] > 1:
        return [W.decode_template(case["layers"], case["steps"])] * case["requests"]
    depths = (16, 32, 80) if case["layers"] == 0 else (case["layers"],)
    return [W.prefill_template(depths[r % len(depths)]) for r in range(case["requests"])]


def _links(case):
    D = case["accelerators"]
    if case["links"] == "uniform":
        return W.uniform_links(D, 400_000, 10)
    node = np.arange(D) // ACCELERATORS_PER_NODE
    same = (node[:, None] == node[None, :]).reshape(-1)
    return np.where(same, 400_000, 50_000).astype(np.int64), np.where(same, 10, 25).astype(np.int64)


def _graph(case, rng):
    """The graph's description, its request of every op and its first ops."""
    ts = _templates(case)
    D, R = case["accelerators"], case["requests"]
    offs = np.concatenate([[0], np.cumsum([t.n for t in ts])]).astype(np.int64)
    n = int(offs[-1])
    edges = np.concatenate([[0], np.cumsum([t.pred_idx.size for t in ts])])
    pred_off = np.concatenate([[0]] + [t.pred_off[1:] + e for t, e in zip(ts, edges)])
    pred_idx = np.concatenate([t.pred_idx + o for t, o in zip(ts, offs)])
    kind = np.concatenate([t.kind for t in ts])
    step = np.concatenate([t.step for t in ts])
    req = np.repeat(np.arange(R), np.diff(offs)).astype(np.int32)
    dur = W.lognormal_durations(rng, n)
    cap = 80 * W.GiB
    if case["steps"] > 1:
        out_bytes = W.uniform_bytes(rng, n, MiB, 16 * MiB)
        kv0 = rng.integers(1, 5, size=R, dtype=np.int64) * MiB
        kv = kind == W.LAYER_OPS.index("kvw")
        out_bytes[kv] = kv0[req[kv]] * (step[kv] + 1)
        # about a third of random placements of the listed case exceed it
        cap = int(1.92 * case["layers"] * case["steps"] * kv0.sum() / D) + 512 * MiB
    else:
        out_bytes = W.uniform_bytes(rng, n, MiB, 256 * MiB)
    arrival = np.zeros(R, np.int64)
    if case["arrivals_s"]:
        arrival = np.sort(rng.integers(0, int(case["arrivals_s"] * 1e6), size=R))
        arrival[0] = 0
    release = np.zeros(n, np.int64)
    release[offs[:-1]] = arrival
    if case["online"]:
        # the first half of the requests is online: eight layers at a time,
        # each segment released an idle gap after the one before it
        est = W.contention_free_start(pred_off, pred_idx, dur, release)
        for r in range((R + 1) // 2):
            wait = 0
            for l in range(8, ts[r].n // 12, 8):
                first, last = int(offs[r]) + 1 + 12 * l, int(offs[r]) + 12 * l
                gap = int(np.clip(rng.lognormal(math.log(2.55e6), GAP_SIGMA), 1e4, 2e7))
                wait += gap
                release[first] = int(est[last] + dur[last]) + wait
    dl = W.deadlines_from_critical_path(pred_off, pred_idx, dur, release, req, R, arrival,
                                        rng.integers(12, 21, size=R, dtype=np.int64), 10)
    bw, lat = _links(case)
    types = {}
    if case["types"] > 1:
        slower = rng.uniform(1.3, 2.5, size=KINDS)
        types = dict(dev_type=(np.arange(D) * 2 // D).astype(np.uint8),
                     dur_by_type=np.stack([dur, np.maximum(1, np.rint(dur * slower[kind + 2]).astype(np.int64))], 1))
    desc = W.GmgDesc(n_dev=D, pred_off=pred_off, pred_idx=pred_idx, dur=dur, out_bytes=out_bytes, release=release,
                     req_id=req, scored=np.ones(n, np.uint8), deadline=dl, cap=np.full(D, cap, np.int64),
                     base=np.zeros(D, np.int64), avail0=np.zeros(D, np.int64), bw=bw, lat=lat, **types).normalized()
    return desc, kind, offs


def _base_row(desc, offs):
    """Each request's first half on one accelerator, its second half on the next."""
    row = np.zeros(W.placement_ld(desc.n_ops), np.uint8)
    for r in range(offs.size - 1):
        half = int(offs[r] + offs[r + 1]) // 2
        row[offs[r]:half] = 2 * r % desc.n_dev
        row[half:offs[r + 1]] = (2 * r + 1) % desc.n_dev
    return row


def _move_lists(case, rng, desc, row, offs):
    """1 to `moves` ops of the offline requests, each to another accelerator."""
    lo = int(offs[(case["requests"] + 1) // 2]) if case["online"] and case["requests"] > 1 else 0
    n, D = desc.n_ops, desc.n_dev
    lists = [np.unique(rng.integers(lo, n, size=rng.integers(1, case["moves"] + 1))) for _ in range(case["candidates"])]
    ops = np.concatenate(lists)
    to = rng.integers(0, D - 1, size=ops.size)
    to += to >= row[ops]
    return W.Moves(np.concatenate([[0], np.cumsum([x.size for x in lists])]).astype(np.int32), ops.astype(np.int32),
                   to.astype(np.uint8))


def _rows(case, seed, desc, offs, device):
    """Candidate placements, uint8 [candidates, ld]."""
    gen = torch.Generator(device=device).manual_seed(seed)
    K, n, D = case["candidates"], desc.n_ops, desc.n_dev
    rows = torch.zeros((K, W.placement_ld(n)), dtype=torch.uint8, device=device)
    if case["placement"] == "random":
        rows[:, :n] = torch.randint(0, D, (K, n), dtype=torch.uint8, device=device, generator=gen)
        return rows
    # 1, 2, 4 or 8 contiguous stages per request
    for r in range(offs.size - 1):
        a, b = int(offs[r]), int(offs[r + 1])
        stages = 1 << torch.randint(0, 4, (K, 1), device=device, generator=gen)
        stage = torch.arange(b - a, device=device)[None, :] * stages // (b - a)
        acc = torch.randint(0, D, (K, 8), dtype=torch.uint8, device=device, generator=gen)
        rows[:, a:b] = torch.gather(acc, 1, stage)
    return rows


def _partitions(D):
    """Every accelerator, then every aligned group of 2, 4, ...: CSR."""
    groups = [list(range(a, min(D, a + s))) for s in (1, 2, 4) for a in range(0, D, s)]
    return (np.concatenate([[0], np.cumsum([len(x) for x in groups])]).astype(np.int32),
            np.concatenate(groups).astype(np.uint8))


# ---------------------------------------------------------------------------
# What a program has in hand before the call, and the call
# ---------------------------------------------------------------------------

def prepare(case, seed):
    device = torch.device("cuda")
    if case["path"] == "estimators":
        return _prepare_estimators(case, seed, device)
    rng = np.random.default_rng(np.random.SeedSequence([seed, 1]))
    desc, kind, offs = _graph(case, rng)
    g = G.gmg_create(desc, device=device)
    K, R, D, n = case["candidates"], desc.n_req, desc.n_dev, desc.n_ops
    s = {"case": case, "g": g}
    if case["path"] == "round":
        return _prepare_round(case, s, desc, kind, offs, device)
    s["traced"] = None
    if case["traced"]:
        s["traced"] = torch.arange(min(case["traced"], K), dtype=torch.int32, device=device)
    s["out"] = G.SimOut.empty(K, D, R, device, req_done=True, n_trace=0 if s["traced"] is None else s["traced"].numel(),
                              n_ops=n)
    s["scratch"] = G.Scratch(device)
    s["best"] = torch.empty(2, dtype=torch.int64, device=device)
    if case["path"] == "batch":
        s["rows"] = _rows(case, seed, desc, offs, device)
    else:
        row = _base_row(desc, offs)
        s["row"] = torch.from_numpy(row).to(device)
        s["moves"] = G.moves_to_device(_move_lists(case, rng, desc, row, offs), device)
        # more than 32 accelerators take a pure-latency base in both modes
        s["arbitrated_base"] = case["arbitrated"] and D <= 32
        if case["base"] == "kept":
            s["base"] = G.base_create(g, s["row"], arbitrated=s["arbitrated_base"])
    return s


def _prepare_round(case, s, desc, kind, offs, device):
    n, D = desc.n_ops, desc.n_dev
    ld = W.placement_ld(n)
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).to(device)  # noqa: E731
    # the first sixteenth of every request has run, the next few ops are issued
    state = np.zeros(n, np.uint8)
    for r in range(offs.size - 1):
        a, m = int(offs[r]), int(offs[r + 1] - offs[r])
        state[a:a + m // 16] = 2
        state[a + m // 16:a + m // 16 + 3] = 1
    layer = np.concatenate([t.layer for t in _templates(case)])
    last = np.repeat([t.layer.max() for t in _templates(case)], np.diff(offs))
    role = np.clip(layer, 0, None) * 4 // (last + 1)
    role[kind == -2] = 3
    part_off, part_dev = _partitions(D)
    size = np.diff(part_off)
    # one graph template: a quarter of the layers per role, spread over the partition
    mapping = np.stack([q * size // 4 for q in range(4)], axis=1)
    s["state0"], s["place0"] = dev(state, np.uint8), dev(_base_row(desc, offs), np.uint8)
    s["round"] = G.Round(s["g"], s["state0"].clone(), s["place0"].clone(), dev(desc.deadline[desc.req_id], np.int64),
                         dev(np.zeros(n), np.int32), dev(role, np.int32), dev(part_off, np.int32),
                         dev(part_dev, np.uint8), dev(mapping.reshape(-1), np.int32), 4, 128, 64,
                         score_mode=case["score_mode"])
    s["round"].batch.zero_()
    assert s["round"].n_part == case["candidates"] and s["round"].ld == ld
    return s


def _feedback(case, seed, device):
    """Two batches of executor feedback (an earlier, smaller one and the one to
    incorporate) and the ops to predict; true models with measurement noise."""
    gen = torch.Generator(device=device).manual_seed(seed)
    f64 = dict(dtype=torch.float64, device=device)
    uni = lambda *shape: torch.rand(shape, generator=gen, **f64)  # noqa: E731
    E, D = case["types"] * KINDS, case["accelerators"]
    L = D * D
    beta, inv_bw = 1 + 39 * uni(E, FEATURES), 1.0 / (50_000 + 350_000 * uni(L))
    f = {"op": [], "link": []}
    for part in (4, 1):
        per = max(FEATURES + 1, case["samples"] // part)
        x = 10 * uni(E, per, FEATURES)
        x[..., -1] = 1.0
        y = (x * beta[:, None, :]).sum(-1) + 2 * torch.randn((E, per), generator=gen, **f64)
        f["op"].append((per, x.reshape(-1, FEATURES), y.reshape(-1)))
        per = max(4, case["link_samples"] // part)
        size = MiB + 255 * MiB * uni(L, per)
        y = size * inv_bw[:, None] + 10 + 0.5 * torch.randn((L, per), generator=gen, **f64)
        f["link"].append((per, torch.stack([size, torch.ones_like(size)], -1).reshape(-1, 2), y.reshape(-1)))
    kind = torch.randint(0, KINDS, (case["ops"], 1), generator=gen, device=device)
    f["est_of"] = (kind + KINDS * torch.arange(case["types"], device=device)).to(torch.int32).contiguous()
    f["features"] = 10 * uni(case["ops"], FEATURES)
    f["features"][:, -1] = 1.0
    f["default"] = torch.randint(5, 50_000, (case["ops"],), generator=gen, device=device)
    return f


def _prepare_estimators(case, seed, device):
    f = _feedback(case, seed, device)
    D = case["accelerators"]
    s = {"case": case, "in": f, "D": D}
    for name, E, F in (("op", case["types"] * KINDS, FEATURES), ("link", D * D, 2)):
        est = G.Estimators(E, F, device)
        off = [torch.arange(E + 1, dtype=torch.int32, device=device) * per for per, _, _ in f[name]]
        tmp = est.tmp_for(max(y.numel() for _, _, y in f[name]))
        est.update(off[0], f[name][0][1], f[name][0][2], tmp=tmp)
        s[name] = {"est": est, "prior": est.state.clone(), "off": off[1], "x": f[name][1][1], "y": f[name][1][2],
                   "tmp": tmp}
    s["dur"] = torch.empty((case["ops"], case["types"]), dtype=torch.int64, device=device)
    s["bw"] = torch.full((D * D,), 400_000, dtype=torch.int64, device=device)
    s["lat"] = torch.full((D * D,), 10, dtype=torch.int64, device=device)
    return s


def _results(out, best):
    return dict({k: v for k, v in out.__dict__.items() if v is not None}, best=best)


def run(s):
    case = s["case"]
    if case["path"] == "estimators":
        f = s["in"]
        for m in (s["op"], s["link"]):
            m["est"].state.copy_(m["prior"])  # the statistics before this batch
            m["est"].update(m["off"], m["x"], m["y"], tmp=m["tmp"])
        dur = s["op"]["est"].predict_durations(f["est_of"], f["features"], f["default"], out=s["dur"])
        bw, lat = s["link"]["est"].links(s["D"], s["bw"], s["lat"])
        op_beta, op_fitted = s["op"]["est"].coefficients()
        link_beta, link_fitted = s["link"]["est"].coefficients()
        return {"op_beta": op_beta, "op_fitted": op_fitted, "link_beta": link_beta, "link_fitted": link_fitted,
                "dur": dur, "bw": bw, "lat": lat}
    if case["path"] == "round":
        r = s["round"]
        r.state.copy_(s["state0"])  # the schedule as the executors report it
        r.place.copy_(s["place0"])
        r.step()
        return dict(_results(r.out, r.best), info=r.info, batch=r.batch, rows=r.rows, place=r.place, state=r.state)
    if case["path"] == "batch":
        out = G.sim_batch(s["g"], s["rows"], out=s["out"], scratch=s["scratch"], trace_k=s["traced"],
                          arbitrated=case["arbitrated"])
    else:
        base = s.get("base") or G.base_create(s["g"], s["row"], arbitrated=s["arbitrated_base"])
        out = G.sim_incremental(s["g"], base, *s["moves"], out=s["out"], scratch=s["scratch"], trace_k=s["traced"],
                                arbitrated=case["arbitrated"])
    return _results(out, G.select_best(out, score_mode=case["score_mode"], best=s["best"]))


# ---------------------------------------------------------------------------
# What a pass cannot do without, and how its results are compared
# ---------------------------------------------------------------------------

def work(case):
    """Bytes of the inputs read once and the outputs written once.  The
    simulations are integer event processing (no floating-point operations)."""
    if case["path"] == "estimators":
        D, F, E = case["accelerators"], FEATURES, case["types"] * KINDS
        so, sl = E * max(F + 1, case["samples"]), D * D * max(4, case["link_samples"])
        N, T = case["ops"], case["types"]
        stats = 8 * (E * (F * (F + 1) // 2 + 2 * F + 1) + D * D * 8)
        return {"bytes": 8 * (so * (F + 1) + sl * 3) + N * (12 * T + 8 * F + 8) + 3 * stats,
                "flops": 2 * (so * (F * (F + 1) // 2 + F) + sl * 5 + N * T * F)}
    ts = _templates(case)
    n, e = sum(t.n for t in ts), sum(t.pred_idx.size for t in ts)
    K, D, R = case["candidates"], case["accelerators"], case["requests"]
    graph = n * (8 * case["types"] + 8 + 8 + 4) + 4 * e
    per = 52 + 8 * D + 8 * R + (5 * (case["moves"] + 1) // 2 if case["path"] == "moves" else n)
    once = 16 * min(case["traced"], K) * n + (n if case["path"] == "moves" else 0)
    if case["path"] == "round":
        per, once = 52 + 8 * D + n, 12 * n
    return {"bytes": graph + K * per + once, "flops": 0}


def tolerance(case):
    if case["path"] != "estimators":
        return "exact"
    # measured against least squares: 6e-14 and below; a predicted duration may
    # round the other way
    return {"rel": 1e-12, "max": 4e-11, "differ": 1e-4}


def exact(case, seed):
    """Least squares over both feedback batches and what follows from it; the
    simulations' whole numbers are compared as they are."""
    if case["path"] != "estimators":
        return None
    f = _feedback(case, seed, torch.device("cuda"))
    D = case["accelerators"]
    beta = {}
    for name in ("op", "link"):
        parts = [(x.cpu().numpy().reshape(-1, per, x.shape[1]), y.cpu().numpy().reshape(-1, per)) for per, x, y in f[name]]
        X, Y = (np.concatenate([p[i] for p in parts], axis=1) for i in (0, 1))
        beta[name] = np.stack([np.linalg.lstsq(x, y, rcond=None)[0] for x, y in zip(X, Y)])
    est_of, x = f["est_of"].cpu().numpy(), f["features"].cpu().numpy()
    dur = np.maximum(1, np.rint(np.einsum("ntf,nf->nt", beta["op"][est_of], x))).astype(np.int64)
    alpha, c = beta["link"].T
    bw = np.maximum(1, np.rint(1.0 / alpha)).astype(np.int64)
    lat = np.maximum(0, np.rint(c)).astype(np.int64)
    bw[::D + 1], lat[::D + 1] = 400_000, 10
    return {"op_beta": beta["op"], "op_fitted": np.ones(len(beta["op"]), np.int32), "link_beta": beta["link"],
            "link_fitted": np.ones(D * D, np.int32), "dur": dur, "bw": bw, "lat": lat}
