"""The workloads this library is timed on, through its public binding.

Each case is one thing a user has the library do: a fixpoint over a resident
relation and its result in device memory, a whole request from host edges to a
host result, a batch, a served mix, triangle counting, or the sorted-array
primitives.  Graphs come from the seeded generators of the package, with the
sizes of its workloads, batch mix and served mix.
"""
import functools
import math

import numpy as np
import torch

from paper_2607_17571_gb300 import inputs as I
from paper_2607_17571_gb300 import wg

# Device memory the service may hold (a fixed budget, as a server sets one);
# the rest of the card is the caller's, for results.
BUDGET = 160 << 30


def listed():
    return [
        # the smallest fixpoint in use: launches and host round trips count
        {"name": "tc_er_1k", "kind": "tc_er", "nodes": 1000, "edges": 3000},
        # an ordinary skewed graph (hubs), closure of some 4e7 tuples
        {"name": "tc_rmat15_100k", "kind": "tc_rmat", "scale": 15, "edges": 100_000},
        # the benchmark's workload: closure of some 5e8 tuples, 16-bit ranks
        {"name": "tc_rmat17_400k", "kind": "tc_rmat", "scale": 17, "edges": 400_000},
        # the largest: ranks need 17 bits (64-bit keys), closure of some 1e9 tuples
        {"name": "tc_rmat19_400k", "kind": "tc_rmat", "scale": 19, "edges": 400_000},
        # a wide, sparse relation: many vertices, each reaching few others
        {"name": "tc_sparse_400k", "kind": "tc_er", "nodes": 400_000, "edges": 360_000},
        # deep recursion: one iteration per vertex of a long chain, few tuples in each
        {"name": "tc_chain_1000", "kind": "tc_chain", "nodes": 1000},
        # same-generation over a family forest with cross edges
        {"name": "sg_forest_60k", "kind": "sg", "nodes": 60_000},
        # many small uneven TC queries submitted at once
        {"name": "batch_64", "kind": "batch", "queries": 64},
        # TC and SG requests of very different sizes that arrive in waves
        {"name": "serve_48", "kind": "serve", "requests": 48},
        # triangle counting on an undirected skewed graph
        {"name": "tri_rmat16_800k", "kind": "tri", "scale": 16, "edges": 800_000},
        # one whole request: host edges in, load, fixpoint, sorted host result out
        {"name": "request_er_3k", "kind": "request", "nodes": 3000, "edges": 6000},
        # the sorted-array stages on a caller's own buffers: sort, dedup + set
        # difference, merge
        {"name": "stages_u64_16m", "kind": "stages", "keys": 1 << 24, "full": 1 << 24,
         "key_bytes": 8, "bits": 34},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tc_er", "tc_rmat", "tc_rmat", "tc_sparse", "tc_chain", "sg", "batch",
                       "serve", "tri", "request", "stages"])
    if kind == "tc_er":
        n = _log(rng, 64, 16384)
        return {"kind": "tc_er", "nodes": n, "edges": round(n * rng.uniform(1.2, 3.0))}
    if kind == "tc_rmat":
        m = _log(rng, 10_000, 400_000)
        lo = max(10, math.ceil(math.log2(m / 3)))
        return {"kind": "tc_rmat", "scale": rng.randint(lo, max(lo, 19)), "edges": m}
    if kind == "tc_sparse":
        n = _log(rng, 20_000, 400_000)
        return {"kind": "tc_er", "nodes": n, "edges": round(n * rng.uniform(0.5, 0.9))}
    if kind == "tc_chain":
        return {"kind": "tc_chain", "nodes": _log(rng, 50, 1000)}
    if kind == "sg":
        return {"kind": "sg", "nodes": _log(rng, 1000, 60_000)}
    if kind == "batch":
        return {"kind": "batch", "queries": _log(rng, 4, 64)}
    if kind == "serve":
        return {"kind": "serve", "requests": _log(rng, 4, 48)}
    if kind == "tri":
        m = _log(rng, 10_000, 400_000)
        return {"kind": "tri", "scale": max(10, math.ceil(math.log2(m / 6))), "edges": 2 * m}
    if kind == "request":
        n = _log(rng, 200, 3000)
        return {"kind": "request", "nodes": n, "edges": round(n * rng.uniform(1.2, 3.0))}
    kb = rng.choice([4, 8])
    return {"kind": "stages", "keys": _log(rng, 1000, 1 << 24), "full": _log(rng, 1000, 1 << 24),
            "key_bytes": kb, "bits": rng.randint(26, 32) if kb == 4 else rng.randint(34, 48)}


# ---------------------------------------------------------------- inputs
def _graph(case, seed):
    k = case["kind"]
    if k in ("tc_er", "request"):
        return I.er_graph(case["nodes"], case["edges"], seed)
    if k == "tc_rmat":
        return I.rmat_dag16(case["scale"], case["edges"], seed)
    if k == "tc_chain":  # a chain through distinct ids spread over all of uint32
        ids = np.random.default_rng(seed).choice(1 << 32, size=case["nodes"], replace=False)
        ids = ids.astype(np.uint32)
        return I.EdgeList(ids[:-1], ids[1:], {})
    if k == "sg":
        return _forest(case["nodes"], seed)
    if k == "tri":
        return I.rmat_sym(case["scale"], case["edges"] // 2, seed)
    raise KeyError(k)


def _forest(n, seed):
    while True:  # (a forest that dies out before it has n nodes is drawn again)
        try:
            return I.sg_forest(n, max(8, n // 1500), 2.0, 0.01, seed)
        except RuntimeError:
            seed += 1 << 20


def _requests(case, seed):
    """(kind, graph) of every query of a batch or served case."""
    if case["kind"] == "batch":
        # the batch mix, its node counts spread evenly over their range so that
        # two draws are alike in total work
        q, out = case["queries"], []
        u = np.random.default_rng(seed).uniform(size=(q, 2))
        for i in range(q):
            n = int(round(64 * 256.0 ** ((i + u[i, 0]) / q)))
            out.append(("tc", I.er_graph(n, int(round(n * (1.2 + 1.8 * u[i, 1]))), seed + i)))
        order = np.random.default_rng(seed + 1).permutation(q)
        return [out[i] for i in order]
    return [I.serve_request(r, seed & 0xFFFFFF, rmat_edges=(10_000, 150_000))
            for r in range(case["requests"])]


@functools.cache
def _ctx():
    return wg.Context(0, mem_budget=BUDGET)


class _Relations:
    """Resident relations, freed with the state that holds them."""

    def __init__(self, graphs):
        self.rels = [_ctx().load(g.src, g.dst) for g in graphs]

    def __del__(self):
        for r in self.rels:
            r.free()


def prepare(case, seed):
    k = case["kind"]
    if k == "stages":
        dt = torch.int32 if case["key_bytes"] == 4 else torch.int64
        g = torch.Generator(device="cuda").manual_seed(seed)
        n, f, top = case["keys"], case["full"], 1 << case["bits"]
        # a full relation of f distinct sorted keys, and candidates with
        # duplicates, some of them already in it (32-bit keys: the bit patterns,
        # in unsigned order)
        full = torch.randint(1, top // f + 1, (f,), generator=g, device="cuda").cumsum(0) - 1
        cand = torch.randint(0, top, (n,), generator=g, device="cuda")
        cand[: n // 4] = full[torch.randint(0, f, (n // 4,), generator=g, device="cuda")]
        cand = cand[torch.randperm(n, generator=g, device="cuda")]
        _ctx()
        state = {"case": case, "cand": cand.to(dt), "full": full.to(dt),
                 "new": torch.zeros(n, dtype=dt, device="cuda"),
                 "merged": torch.zeros(n + f, dtype=dt, device="cuda")}
        torch.cuda.synchronize()
        return state
    if k in ("batch", "serve"):
        reqs = _requests(case, seed)
        kinds = [wg.WG_SG if q == "sg" else wg.WG_TC for q, _ in reqs]
        rels = _Relations([g for _, g in reqs])
    else:
        g = _graph(case, seed)
        if k == "tri":
            return {"case": case, "rels": _Relations([g])}
        if k == "request":  # the reusable page-locked I/O buffers of a server
            src, dst = wg.pinned(len(g), np.uint32), wg.pinned(len(g), np.uint32)
            out = wg.pinned(case["nodes"] ** 2)
            src[:], dst[:], out[:] = g.src, g.dst, 0
            return {"case": case, "src": src, "dst": dst, "out": out}
        kinds, rels = [], _Relations([g])
    # the caller's result buffer, large enough for what such a workload returns
    keys = torch.zeros(_capacity(case), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    return {"case": case, "kinds": kinds, "rels": rels, "keys": keys}


# ---------------------------------------------------------------- one pass
def _padded(deltas, n):
    """Per-iteration delta sizes in an array of n entries (zeros after the last)."""
    out = np.zeros(n, dtype=np.int64)
    out[: len(deltas)] = deltas
    return out


def _answer(q, case, keys):
    st = q.poll()
    return {"keys": keys, "tuples": st.n_tuples, "iterations": st.iterations,
            "candidates": st.candidates,
            "deltas": _padded(q.delta_sizes(), 1 << 14 if case["kind"] != "tc_chain" else 1 << 10)}


def _many(state):
    """Queries submitted together (batch) or in four waves (served), their
    results gathered into one device buffer when all are done."""
    ctx, keys = _ctx(), state["keys"]
    reqs = list(zip(state["kinds"], state["rels"].rels))
    waves = 1 if state["case"]["kind"] == "batch" else 4
    step = -(-len(reqs) // waves)
    hs = []
    for at in range(0, len(reqs), step):
        hs += ctx.submit(reqs[at:at + step])
        ctx.serve_step(4)
    while ctx.serve_step(16):
        pass
    ctx.take_completed()
    st, at, deltas = [h.poll() for h in hs], 0, []
    for h in hs:
        at += h.result_device(keys.data_ptr() + 8 * at, keys.numel() - at)
        deltas.append(_padded(h.delta_sizes(), 1 << 10))
        h.free()
    return {"keys": keys, "tuples": np.array([s.n_tuples for s in st], dtype=np.int64),
            "iterations": np.array([s.iterations for s in st]),
            "candidates": np.array([s.candidates for s in st], dtype=np.int64),
            "deltas": np.concatenate(deltas)}


def run(state):
    case, ctx = state["case"], _ctx()
    k = case["kind"]
    if k == "stages":
        kb, full, new, merged = case["key_bytes"], state["full"], state["new"], state["merged"]
        cand = state["cand"].clone()
        torch.cuda.current_stream().synchronize()  # the context works on its own stream
        ctx.sort_keys(cand.data_ptr(), cand.numel(), kb, case["bits"])
        n = ctx.unique_diff(cand.data_ptr(), cand.numel(), full.data_ptr(), full.numel(),
                            new.data_ptr(), kb)
        ctx.merge_disjoint(full.data_ptr(), full.numel(), new.data_ptr(), n, merged.data_ptr(), kb)
        return {"sorted": cand, "new": new, "n_new": n, "merged": merged}
    if k in ("batch", "serve"):
        return _many(state)
    if k == "tri":
        return {"triangles": ctx.triangles(state["rels"].rels[0])}
    if k == "request":
        rel = ctx.load(state["src"], state["dst"])
        q = ctx.tc(rel)
        q.wait()
        q.result(out=state["out"])
        out = _answer(q, case, state["out"].view(np.int64))
        q.free()
        rel.free()
        return out
    rel, keys = state["rels"].rels[0], state["keys"]
    q = ctx.sg(rel) if k == "sg" else ctx.tc(rel)
    q.wait()
    q.result_device(keys.data_ptr(), keys.numel())
    out = _answer(q, case, keys)
    q.free()
    return out


# ---------------------------------------------------------------- what a pass cannot do without
def _er_tuples(n, m):
    """Expected closure of a directed ER graph: pairs from the giant in-component
    to the giant out-component, and below the threshold the mean reach."""
    d, g = m / n, 0.5
    if d < 1:
        return n * d / (1 - d)
    for _ in range(200):
        g = 1 - math.exp(-d * g)
    return (g * n) ** 2


def _rmat_tuples(scale, m):
    """Fit to the closures of the package's R-MAT workloads (3.7e7 at 2^15 / 100k
    edges, 4.8e8 at 2^17 / 400k, 1.0e9 at 2^19 / 400k)."""
    return 3e-3 * m * m * min(2.2, max(1.0, (1 << scale) / m * 1.6))


def _sg_tuples(n):
    return 0.02 * n * n


def _capacity(case):
    """Tuples a caller's result buffer holds: above what the seeds' draws vary by."""
    k = case["kind"]
    if k == "tc_er":
        n = case["nodes"]
        return n * n if n <= 3000 else int(min(n * n, 1.6 * _er_tuples(n, case["edges"]) + 40 * n))
    if k == "tc_rmat":
        return int(1.8 * _rmat_tuples(case["scale"], case["edges"])) + 1_000_000
    if k == "tc_chain":
        return case["nodes"] ** 2 // 2
    if k == "sg":
        return int((0.5 if case["nodes"] < 10_000 else 0.12) * case["nodes"] ** 2)
    if k == "batch":
        q = case["queries"]
        return sum(int(64 * 256 ** ((i + 1) / q) + 1) ** 2 for i in range(q))
    return int(2.5 * work(case)["bytes"] / 8) + 3 * 16384 ** 2


def work(case):
    """Bytes of the edges read once and the sorted result written once (8 bytes a
    tuple); a result's size is the generators' expected one."""
    k = case["kind"]
    if k in ("tc_er", "request"):
        b = 8 * case["edges"] + 8 * _er_tuples(case["nodes"], case["edges"])
    elif k == "tc_rmat":
        b = 8 * case["edges"] + 8 * _rmat_tuples(case["scale"], case["edges"])
    elif k == "tc_chain":
        b = 8 * case["nodes"] + 4 * case["nodes"] ** 2
    elif k == "sg":
        b = 8 * case["nodes"] + 8 * _sg_tuples(case["nodes"])
    elif k == "batch":
        q = case["queries"]
        b = sum(8 * _er_tuples(n, 2.1 * n) for n in (64 * 256 ** ((i + 0.5) / q) for i in range(q)))
    elif k == "serve":
        ns = [64 * 256 ** ((i + 0.5) / 64) for i in range(64)]
        ms = [10_000 * 15 ** ((i + 0.5) / 64) for i in range(64)]
        one = (0.25 * sum(map(_sg_tuples, ns)) + 0.525 * sum(_er_tuples(n, 2.1 * n) for n in ns) +
               0.225 * sum(_rmat_tuples(math.ceil(math.log2(m / 3)), m) for m in ms)) / 64
        b = case["requests"] * 8 * one
    elif k == "tri":
        b = 4 * case["edges"] + 8  # edges and their index read once, one count written
    else:
        kb, n, f = case["key_bytes"], case["keys"], case["full"]
        # sort: read and write; dedup + difference: read both, write the new; merge
        b = kb * (2 * n + (n + f + 0.7 * n) + 2 * (f + 0.7 * n))
    return {"bytes": float(b), "flops": 0.0}


# ---------------------------------------------------------------- 64-bit reference
def exact(case, seed):
    """Outputs are whole numbers; the smaller closures and the stages are given in
    plain torch / numpy."""
    k = case["kind"]
    if k == "stages":
        s = prepare(case, seed)
        mask = 0xFFFFFFFF if case["key_bytes"] == 4 else (1 << 63) - 1
        key, full, dt = s["cand"].long() & mask, s["full"].long() & mask, s["cand"].dtype
        new = torch.unique(key)
        at = torch.searchsorted(full, new).clamp(max=full.numel() - 1)
        new = new[full[at] != new]
        n = new.numel()
        s["new"][:n] = new.to(dt)
        s["merged"][: n + full.numel()] = torch.cat([full, new]).sort().values.to(dt)
        return {"sorted": key.sort().values.to(dt), "new": s["new"], "n_new": n,
                "merged": s["merged"]}
    if k not in ("tc_er", "tc_chain", "request") or case["nodes"] > 3000:
        return None
    g = _graph(case, seed)
    ids, e = np.unique(np.stack([g.src, g.dst]), return_inverse=True)
    n = ids.shape[0]
    e = torch.from_numpy(e.reshape(2, -1)).cuda()
    E = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    E[e[0], e[1]] = 1
    full, delta, deg = E > 0, E > 0, E.sum(1)
    sizes, cand = [int(delta.sum())], int(delta.sum())
    while sizes[-1]:
        cand += int((delta.double() @ deg).sum())
        delta = (delta.double() @ E > 0) & ~full
        full |= delta
        sizes.append(int(delta.sum()))
    x, y = (t.cpu().numpy() for t in full.nonzero(as_tuple=True))
    keys = np.zeros(case["nodes"] ** 2 if k == "request" else _capacity(case), dtype=np.uint64)
    keys[: x.shape[0]] = (ids[x].astype(np.uint64) << np.uint64(32)) | ids[y].astype(np.uint64)
    return {"keys": keys.view(np.int64), "tuples": x.shape[0], "iterations": len(sizes) - 1,
            "candidates": cand, "deltas": _padded(sizes, 1 << 10 if k == "tc_chain" else 1 << 14)}
