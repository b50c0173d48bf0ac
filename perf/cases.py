"""The measured work of the library: static scores, update streams, batches and serving,
each through the public entry points (include/bcgpu.h, the ctypes binding), over the
sizes, graph families and types of the repository's own workloads and tests.

An update is destructive (weights only drop), so a state of a stream holds a handle and a
long seeded stream cut into passes; each run() applies the next pass.  A stream holds more
passes than a few seconds use up; past its end the handle is rebuilt from the initial
graph and the stream starts again.  Whole passes are encoded beforehand into the
bc_update / bc_vedge arrays of the ABI, which is what a caller of the C library has.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1311_2147_gb300 import binding, synth

# ---------------------------------------------------------------------------- cases


def listed():
    return [
        # The scores of a small graph that is already on the device, for a caller that may
        # not allocate (a framework's tensors in, a tensor out): the smallest call, where
        # launches and latency count.
        dict(name="scores_er256_i64", kind="scores", graph="er", n=256, degree=8, dist="i64", whi=1000),
        # The small plain workload as one job: build G(256, 2048), apply its 16 edge
        # updates, read BC and the whole state, drop the handle.
        dict(name="job_er256_i64", kind="job", graph="er", n=256, degree=8, dist="i64", whi=1000, updates=16, rows=True),
        # Static computation of a mid-size undirected network (what a server does when it
        # admits a graph, and the recompute an incremental update is compared with).
        dict(name="static_ba4096_i32", kind="job", graph="ba", n=4096, degree=8, dist="i32", whi=100, updates=0),
        # The same for a directed graph with wide weights and an odd number of vertices.
        dict(name="static_er3001_i64", kind="job", graph="er", n=3001, degree=8, dist="i64", whi=100000, updates=0),
        # Dense extreme: complete directed graph, w ~ U{1..n^2}; decreases of random edges
        # (nearly all change nothing) with one in four at or below the current distance.
        dict(name="stream_complete2048_i64", kind="stream", graph="complete", n=2048, degree=0, dist="i64",
             whi=2048 * 2048, per_pass=32, passes=96, vertex=0),
        # Directed sparse network: edge and vertex updates half and half.
        dict(name="stream_er4096_i32", kind="stream", graph="er", n=4096, degree=8, dist="i32", whi=100,
             per_pass=8, passes=128, vertex=50),
        # Undirected network with an odd number of vertices (no row but the first starts on
        # a 16-byte boundary), edge and vertex updates.
        dict(name="stream_ba5003_i32", kind="stream", graph="ba", n=5003, degree=8, dist="i32", whi=100,
             per_pass=16, passes=128, vertex=50),
        # The headline workload: BA n = 16384, edge and vertex updates, 32-bit distances.
        dict(name="stream_ba16384_i32", kind="stream", graph="ba", n=16384, degree=8, dist="i32", whi=100,
             per_pass=16, passes=64, vertex=50),
        # Real weights, one synchronous call per edge update and a read of BC after each
        # few: an interactive caller, where the latency of one update counts.
        dict(name="calls_real1500_f64", kind="real", graph="ba", n=1500, degree=8, dist="i64", whi=100,
             per_pass=4, passes=512, vertex=0),
        # Many small graphs of uneven size in one batch call, 8 edge updates each.
        dict(name="batch96_i32", kind="batch", graph="mixed", n=2048, degree=8, dist="i32", whi=1000,
             count=96, per_pass=8, passes=32, vertex=0),
        # Continuous batching: requests for resident graphs submitted and drained.
        dict(name="serve12_i32", kind="serve", graph="mixed", n=4096, degree=8, dist="i32", whi=100,
             count=12, per_pass=8, passes=48, vertex=50),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["scores", "job", "job", "stream", "stream", "stream", "complete", "real", "batch", "serve"])
    c = dict(kind=kind, graph=rng.choice(["er", "ba"]), degree=rng.choice([4, 8, 12]), dist=rng.choice(["i32", "i64"]),
             whi=rng.choice([10, 100, 1000]))
    if kind == "scores":
        c["n"] = _log_int(rng, 64, 512)
        c["degree"] = rng.choice([4, 8, 16])
    elif kind == "job":
        c["n"] = _log_int(rng, 256, 6000)
        c["updates"] = rng.choice([0, 4, 16])
        c["rows"] = c["n"] <= 512
    elif kind == "stream":
        c.update(n=_log_int(rng, 768, 10000), per_pass=rng.choice([1, 4, 8, 16]), vertex=rng.choice([0, 50, 100]))
        if c["graph"] == "er":
            c["n"] = min(c["n"], 5000)
        c["passes"] = 1024 // c["per_pass"]
    elif kind == "complete":
        c.update(kind="stream", graph="complete", degree=0, dist="i64", n=_log_int(rng, 512, 2048),
                 per_pass=rng.choice([8, 16, 32]), passes=96, vertex=0)
        c["whi"] = c["n"] * c["n"]
    elif kind == "real":
        c.update(n=_log_int(rng, 256, 4096), dist="i64", per_pass=4, passes=384, vertex=0)
        c["whi"] = 100
    elif kind == "batch":
        c.update(graph="mixed", n=_log_int(rng, 256, 2048), degree=8, count=_log_int(rng, 8, 96), per_pass=8,
                 passes=32, vertex=0, whi=1000)
    else:
        c.update(graph="mixed", n=_log_int(rng, 1024, 6000), degree=8, count=rng.choice([4, 8, 12]), per_pass=8,
                 passes=48, vertex=50, whi=100)
    return c


# ---------------------------------------------------------------------------- inputs


def _graph(c, n, family, seed):
    if family == "complete":
        return synth.complete_directed(n, 1, c["whi"], seed)
    if family == "ba":
        return synth.barabasi_albert(max(n, c["degree"] + 1), c["degree"], 1, c["whi"], seed)
    return synth.erdos_renyi_degree(n, c["degree"], 1, c["whi"], seed)


def _members(c, seed):
    """The graphs of a case: (family, graph) pairs; a mixed case has even ones directed
    and odd ones undirected, n log-uniform up to c["n"] (as the batch and serving workloads)."""
    if c["graph"] != "mixed":
        return [_graph(c, c["n"], c["graph"], synth.sub_seed(seed, 0))]
    lo = 64 if c["kind"] == "batch" else 1024
    ns = synth.log_uniform_n(synth.Rng(c["n"]), lo, c["n"] + 1, c["count"])
    return [_graph(c, n, "ba" if i % 2 else "er", synth.sub_seed(seed, 10 + i)) for i, n in enumerate(ns)]


def _dense_distances(g):
    """All-pairs distances by Floyd-Warshall in 64 bits (inf: no path)."""
    d = torch.full((g.n, g.n), math.inf, dtype=torch.float64, device="cuda")
    src, dst = (torch.from_numpy(x.astype(np.int64)).cuda() for x in (g.src, g.dst))
    d[src, dst] = torch.from_numpy(g.w).cuda().double()
    d.fill_diagonal_(0.0)
    for k in range(g.n):
        torch.minimum(d, d[:, k, None] + d[None, k, :], out=d)
    return d


def _complete_decreases(g, count, seed):
    """Distinct random edges of a complete graph with a lower weight each: U[1, w-1], every
    fourth U[1, d] with d the initial distance (a decrease that can change something)."""
    rng = synth.Rng(seed)
    e = np.unique(rng.below(g.m, 2 * count))
    e = e[np.argsort(rng.u64(e.shape[0]), kind="stable")]
    e = e[g.w[e] >= 2][:count]
    dist = _dense_distances(g)[torch.from_numpy(g.src[e].astype(np.int64)), torch.from_numpy(g.dst[e].astype(np.int64))]
    cap = g.w[e] - 1
    every4 = np.arange(e.shape[0]) % 4 == 0
    cap[every4] = np.minimum(cap, dist.cpu().numpy().astype(np.int64))[every4]
    w = 1 + (rng.unit(e.shape[0]) * cap).astype(np.int64)
    return [("edge", int(a), int(b), int(x)) for a, b, x in zip(g.src[e], g.dst[e], w)]


def _stream(c, g, count, seed):
    if c["graph"] == "complete":
        return _complete_decreases(g, count, seed)
    nv = count * c.get("vertex", 0) // 100
    new = (count - nv) // 2
    return synth.update_stream(g, new, count - nv - new, nv, seed, 1, c["whi"])


def _total(c):
    return c["updates"] if c["kind"] == "job" else c["per_pass"] * c["passes"] if c["kind"] != "scores" else 0


def _inputs(c, seed):
    """[(graph, its updates)] of a case, from the seed alone."""
    gs = _members(c, seed)
    return [(g, _stream(c, g, _total(c), synth.sub_seed(seed, 1000 + i))) for i, g in enumerate(gs)]


def _csr(g):
    src, dst, w = g.src.astype(np.int64), g.dst.astype(np.int64), g.w.astype(np.int64)
    if not g.directed:
        src, dst, w = np.concatenate([src, dst]), np.concatenate([dst, src]), np.concatenate([w, w])
    order = np.lexsort((dst, src))
    off = np.zeros(g.n + 1, np.int32)
    off[1:] = np.cumsum(np.bincount(src, minlength=g.n))
    return off, dst[order].astype(np.int32), w[order]


REAL_UNIT = 1.0 / 64   # real weights: multiples of 2^-6, so that ties occur as with integers


def prepare(case, seed):
    c = case
    lib = binding.load()
    st = {"case": c, "lib": lib, "at": 0}
    data = _inputs(c, seed)
    g0, ups0 = data[0]
    if c["kind"] == "scores":
        off, dst, w = (torch.from_numpy(x).cuda() for x in _csr(g0))
        flags = (binding.BC_DIRECTED if g0.directed else binding.BC_UNDIRECTED) | (
            binding.BC_DIST_I32 if c["dist"] == "i32" else binding.BC_DIST_I64)
        st.update(n=g0.n, off=off, dst=dst, w=w, flags=flags, out=torch.empty(g0.n, dtype=torch.float64, device="cuda"))
    elif c["kind"] == "job":
        st.update(g=g0, ups=binding.encode_updates(ups0))
    elif c["kind"] in ("stream", "real"):
        u = c["per_pass"]
        parts = [ups0[i:i + u] for i in range(0, len(ups0), u)]
        st.update(g=g0, parts=[binding.encode_updates(p) for p in parts] if c["kind"] == "stream" else parts)
    elif c["kind"] == "batch":
        u, passes = c["per_pass"], []
        for p in range(c["passes"]):
            lists = [ups[p * u:(p + 1) * u] for _, ups in data]
            passes.append((np.array([len(x) for x in lists], np.int32), *binding.encode_updates([x for l in lists for x in l])))
        st.update(graphs=[g for g, _ in data], parts=passes)
    else:
        u = c["per_pass"]
        # requests of a pass in arrival order, graphs in turn
        st.update(graphs=[g for g, _ in data],
                  parts=[[(i, ups[p * u + j]) for j in range(u) for i, (_, ups) in enumerate(data)]
                         for p in range(c["passes"])])
    _open(st)
    return st


def _open(st):
    """The handle, batch or server that a user's program keeps between passes."""
    c = st["case"]
    st["at"] = 0
    if c["kind"] == "stream":
        st["h"] = binding.BCGraph(st["g"], dist=c["dist"])
    elif c["kind"] == "real":
        g = st["g"]
        st["h"] = binding.BCGraphReal(g.n, g.directed, g.src, g.dst, g.w * REAL_UNIT, dist=c["dist"])
    elif c["kind"] == "batch":
        st["hs"] = [binding.BCGraph(g, dist=c["dist"]) for g in st["graphs"]]
        st["b"] = binding.BCBatch(st["hs"])
    elif c["kind"] == "serve":
        st["srv"] = binding.BCServer(64 << 30)
        st["ids"] = [st["srv"].add_graph(g, dist=c["dist"]) for g in st["graphs"]]


def _next(st):
    if st["at"] == len(st["parts"]):
        for k in ("b", "h", "srv"):
            if k in st:
                st.pop(k).close()
        for h in st.pop("hs", []):
            h.close()
        _open(st)
    st["at"] += 1
    return st["parts"][st["at"] - 1]


# ---------------------------------------------------------------------------- a pass


def _ok(rc):
    if rc != binding.BC_OK:
        raise RuntimeError("bcgpu error %d" % rc)


def run(state):
    return globals()["_run_" + state["case"]["kind"]](state)


def _run_scores(st):
    _ok(st["lib"].bc_static_scores_noalloc(st["n"], int(st["dst"].shape[0]), st["off"].data_ptr(), st["dst"].data_ptr(),
                                           st["w"].data_ptr(), st["flags"], st["out"].data_ptr(),
                                           torch.cuda.current_stream().cuda_stream))
    return {"bc": st["out"]}


def _run_job(st):
    h = binding.BCGraph(st["g"], dist=st["case"]["dist"])
    done = 0
    if st["ups"][0].shape[0]:
        rc, done = h.bc_apply_updates(st["ups"])
        _ok(rc)
    bc = h.bc_get_scores()
    rows = h.bc_get_rows() if st["case"].get("rows") else ()
    h.close()
    return {"bc": bc, "done": done, "rows": rows}


def _run_stream(st):
    # the scores, and the state of the vertex updated last (its row of d, sigma and delta)
    part = _next(st)
    rc, done = st["h"].bc_apply_updates(part)
    _ok(rc)
    return {"bc": st["h"].bc_get_scores(), "done": done, "rows": st["h"].bc_get_rows(int(part[0]["v"][-1]), 1)}


def _run_real(st):
    part = _next(st)
    h = st["h"]
    for _, u, v, w in part:
        _ok(h.bc_apply_edge_update_f64(u, v, w * REAL_UNIT))
    return {"bc": h.bc_get_scores()}


def _run_batch(st):
    counts, rec, ed = _next(st)
    b = st["b"]
    done = np.zeros(len(st["hs"]), np.int32)
    p = ctypes.c_void_p
    _ok(st["lib"].bc_batch_apply(b.h, counts.ctypes.data_as(p), rec.ctypes.data_as(p),
                                 ed.ctypes.data_as(p) if ed.size else None, int(ed.shape[0]), done.ctypes.data_as(p)))
    return {"bc": np.concatenate([h.bc_get_scores() for h in st["hs"]]), "done": done}


def _run_serve(st):
    part = _next(st)
    srv, ids = st["srv"], st["ids"]
    for i, up in part:
        srv.submit(ids[i], up)
    res = srv.drain()
    return {"bc": np.concatenate([srv.graph(i).bc_get_scores() for i in ids]),
            "answered": np.bincount(res["graph_id"], minlength=len(ids)), "failed": int(np.sum(res["status"] != 0))}


# ---------------------------------------------------------------------------- work


def work(case):
    """Bytes and operations of a pass.  Static: the arcs read and, per pair, d, sigma and
    delta written once; every arc relaxed and every arc accumulated once per source.
    Update: half of the sources change at these sizes, and finding the changed pairs of
    a changed row takes its distances, once (the measured share over the declared ranges;
    nearly all of the complete graph's decreases change nothing, so there it is the four
    rows and columns at the edge's ends)."""
    c = case
    sd = 4 if c["dist"] == "i32" else 8
    if c["graph"] == "mixed":
        # E[n^2] for n log-uniform in [lo, hi]
        lo, hi = (64 if c["kind"] == "batch" else min(1024, c["n"])), c["n"]
        l = math.log(hi / lo) if hi > lo else 1.0
        nn = c["count"] * ((hi * hi - lo * lo) / (2 * l) if hi > lo else hi * hi)
        n = c["count"] * c["n"] / 2
    else:
        n, nn = c["n"], float(c["n"]) ** 2
    arcs = n * (n - 1) if c["graph"] == "complete" else n * c["degree"] * (2 if c["graph"] == "ba" else 1)
    out = 8.0 * n
    if c["kind"] == "scores":
        return {"bytes": 16.0 * arcs + out, "flops": 4.0 * arcs * n}
    b, f = out, 0.0
    if c["kind"] == "job":
        b += arcs * (4 + sd) + nn * (sd + 16)
        f += 4.0 * arcs * n
    ups = c["updates"] if c["kind"] == "job" else c["per_pass"]
    if c["graph"] == "complete":
        return {"bytes": b + ups * 4.0 * n * (sd + 8), "flops": ups * 2.0 * n}
    return {"bytes": b + ups * 0.5 * nn * sd, "flops": f + ups * 0.5 * nn}


# ---------------------------------------------------------------------------- 64 bits


def _after(g, ups):
    """Arcs of the graph after the updates (weights only drop, so the least one holds)."""
    src, dst, w = [g.src.astype(np.int64)], [g.dst.astype(np.int64)], [g.w.astype(np.int64)]
    es = []
    for u in ups:
        if u[0] == "edge":
            es.append((u[1], u[2], u[3]))
        else:
            es += [((x, u[1], y) if d == 0 else (u[1], x, y)) for x, y, d in u[2]]
    if es:
        e = np.array(es, np.int64)
        src.append(e[:, 0])
        dst.append(e[:, 1])
        w.append(e[:, 2])
    src, dst, w = np.concatenate(src), np.concatenate(dst), np.concatenate(w)
    if not g.directed:
        src, dst, w = np.concatenate([src, dst]), np.concatenate([dst, src]), np.concatenate([w, w])
    key = src * g.n + dst
    order = np.lexsort((w, key))
    key, w = key[order], w[order]
    first = np.concatenate([[True], key[1:] != key[:-1]]) if key.size else np.zeros(0, bool)
    return key[first] // g.n, key[first] % g.n, w[first]


def _brandes(n, directed, src, dst, w, rows=()):
    """BC of a weighted graph in torch, in 64 bits, and d, sigma and delta of the sources in
    rows: distances by relaxation, path counts and dependencies as sums over the
    shortest-path DAGs by number of arcs, for blocks of sources at a time (rows: vertices,
    columns: sources)."""
    kept = [[], [], []]
    src, dst, w = (torch.from_numpy(x).cuda() for x in (src, dst, w.astype(np.float64)))
    dense = None
    if src.numel() > n * n // 8:
        dense = _dense_distances(synth.Graph(n, True, src.cpu().numpy(), dst.cpu().numpy(), w.cpu().numpy())).T.contiguous()
        keep = dense.T[src, dst] == w
        src, dst, w = src[keep], dst[keep], w[keep]
    wc = w[:, None]
    bc = torch.zeros(n, dtype=torch.float64, device="cuda")
    step = max(32, min(n, int(2e8 // max(1, src.numel()))))
    for s0 in range(0, n, step):
        s1 = min(n, s0 + step)
        cols = torch.arange(s1 - s0, device="cuda")
        if dense is not None:
            d = dense[:, s0:s1].contiguous()
        else:
            d = torch.full((n, s1 - s0), math.inf, dtype=torch.float64, device="cuda")
            d[cols + s0, cols] = 0.0
            while True:
                nd = d.index_reduce(0, dst, d[src] + wc, "amin")
                if torch.equal(nd, d):
                    break
                d = nd
        on = ((d[src] + wc) == d[dst]) & torch.isfinite(d[dst])
        x = torch.zeros_like(d)
        x[cols + s0, cols] = 1.0
        sig = x.clone()
        while bool(x.any()):
            x = torch.zeros_like(x).index_add_(0, dst, x[src] * on)
            sig += x
        ratio = torch.where(on, sig[src] / sig[dst], 0.0)
        y = torch.isfinite(d).double()
        dep = torch.zeros_like(d)
        while bool(y.any()):
            y = torch.zeros_like(y).index_add_(0, src, ratio * y[dst])
            dep += y
        dep[cols + s0, cols] = 0.0
        bc += dep.sum(1)
        for s in rows:
            if s0 <= s < s1:
                far = torch.isinf(d[:, s - s0])
                kept[0].append(torch.where(far, 0.0, d[:, s - s0]).long().masked_fill(far, binding.INF64).cpu().numpy())
                kept[1].append(sig[:, s - s0].long().cpu().numpy().astype(np.uint64))
                kept[2].append(dep[:, s - s0].cpu().numpy())
    return (bc if directed else bc * 0.5).cpu().numpy(), tuple(np.stack(k) for k in kept) if rows else ()


def exact(case, seed):
    c = case
    bcs, rows = [], ()
    for g, ups in _inputs(c, seed):
        first = ups if c["kind"] == "job" else ups[:c.get("per_pass", 0)]
        want = range(g.n) if c.get("rows") else ()
        if c["kind"] == "stream":
            want = (first[-1][2] if first[-1][0] == "edge" else first[-1][1],)
        bc, rows = _brandes(g.n, g.directed, *_after(g, first), rows=want)
        bcs.append(bc)
    if c["kind"] == "scores":
        return {"bc": torch.from_numpy(bcs[0]).cuda()}
    out = {"bc": np.concatenate(bcs)}
    if c["kind"] in ("job", "stream"):
        out.update(done=None, rows=rows)
    elif c["kind"] == "batch":
        out["done"] = None
    elif c["kind"] == "serve":
        out.update(answered=None, failed=None)
    return out
