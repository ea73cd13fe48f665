"""The work users have this framework do, as cases a timing program can run.

Index creation (Listing 1 of arXiv 2103.14688) on the graphs and query automata of the
repository's own workloads: regular queries and Dyck-4 from the smallest graphs to the
largest supported one, the worst case of many iterations, multiple-source runs, a batch of
independent queries, a server with a resident graph, and path extraction from an answer.

A case is a dict of plain values; ``kind`` says which entry points a pass calls:

* ``query``    load_graph_device, run, reachable_words: an application re-runs its query
               whenever the graph has changed, and reads the whole answer;
* ``rsm``      load_rsm, run, reachable_words: one graph, another query each time;
* ``sources``  load_graph_device, run_sources, closure_rows of the sources' start rows;
* ``batch``    batch_run of many (graph, RSM) pairs, every start box's answer read;
* ``server``   submit, step until every query is done, every answer read and released;
* ``paths``    load_graph_device, run, extract_paths for some pairs of vertices.

Answers are bit matrices (as int64 words) and whole numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2103_14688_gb300 import cfpq, workloads as W

OUT_DEGREE_ZIPF = 3.0  # mean out-degree of the Zipf graphs (Dyck-4, served)
OUT_DEGREE_ER = 4.0    # mean out-degree of the batch's graphs


def listed():
    return [
        # a small regular query: the latency of one call (answer of a few KB)
        {"name": "rpq_n200", "kind": "query", "query": "rpq", "n": 200, "out_deg": 3},
        # a regular query on a graph of a thousand vertices: many short launches
        {"name": "rpq_n1000", "kind": "query", "query": "rpq", "n": 1000, "out_deg": 4},
        # the benchmark's regular query
        {"name": "rpq_n8192", "kind": "query", "query": "rpq", "n": 8192, "out_deg": 8},
        # a regular query on a large sparse graph, a ragged size
        {"name": "rpq_sparse_n30011", "kind": "query", "query": "rpq", "n": 30011, "out_deg": 2},
        # a^n b^n on two coprime cycles: thousands of short iterations
        {"name": "cycles_63_64", "kind": "query", "query": "cycles", "n": 63, "out_deg": 1},
        # Dyck-4 (context-free reachability) where the answer is still small, a ragged size
        {"name": "dyck4_n3001", "kind": "query", "query": "dyck", "n": 3001, "out_deg": 3},
        # Dyck-4 of a medium graph, another grammar loaded each time (the plan is made anew)
        {"name": "dyck4_rsm_n16384", "kind": "rsm", "query": "dyck", "n": 16384, "out_deg": 3},
        # the benchmark's Dyck-4, the largest graph that is supported
        {"name": "dyck4_n65536", "kind": "query", "query": "dyck", "n": 65536, "out_deg": 3},
        # reachability from a few vertices of a large sparse graph
        {"name": "sources16_n65536", "kind": "sources", "query": "rpq", "n": 65536, "out_deg": 2, "sources": 16},
        # independent queries over graphs of mixed sizes in one call
        {"name": "batch_48", "kind": "batch", "queries": 48, "n_min": 256, "n_max": 8192, "grammars": 4},
        # a resident graph serving a burst of different queries
        {"name": "server_12_n12000", "kind": "server", "n": 12000, "queries": 12, "grammars": 5},
        # the paths behind some pairs of a Dyck-4 answer
        {"name": "dyck4_paths_n4096", "kind": "paths", "query": "dyck", "n": 4096, "out_deg": 3, "pairs": 8,
         "max_len": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rpq", "rpq", "dyck", "dyck", "cycles", "rsm", "sources", "batch", "server", "paths"])
    if kind == "rpq":
        n = _log_int(rng, 100, 32768)
        return {"kind": "query", "query": "rpq", "n": n, "out_deg": rng.randint(2, 8 if n <= 8192 else 3)}
    if kind == "dyck":
        return {"kind": "query", "query": "dyck", "n": _log_int(rng, 100, 40000), "out_deg": 3}
    if kind == "cycles":
        return {"kind": "query", "query": "cycles", "n": rng.randint(5, 63), "out_deg": 1}
    if kind == "rsm":
        return {"kind": "rsm", "query": rng.choice(["dyck", "rpq"]), "n": _log_int(rng, 500, 16384), "out_deg": 3}
    if kind == "sources":
        return {"kind": "sources", "query": "rpq", "n": _log_int(rng, 2000, 65536), "out_deg": rng.randint(2, 3),
                "sources": _log_int(rng, 1, 64)}
    if kind == "batch":
        return {"kind": "batch", "queries": rng.randint(4, 48), "n_min": 256, "n_max": _log_int(rng, 600, 8192),
                "grammars": rng.randint(1, 10 ** 6)}
    if kind == "server":
        return {"kind": "server", "n": _log_int(rng, 1000, 12000), "queries": rng.randint(2, 12),
                "grammars": rng.randint(1, 10 ** 6)}
    return {"kind": "paths", "query": "dyck", "n": _log_int(rng, 600, 4096), "out_deg": 3, "pairs": rng.randint(2, 8),
            "max_len": rng.choice([4, 6, 8])}


def _rng(seed, salt):
    return np.random.Generator(np.random.PCG64([int(seed), salt]))


def _permuted(g, rng):
    """The graph with its vertices renumbered and its edges in another order."""
    p = rng.permutation(g.n).astype(np.uint32)
    o = rng.permutation(g.m)
    return W.Graph(g.n, g.n_terminals, p[g.src][o], g.lbl[o], p[g.dst][o])


def _graph_and_rsm(case, seed):
    if case["query"] == "rpq":
        return W.rpq_abc(n=case["n"], out_deg=case["out_deg"], seed=int(seed))
    if case["query"] == "cycles":
        g, r = W.two_cycles(case["n"], case["n"] + 1)
        return _permuted(g, _rng(seed, 1)), r
    return W.dyck_zipf(n=case["n"], seed=int(seed))


def _batch(case, seed):
    """The batch: sizes, labels and grammars by ``grammars``, edges by the seed."""
    shape, edges = _rng(case["grammars"], 2), _rng(seed, 3)
    out = []
    for _ in range(case["queries"]):
        n = int(shape.integers(case["n_min"], case["n_max"] + 1))
        labels = int(shape.integers(2, 7))
        out.append((W.er_graph(n, OUT_DEGREE_ER, labels, edges), W.random_grammar(shape, labels, 3, 24)[2]))
    return out


def _pool(case):
    shape = _rng(case["grammars"], 4)
    return [W.random_grammar(shape, 8, 3, 32)[2] for _ in range(case["queries"])]


def _device_edges(g):
    return tuple(torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda() for a in (g.src, g.lbl, g.dst))


def _bracket_pairs(g, count, rng):
    """Pairs (x, z) joined by an edge o_i followed by an edge c_i: pairs of the Dyck-4 answer."""
    k = g.n_terminals // 2
    by_src = np.argsort(g.src, kind="stable")
    start = np.searchsorted(g.src[by_src], np.arange(g.n + 1))
    found = []
    for e in rng.permutation(g.m).tolist():
        if g.lbl[e] >= k:
            continue
        y = int(g.dst[e])
        for f in by_src[start[y]:start[y + 1]].tolist():
            if g.lbl[f] == g.lbl[e] + k:
                found.append((int(g.src[e]), int(g.dst[f])))
                break
        if len(found) == count:
            break
    return found


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "batch":
        state["ctx"] = cfpq.Context()
        state["queries"] = _batch(case, seed)
        return state
    if kind == "server":
        g = W.zipf_graph(case["n"], 8, int(seed))
        state["server"] = cfpq.Server(g, memory_budget=48 << 30)
        state["pool"] = _pool(case)
        return state
    g, r = _graph_and_rsm(case, seed)
    ctx = cfpq.Context()
    ctx.load_graph(g)
    ctx.load_rsm(r)
    state.update(ctx=ctx, rsm=r, n=g.n, n_terminals=g.n_terminals, edges=_device_edges(g))
    if kind == "sources":
        src = np.sort(_rng(seed, 5).choice(g.n, size=min(case["sources"], g.n), replace=False))
        state["sources"] = src.astype(np.uint32)
        start = int(r.box_start[r.start_box])
        state["rows"] = [(start, int(v)) for v in src]
    if kind == "paths":
        state["max_len"] = case["max_len"]
        state["pairs"] = _bracket_pairs(g, case["pairs"], _rng(seed, 6))
    return state


def _words(w):
    return w.view(np.int64)


def run(state):
    kind = state["kind"]
    if kind == "batch":
        ctx = state["ctx"]
        per, _ = ctx.batch_run(state["queries"])
        return {"answers": [_words(ctx.batch_reachable_words(q, r.start_box)) for q, (_, r) in
                            enumerate(state["queries"])],
                "iterations": np.array([s.iterations for s in per], dtype=np.int64)}
    if kind == "server":
        server = state["server"]
        tickets = [server.submit(r) for r in state["pool"]]
        while server.step() != (0, 0):
            pass
        answers = []
        for t, r in zip(tickets, state["pool"]):
            answers.append(_words(server.result_words(t, r.start_box)))
            server.release(t)
        return {"answers": answers}
    ctx = state["ctx"]
    if kind == "rsm":
        ctx.load_rsm(state["rsm"])
    else:
        ctx.load_graph_device(state["n"], state["n_terminals"], *state["edges"])
    if kind == "sources":
        st = ctx.run_sources(state["sources"])
        return {"rows": ctx.closure_rows(state["rows"]), "iterations": int(st.iterations)}
    st = ctx.run()
    if kind == "paths":
        edges, lengths, truncated = [], [], []
        for vs, vf in state["pairs"]:
            paths, cut = ctx.extract_paths(0, vs, vf, state["max_len"])
            truncated.append(cut)
            for p in paths:
                lengths.append(len(p))
                edges.extend(p)
        return {"edges": np.array(edges, dtype=np.int64).reshape(-1, 3), "lengths": np.array(lengths, dtype=np.int64),
                "truncated": np.array(truncated, dtype=np.int64), "iterations": int(st.iterations)}
    return {"answers": [_words(ctx.reachable_words(b)) for b in range(state["rsm"].n_boxes)],
            "iterations": int(st.iterations)}


def _closure_blocks(r):
    """Pairs of states joined by one or more transitions: the state blocks of the index that can hold a pair."""
    reach = np.zeros((r.n_states, r.n_states), dtype=bool)
    reach[r.tr_from, r.tr_to] = True
    for k in range(r.n_states):
        reach |= np.outer(reach[:, k], reach[k])
    return int(reach.sum())


def _matrix_bytes(n):
    return n * ((n + 63) // 64) * 8


def work(case):
    """Bytes of one pass: the edges read, the index (closure blocks and answers) written, and what is read back of
    it.  The operations have no closed form (a fixpoint whose length depends on the graph): counted as none."""
    kind = case["kind"]
    if kind == "batch":
        return {"bytes": sum(12 * OUT_DEGREE_ER * g.n + (_closure_blocks(r) + r.n_boxes + 1) * _matrix_bytes(g.n)
                             for g, r in _batch(case, 0)), "flops": 0}
    if kind == "server":
        m = _matrix_bytes(case["n"])
        return {"bytes": 12 * OUT_DEGREE_ZIPF * case["n"] + sum((_closure_blocks(r) + r.n_boxes + 1) * m for r in
                                                                _pool(case)), "flops": 0}
    r = {"rpq": W.abc_dfa_rsm, "cycles": W.anbn_rsm, "dyck": W.dyck_rsm}[case["query"]]()
    n = 2 * case["n"] if case["query"] == "cycles" else case["n"]
    edges = 12 * case["out_deg"] * n
    m = _matrix_bytes(n)
    if kind == "sources":
        # one row of every closure block per source at the least, and the sources' rows read back
        return {"bytes": edges + case["sources"] * (_closure_blocks(r) * m // n + r.n_states * n), "flops": 0}
    index = (_closure_blocks(r) + r.n_boxes) * m
    return {"bytes": edges + index + (0 if kind == "paths" else r.n_boxes * m), "flops": 0}


def exact(case, seed):
    """The answer by plain matrix products in 64 bits, where that is quick: pairs (x, y) with x -> y derivable,
    the least fixpoint of reach(start) = I, reach(to) |= reach(from) . label, answer = reach(final)."""
    if case["kind"] not in ("query", "rsm") or case["n"] > 512:
        return None
    g, r = _graph_and_rsm(case, seed)
    n = g.n
    term = np.zeros((g.n_terminals, n, n))
    term[g.lbl, g.src, g.dst] = 1.0
    answer = np.zeros((r.n_boxes, n, n))
    reach = np.zeros((r.n_states, n, n))
    reach[np.asarray(r.box_start)] = np.eye(n)
    while True:
        changed = True
        while changed:
            changed = False
            for f, kind, sym, to in zip(r.tr_from, r.tr_kind, r.tr_sym, r.tr_to):
                step = reach[f] @ (term[sym] if kind == W.TERM else answer[sym])
                new = ((reach[to] + step) > 0).astype(np.float64)
                if (new != reach[to]).any():
                    reach[to] = new
                    changed = True
        new_answer = np.zeros_like(answer)
        for s in range(r.n_states):
            if r.state_final[s]:
                b = r.state_box[s]
                new_answer[b] = np.maximum(new_answer[b], reach[s])
        if (new_answer == answer).all():
            break
        answer = new_answer
    pad = np.zeros((r.n_boxes, n, (n + 63) // 64 * 64), dtype=bool)
    pad[:, :, :n] = answer > 0
    words = np.packbits(pad, axis=2, bitorder="little").view(np.int64)
    return {"answers": [np.ascontiguousarray(words[b]) for b in range(r.n_boxes)], "iterations": None}
