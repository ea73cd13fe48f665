"""Rows of thousands of edges, which the CSR gather's whole CTA shares: about the 512 edges where
that begins, several in an item, more than an item lists (dense graphs, two such sources a
row), and with rows of few edges beside them in a warp.  Answers equal the oracle's at sampled
source vertices; rows changed are counted once a pass."""
import numpy as np
import pytest

import oracle
from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu
T = W.TERM
# (a | b)+ c?: two sources a block, one component over another
RSM = W.make_rsm(3, [0], [0, 0, 0], [1, 2],
                 [(s, T, lab, 1) for s in (0, 1) for lab in (0, 1)] + [(1, T, 2, 2)])


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


def _graph(n, hubs, degs, seed):
    """A chain of 50 vertices, vertices of one or two edges, and `hubs` neighbouring vertices of
    each degree in `degs` under every label."""
    rng = np.random.Generator(np.random.PCG64(seed))
    s, l, d = [np.arange(49)], [np.arange(49) % 2], [np.arange(1, 50)]
    few = rng.integers(50, n, n // 4)
    s.append(few), l.append(rng.integers(0, 3, len(few))), d.append(rng.integers(0, n, len(few)))
    rows = 60 + np.arange(hubs * len(degs))
    assert rows[-1] < n
    for i, v in enumerate(rows):
        for lab in range(3):
            to = rng.choice(n, size=min(n, degs[i % len(degs)]), replace=False)
            s.append(np.full(len(to), v)), l.append(np.full(len(to), lab)), d.append(to)
    g = W.Graph(n, 3, *(np.concatenate(a).astype(np.uint32) for a in (s, l, d)))
    return g, sorted({0, 20, 49, 60, 61, int(rows[-1]), n - 1} | set(rng.integers(0, n, 4).tolist()))


@pytest.mark.parametrize("n,hubs,degs", [(600, 80, [600]), (700, 3, [511, 512, 513]), (1030, 2, [1000, 2]),
                                         (2100, 70, [530]), (5000, 2, [511, 512, 513, 768, 769, 4999]),
                                         (9000, 3, [9000, 5]), (20000, 2, [600, 20000]), (40000, 2, [40000, 513])])
def test_shared_hubs(C, n, hubs, degs):
    g, src = _graph(n, hubs, degs, n + hubs)
    want = oracle.worklist(g, RSM, sources=src)[0]
    for opts in ({"max_rounds": 1 << 19}, {"max_rounds": 1 << 19, "loop_mode": C.CFPQ_LOOP_HOST}, {}):
        with C.Context(no_single_cta=1, **opts) as ctx:
            ctx.load_graph(g)
            ctx.load_rsm(RSM)
            st = ctx.run()
            assert st.rows_changed <= st.rounds * 4 * n  # (blocks C[0, 1], C[0, 2], C[1, 1], C[1, 2])
            full = ctx.reachable_words(0)
            got = np.unpackbits(full[src].view(np.uint8), axis=1, bitorder="little")[:, :n].astype(bool)
            assert (got == want[src]).all()
            ctx.run_sources(src)
            assert (ctx.reachable_words(0)[src] == full[src]).all()


@pytest.mark.parametrize("n", [1030, 5000])
def test_reloads_change_the_variant(C, n):
    """One context, graphs of one shape with and without such rows in turn."""
    import torch
    few, src = _graph(n, 2, [400, 3], 1)
    many, src2 = _graph(n, 2, [1000, 3], 2)
    src = sorted(set(src) | set(src2))
    with C.Context(no_single_cta=1, max_rounds=1 << 19) as ctx:
        ctx.load_rsm(RSM)
        for i, g in enumerate((few, many, few, many, many)):
            if i % 2:
                e = [torch.from_numpy(a.view(np.int32)).cuda() for a in (g.src, g.lbl, g.dst)]
                ctx.load_graph_device(g.n, g.n_terminals, *e)
            else:
                ctx.load_graph(g)
            ctx.run()
            got = np.unpackbits(ctx.reachable_words(0)[src].view(np.uint8), axis=1, bitorder="little")[:, :n]
            assert (got.astype(bool) == oracle.worklist(g, RSM, sources=src)[0][src]).all()
