"""Blocks that read no closure row (product edges, CSR rows of pure-terminal
blocks): rows owned by a warp and by a CTA (n up to and above 8192), one and
two labels in the block read, hub vertices with hundreds of edges, nullable
boxes, graphs without edges of a label, more sources than the packed ones.
The answers equal the oracle's, and every mode takes as many iterations."""
import numpy as np
import pytest

import oracle
from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


def _graph(n, m, labels, seed, hub=True, skip=None):
    rng = np.random.Generator(np.random.PCG64(seed))
    src, dst = rng.integers(0, n, m), rng.integers(0, n, m)
    lbl = rng.integers(0, labels, m)
    if hub:  # a vertex with an edge to every 7th vertex
        k = n // 7
        src[:k], dst[:k] = n // 2, np.arange(k) * 7
    if skip is not None:
        lbl[lbl == skip] = 0
    return W.Graph(n, labels, src.astype(np.uint32), lbl.astype(np.uint32), dst.astype(np.uint32))


def _rsm(kind):
    T, N = W.TERM, W.NONTERM
    if kind == "two labels":  # S -> a | S (b | c): the block read joins two labels
        return W.make_rsm(3, [0], [0] * 3, [2], [(0, T, 0, 2), (0, N, 0, 1), (1, T, 1, 2), (1, T, 2, 2)])
    if kind == "nullable":    # S -> eps | a S b
        return W.make_rsm(4, [0], [0] * 4, [0, 3], [(0, T, 0, 1), (1, N, 0, 2), (2, T, 1, 3)])
    if kind == "two boxes":   # A -> a B c | b,  B -> b | A a
        return W.make_rsm(8, [0, 5], [0, 0, 0, 0, 0, 1, 1, 1], [4, 7],
                          [(0, T, 0, 1), (1, N, 1, 2), (2, T, 2, 4), (0, T, 1, 4),
                           (5, T, 1, 7), (5, N, 0, 6), (6, T, 0, 7)])
    # "many sources": q0 -S-> u_i -l-> F for twenty states u_i
    tr = [(0, T, 0, 1)]
    for i in range(20):
        tr += [(0, N, 0, 2 + i), (2 + i, T, i % 3, 1)]
    return W.make_rsm(22, [0], [0] * 22, [1], tr)


@pytest.mark.parametrize("kind", ["two labels", "nullable", "two boxes", "many sources"])
@pytest.mark.parametrize("n,m,skip", [(600, 900, None), (777, 800, 2), (8192, 12000, None), (8193, 12000, None),
                                      (17000, 20000, 1)])
def test_expanded_blocks(C, kind, n, m, skip):
    g, r = _graph(n, m, 3, n + len(kind), skip=skip), _rsm(kind)
    out = []
    for opts in ({"closure_mode": C.CFPQ_CLOSURE_BITPACKED}, {}, {"closure_mode": C.CFPQ_CLOSURE_TC_FP4}):
        with C.Context(no_single_cta=1, **opts) as ctx:
            ctx.load_graph(g)
            ctx.load_rsm(r)
            st = ctx.run()
            out.append((st.iterations, st.edges_added, [ctx.reachable_words(b) for b in range(r.n_boxes)]))
    for it, added, words in out[1:]:
        assert it == out[0][0] and added == out[0][1]
        assert all((a == b).all() for a, b in zip(words, out[0][2]))
    if n <= 777 or kind != "many sources":  # (20 s and more on the larger graphs)
        want = oracle.worklist_words(g, r)
        assert all((a == want[b]).all() for b, a in enumerate(out[0][2]))
