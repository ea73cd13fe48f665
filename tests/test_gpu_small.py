"""The single-CTA fixpoint at the edges of what it takes: one vertex, every row
width (2, 4, 6, 8 words), more boxes than a register mask holds, and states that
leave no room in shared memory for the plan's tables or for the graph's edges.
Answers and closure rows equal the multi-kernel path's, iterations too; answers
equal the oracle's."""
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


def _random(n, m, labels, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return W.Graph(n, labels, rng.integers(0, n, m, dtype=np.uint32), rng.integers(0, labels, m, dtype=np.uint32),
                   rng.integers(0, n, m, dtype=np.uint32))


def _many_boxes(k):
    """Box 0 reads boxes 1 .. k-1; box i reads a terminal or the box after it (box k - 1 nullable)."""
    tr, start, box, fin = [], [], [], []
    for b in range(k):
        q = 2 * b
        start.append(q)
        box += [b, b]
        fin.append(q + 1)
        tr.append((q, W.TERM, b % 2, q + 1))
        if b + 1 < k:
            tr.append((q, W.NONTERM, b + 1, q + 1))
    fin.append(start[-1])
    return W.make_rsm(2 * k, start, box, fin, tr)


CASES = [
    ("one vertex", lambda: (_random(1, 4, 2, 1), W.anbn_rsm())),
    ("two vertices", lambda: (_random(2, 6, 2, 2), W.anbn_rsm())),
    ("no edges", lambda: (_random(70, 0, 2, 3), W.anbn_rsm())),
    ("2 words", lambda: (_random(128, 300, 2, 4), W.anbn_rsm())),
    ("4 words", lambda: (_random(129, 300, 2, 5), W.anbn_rsm())),
    ("6 words", lambda: (_random(300, 700, 2, 6), W.anbn_rsm())),
    ("8 words", lambda: (_random(500, 1500, 1, 7), W.make_rsm(2, [0], [0, 0], [1], [(0, 0, 0, 1), (1, 0, 0, 1)]))),
    ("70 boxes", lambda: (_random(9, 20, 2, 8), _many_boxes(70))),
    ("edges beside the state in global memory", lambda: (W.rpq_abc(n=225, out_deg=4, seed=9)[0], W.abc_dfa_rsm())),
    ("tables in global memory", lambda: (W.rpq_abc(n=229, out_deg=3, seed=10)[0], W.abc_dfa_rsm())),
    ("dense labels in global memory", lambda: (_random(128, 150000, 8, 11), W.anbn_rsm())),
    ("Dyck-4", lambda: W.dyck_zipf(110, seed=12)),
]


@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_single_cta_equals_multi_kernel(C, name, make):
    g, r = make()
    with C.Context() as a, C.Context(no_single_cta=1) as b:
        st = []
        for ctx in (a, b):
            ctx.load_graph(g)
            ctx.load_rsm(r)
            st.append(ctx.run())
        assert st[0].gpu_launches == 1 and st[1].gpu_launches > 1
        assert st[0].iterations == st[1].iterations
        assert st[0].edges_added == st[1].edges_added
        want = oracle.worklist(g, r)
        for box in range(r.n_boxes):
            assert (a.reachable_bits(box) == want[box]).all()
            assert (b.reachable_bits(box) == want[box]).all()
        rows = [(s, v) for s in range(r.n_states) for v in range(0, g.n, max(1, g.n // 7))]
        assert (a.closure_rows(rows) == b.closure_rows(rows)).all()
