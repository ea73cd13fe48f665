"""Vertices with far more edges than the others: rows that the gather takes untested (more
than 32 edges), with and without a changed row among their neighbours, and slices whose
rows have more edges past the fourth than their list holds.  Rows of every width; answers
equal the oracle's at sampled source vertices, the hubs and the chain among them."""
import numpy as np
import pytest

import oracle
from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu
T = W.TERM


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


RSMS = {
    "plus": W.make_rsm(2, [0], [0, 0], [1], [(0, T, 0, 1), (1, T, 0, 1)]),
    # (ab)*: two states in one component
    "pair": W.make_rsm(2, [0], [0, 0], [0], [(0, T, 0, 1), (1, T, 1, 0)]),
    # a* b through a second label, then an acyclic tail
    "tail": W.make_rsm(3, [0], [0, 0, 0], [2], [(0, T, 0, 0), (0, T, 1, 1), (1, T, 0, 2)]),
}


def _graph(n, degs, seed):
    """A chain of 40 vertices of alternating labels (each edge twice, as a and as b), and hubs
    of the given degrees: half their edges anywhere, the first one into the chain's end."""
    rng = np.random.Generator(np.random.PCG64(seed))
    p = rng.permutation(n)
    s, l, d = [], [], []
    for i in range(min(40, n // 2) - 1):
        for lab in (0, 1):
            s.append(p[i]), l.append(lab), d.append(p[i + 1])
    hubs = []
    for k, deg in enumerate(degs):
        h = p[n - 1 - k]
        hubs.append(h)
        to = rng.choice(n, size=min(deg, n), replace=False)
        to[0] = p[min(40, n // 2) // 2]
        for lab in (0, 1) if k % 2 else (0,):
            s += [h] * len(to)
            l += [lab] * len(to)
            d += to.tolist()
    g = W.Graph(n, 2, np.array(s, np.uint32), np.array(l, np.uint32), np.array(d, np.uint32))
    return g, hubs + [int(v) for v in p[:6]]


@pytest.mark.parametrize("rsm", sorted(RSMS))
@pytest.mark.parametrize("n,degs", [(600, [32, 33, 600]), (1000, [250, 5]), (1000, [260] * 3), (2040, [2000] * 3),
                                    (2060, [31, 33, 2000]), (8200, [32, 33, 255, 256, 257, 3000]),
                                    (17000, [511, 512, 513, 9000]), (40000, [40, 256, 257, 30000])])
def test_hub_rows(C, rsm, n, degs):
    (g, src), r = _graph(n, degs, n + len(degs)), RSMS[rsm]
    src = sorted({int(v) for v in src} | {0, n - 1})
    want = oracle.worklist(g, r, sources=src)[0]
    for opts in ({}, {"max_rounds": 1 << 19}):  # (the cap keeps cyclic components on the gather)
        with C.Context(no_single_cta=1, **opts) as ctx:
            ctx.load_graph(g)
            ctx.load_rsm(r)
            ctx.run()
            full = ctx.reachable_words(0)
            got = np.unpackbits(full[src].view(np.uint8), axis=1, bitorder="little")[:, :n].astype(bool)
            assert (got == want[src]).all()
            ctx.run_sources(src)
            assert (ctx.reachable_words(0)[src] == full[src]).all()
