"""Rows the gather visits: every row width (1 to 16 vectors a lane), items of 64
to 1024 rows, rows without edges, hub rows, more sources than the packed ones, and
multiple-source runs (items without a reached row).  Answers equal the oracle's at
sampled source vertices; a multiple-source run's rows equal the full run's."""
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


def _rsm(kind):
    if kind == "wide":   # q0 -l-> u_i -l'-> F through twenty states, and u_0 -a-> u_0
        tr = [(2, T, 0, 2)]
        for i in range(20):
            tr += [(0, T, i % 3, 2 + i), (2 + i, T, (i + 1) % 3, 1)]
        return W.make_rsm(22, [0], [0] * 22, [1], tr)
    if kind == "loop":   # a (b | c)* a: one cyclic level over another
        return W.make_rsm(3, [0], [0] * 3, [2], [(0, T, 0, 1), (1, T, 1, 1), (1, T, 2, 1), (1, T, 0, 2)])
    return W.dyck_rsm(1)


def _graph(n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    m = n + n // 4
    s, d, l = rng.integers(0, n // 2 + 1, m), rng.integers(0, n, m), rng.integers(0, 3, m)  # the upper half has no edges
    s[:70], l[:70] = n // 3, 0   # hubs: 70 edges of one label, 12 of another
    s[70:82], l[70:82] = n // 4, 1
    return W.Graph(n, 3, s.astype(np.uint32), l.astype(np.uint32), d.astype(np.uint32))


@pytest.mark.parametrize("kind", ["wide", "loop", "dyck"])
@pytest.mark.parametrize("n", [130, 4200, 8200, 16400, 33000])
def test_rows_with_work(C, kind, n):
    g, r = _graph(n, n), _rsm(kind)
    src = sorted({0, 1, n // 3, n // 4, n // 2, n - 1} | set(np.random.Generator(np.random.PCG64(n)).integers(0, n, 6).tolist()))
    want = oracle.worklist(g, r, sources=src)[0] if kind != "dyck" else oracle.worklist(g, r)[0] if n <= 4200 else None
    for opts in ({}, {"max_rounds": 1 << 19}):  # (the cap keeps cyclic components on the gather)
        with C.Context(no_single_cta=1, **opts) as ctx:
            ctx.load_graph(g)
            ctx.load_rsm(r)
            it = ctx.run().iterations
            full = ctx.reachable_words(0)
            got = np.unpackbits(full[src].view(np.uint8), axis=1, bitorder="little")[:, :n].astype(bool)
            if want is not None:
                assert (got == want[src]).all()
            st = ctx.run_sources(src)
            assert (ctx.reachable_words(0)[src] == full[src]).all()
            assert st.iterations <= it
