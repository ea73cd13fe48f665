"""Multiple-source runs whose work items span 64 to 1024 rows (they grow with the rows of
a level): one source, some, and every vertex, on graphs where few rows or nearly all are
reached, at sizes that leave a short last item.  The sources' rows equal the full run's
and the oracle's."""
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


@pytest.mark.parametrize("n,out_deg", [(65, 3), (1500, 5), (8200, 1), (8200, 6), (20011, 2), (34001, 2), (65536, 1)])
def test_sources_of_every_item_size(C, n, out_deg):
    g, r = W.rpq_abc(n=n, out_deg=out_deg, seed=n)
    rng = np.random.Generator(np.random.PCG64(n))
    few = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 12)]))
    want = oracle.worklist_words(g, r, sources=few)[0][few]
    with C.Context(no_single_cta=1) as ctx:
        ctx.load_graph(g)
        ctx.load_rsm(r)
        ctx.run()
        full = ctx.reachable_words(0)
        assert (full[few] == want).all()
        for src in (few[:1], few, np.arange(n)):
            ctx.run_sources(src)
            assert (ctx.reachable_words(0)[src] == full[src]).all()
