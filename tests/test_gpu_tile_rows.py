"""The rows and inner rows a tile job keeps: graphs on which most rows of the
label matrix are empty, most output rows are full at once, or the new edges
lead to rows that were never written; sizes on both sides of the units of the
listing kernels (64 rows, 8 x n / 4096 rows) and of the tiles (256 rows).
Every mode gives the bit-packed answer in as many iterations; the smallest
size is compared with the oracle too."""
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


def _brackets(n, src, mid, dst, k, rng, count):
    """Edges x -o_i-> y -c_i-> z with x, y, z drawn from the given vertices."""
    x, y, z = (rng.choice(v, count) for v in (src, mid, dst))
    i = rng.integers(0, k, count)
    s, l, d = np.concatenate([x, y]), np.concatenate([i, k + i]), np.concatenate([y, z])
    return W.Graph(n, 2 * k, s.astype(np.uint32), l.astype(np.uint32), d.astype(np.uint32))


def _graph(shape, n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    v = np.arange(n)
    if shape == "few rows":        # 40 vertices start every path: the other rows stay empty
        few = rng.choice(n, 40, replace=False)
        return _brackets(n, few, few, np.concatenate([few, v[: n // 2]]), 2, rng, 4 * n)
    if shape == "full rows":       # dense enough that the answer fills up within a few iterations
        return _brackets(n, v[: n // 2], v, v[: n // 2], 1, rng, 5 * n)
    return _brackets(n, v[: n // 3], v[n // 3:], v, 3, rng, 3 * n)  # "dead ends": most targets start nothing


@pytest.mark.parametrize("shape", ["few rows", "full rows", "dead ends"])
@pytest.mark.parametrize("n", [2048, 4097, 8191])
def test_every_mode_equals_bitpacked(C, shape, n):
    g = _graph(shape, n, n)
    r = W.dyck_rsm(g.n_terminals // 2)
    answers, iters, tiles = [], [], []
    for opts in ({"closure_mode": C.CFPQ_CLOSURE_BITPACKED}, {}, {"tile_ratio": 4096},
                 {"closure_mode": C.CFPQ_CLOSURE_TC_FP8}, {"closure_mode": C.CFPQ_CLOSURE_TC_FP4}):
        with C.Context(**opts) as ctx:
            ctx.load_graph(g)
            ctx.load_rsm(r)
            st = ctx.run()
            answers.append(ctx.reachable_words(0))
            iters.append(st.iterations)
            tiles.append(st.tile_mmas)
    for a, it in zip(answers[1:], iters[1:]):
        assert (a == answers[0]).all() and it == iters[0]
    assert tiles[0] == 0 and tiles[3] > 0 and tiles[4] > 0
    if n == 2048:
        assert (answers[0] == oracle.worklist_words(g, r)[0]).all()
