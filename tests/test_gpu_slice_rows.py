"""Column slices whose rows do not fill the last stripe of threads (a stripe is 512
rows, slices of up to 2048 rows give each thread two or four): the threads without a
row of their own must leave the slice and the list of edges behind it alone.  Vertex 0,
the row they read instead, gains bits in nearly every sweep: it lies on one long cycle,
with a dozen edges out (all but four of them listed) and a dozen in.  Answers equal the
oracle's, in every one of several runs."""
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


def _rsm(members):
    """One cyclic component of `members` states q_0 -a-> q_1 -a-> ... -a-> q_0, q_0 -a-> q_0 too; q_0 final and a final
    state behind it."""
    if members == 1:
        return W.make_rsm(2, [0], [0, 0], [1], [(0, T, 0, 1), (1, T, 0, 1)])
    tr = [(s, T, 0, (s + 1) % members) for s in range(members)] + [(0, T, 0, 0), (members - 1, T, 1, members)]
    return W.make_rsm(members + 1, [0], [0] * (members + 1), [0, members], tr)


def _graph(n):
    """A cycle through seven eighths of the vertices with hub 0; the others have edges into it, out of it, or none."""
    rng = np.random.Generator(np.random.PCG64(n))
    k = n - n // 8
    rest = np.arange(k, n)
    hub = rng.integers(0, k, 12)
    s = np.concatenate([np.arange(k), np.zeros(12, int), hub, rest[::3], rng.integers(0, k, len(rest[1::3])),
                        rng.integers(0, n, 8)])
    d = np.concatenate([(np.arange(k) + 1) % k, hub[::-1], np.zeros(12, int), rng.integers(0, k, len(rest[::3])), rest[1::3],
                        rng.integers(0, n, 8)])
    lbl = np.zeros(len(s), int)
    lbl[-8:] = 1
    o = rng.permutation(len(s))
    return W.Graph(n, 2, s[o].astype(np.uint32), lbl[o].astype(np.uint32), d[o].astype(np.uint32))


# rows = members * n: below one stripe, just past one, two and three, and full ones
@pytest.mark.parametrize("members,n", [(1, 511), (1, 512), (1, 513), (1, 600), (1, 1000), (1, 1023), (1, 1025), (1, 1100),
                                       (1, 1537), (1, 2047), (2, 257), (2, 550), (2, 700), (2, 1023), (4, 129), (4, 300)])
def test_ragged_last_stripe(C, members, n):
    g, r = _graph(n), _rsm(members)
    want = oracle.worklist_words(g, r)[0]
    with C.Context(no_single_cta=1) as ctx:
        ctx.load_graph(g)
        ctx.load_rsm(r)
        for _ in range(3):
            st = ctx.run()
            assert (ctx.reachable_words(0) == want).all()
            # (closed in one pass of the component's level: no pass repeats)
            assert st.rounds <= 2 * (r.n_states + 1)
