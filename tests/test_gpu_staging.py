"""Graph staging: the one-CTA kernel and the grid-wide ones build the same
adjacency.  Sizes on both sides of the kernel's limits (16384 edges, 12288 counters),
repeated edges, rows longer than the 256 edges up to which repeats are dropped, one
vertex, no edges, edges out of range.  The query reads each label alone, so the
answers are the edges themselves."""
import numpy as np
import pytest

from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


def _rsm(labels):  # box b -> terminal b
    return W.make_rsm(2 * labels, [2 * b for b in range(labels)], [b // 2 for b in range(2 * labels)],
                      [2 * b + 1 for b in range(labels)], [(2 * b, W.TERM, b, 2 * b + 1) for b in range(labels)])


@pytest.mark.parametrize("n,labels,m", [(1, 1, 0), (1, 2, 5), (70, 3, 0), (200, 3, 600), (300, 1, 16384), (300, 1, 16385),
                                        (4096, 3, 9000), (4097, 3, 9000), (5, 2, 12000), (12288, 1, 16000),
                                        (12289, 1, 16000)])
@pytest.mark.parametrize("device", [False, True])
def test_edges(C, n, labels, m, device):
    import torch
    rng = np.random.Generator(np.random.PCG64(n + m))
    s, d = rng.integers(0, n, m, dtype=np.uint32), rng.integers(0, n, m, dtype=np.uint32)
    l = rng.integers(0, labels, m, dtype=np.uint32)
    if m > 100:
        s[: m // 4], l[: m // 4] = n // 2, 0   # one long row
        s[-40:], l[-40:], d[-40:] = s[:40], l[:40], d[:40]
    want = np.zeros((labels, n, (n + 63) // 64), dtype=np.uint64)
    np.bitwise_or.at(want, (l, s, d >> 6), np.uint64(1) << (d & 63).astype(np.uint64))
    with C.Context() as ctx:
        if device:
            ctx.load_graph_device(n, labels, *(torch.from_numpy(a.view(np.int32)).cuda() for a in (s, l, d)))
        else:
            ctx.load_graph(W.Graph(n, labels, s, l, d))
        ctx.load_rsm(_rsm(labels))
        ctx.run()
        for b in range(labels):
            assert (ctx.reachable_words(b) == want[b]).all()


@pytest.mark.parametrize("bad", [(7, 0, 0), (0, 2, 0), (0, 0, 7), (0xFFFFFFFF, 0, 0)])
def test_out_of_range(C, bad):
    s, l, d = (np.array([1, 2, v], dtype=np.uint32) for v in bad)
    l[:2] = 0
    with C.Context() as ctx:
        with pytest.raises(C.CfpqError) as e:
            ctx.load_graph(W.Graph(7, 2, s, l, d))
        assert e.value.status == C.CFPQ_ERR_INVALID_ARG
