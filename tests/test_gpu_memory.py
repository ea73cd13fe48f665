"""Device memory at its limits: what a run needs, and what a context does after a call
that ran out of memory.  The allocator callbacks count the bytes held and can refuse."""
import ctypes

import numpy as np
import pytest

from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu
T = W.TERM


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


class Memory:
    """Allocator callbacks over torch's allocator: bytes held, their peak, and a rule that refuses requests."""

    def __init__(self, C):
        import torch
        torch.cuda.init()
        self.held = self.peak = self.calls = 0
        self.refuse = lambda call, nbytes: False

        def alloc(nbytes, stream, user):
            self.calls += 1
            if self.refuse(self.calls, nbytes):
                return None
            try:
                p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, stream or 0)
            except Exception:
                return None
            self.held += nbytes
            self.peak = max(self.peak, self.held)
            return p

        def free(ptr, nbytes, stream, user):
            torch.cuda.caching_allocator_delete(ptr)
            self.held -= nbytes

        self.options = {"alloc": C.cfpq_alloc_fn(alloc), "free": C.cfpq_free_fn(free)}

    def context(self, C, **opts):
        import torch
        return C.Context(use_torch=False, stream=torch.cuda.current_stream().cuda_stream, **self.options, **opts)


def _plus():
    return W.make_rsm(2, [0], [0, 0], [1], [(0, T, 0, 1), (1, T, 0, 1)])


def _dense(n, m, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return W.Graph(n, 3, rng.integers(0, n, m, dtype=np.uint32), rng.integers(0, 3, m, dtype=np.uint32),
                   rng.integers(0, n, m, dtype=np.uint32))


def _run(ctx, g, r):
    ctx.load_graph(g)
    ctx.load_rsm(r)
    ctx.run()
    return [ctx.reachable_words(b) for b in range(r.n_boxes)]


def test_column_slices_need_no_memory_per_edge(C):
    """A run with column slices fits where the row gather's run of the same query does (its round cap is never
    reached), up to the work lists (1 MiB here); an edge list of its own would be 4 MiB."""
    g, r = _dense(1500, 1 << 20, 1), _plus()
    mem = Memory(C)
    with mem.context(C, max_rounds=1 << 19) as ctx:
        want = _run(ctx, g, r)
    with Memory(C).context(C, memory_budget=mem.peak + (1 << 20)) as ctx:
        for _ in range(2):  # (the second load overwrites the edge copy that holds the first one's list)
            assert (_run(ctx, g, r)[0] == want[0]).all()
    g2 = _dense(1500, 9000, 2)
    with mem.context(C, max_rounds=1 << 19) as ctx:
        want2 = _run(ctx, g2, r)
    with mem.context(C) as ctx:
        for a, w in ((g, want), (g2, want2), (g, want)):
            assert (_run(ctx, a, r)[0] == w[0]).all()
        bad = W.Graph(g.n, g.n_terminals, g.src, g.lbl, np.where(np.arange(g.m) == g.m - 1, g.n, g.dst).astype(np.uint32))
        with pytest.raises(C.CfpqError):  # a load that is refused has overwritten the edge copy too
            ctx.load_graph(bad)
        assert (_run(ctx, g2, r)[0] == want2[0]).all()


def _refused_runs(C, first, r, call, opts):
    """For every allocation that `call` makes on a context that ran `first`: refuse it alone, let `call` fail, and yield
    the context, its memory and whether it failed; ends after the first call that needed no more allocations."""
    for k in range(1, 200):
        mem = Memory(C)
        with mem.context(C, **opts) as ctx:
            _run(ctx, first, r)
            stop = [None]
            try:
                call(ctx, mem, lambda: (stop.__setitem__(0, mem.calls + k),
                                        setattr(mem, "refuse", lambda i, b: i == stop[0])))
                failed = False
            except C.CfpqError as e:
                assert e.status == C.CFPQ_ERR_OUT_OF_MEMORY
                failed = True
            refused = mem.calls >= stop[0]
            mem.refuse = lambda i, b: False
            yield ctx, failed
        if not refused:
            return
    assert False, "more allocations than expected"


RUNS = [("column slices", lambda: (_dense(700, 1500, 3), _dense(1900, 60000, 4), _plus()), {"no_single_cta": 1}),
        ("single CTA", lambda: (_dense(60, 100, 5), _dense(200, 400, 6), _plus()), {}),
        ("tiles", lambda: (W.dyck_zipf(2100, seed=1)[0], W.dyck_zipf(2600, seed=2)[0], W.dyck_rsm(2)), {"no_autotune": 1})]


@pytest.mark.parametrize("name,make,opts", RUNS, ids=[x[0] for x in RUNS])
def test_run_again_after_a_run_out_of_memory(C, name, make, opts):
    """A run of a larger graph whose k-th allocation is refused fails; the same run again gives the graph's answer,
    and so does the smaller graph afterwards."""
    first, then, r = make()
    with C.Context(**opts) as ctx:
        want = [_run(ctx, g, r) for g in (first, then)]

    def call(ctx, mem, refuse_from_here):
        ctx.load_graph(then)
        refuse_from_here()
        ctx.run()

    fails = 0
    for ctx, failed in _refused_runs(C, first, r, call, opts):
        fails += failed
        ctx.run()
        assert all((ctx.reachable_words(b) == want[1][b]).all() for b in range(r.n_boxes))
        ctx.load_graph(first)
        ctx.run()
        assert all((ctx.reachable_words(b) == want[0][b]).all() for b in range(r.n_boxes))
    assert fails >= 5


@pytest.mark.parametrize("after", ["the first graph", "the refused graph"])
@pytest.mark.parametrize("name,make,opts", RUNS[:2], ids=[x[0] for x in RUNS[:2]])
def test_load_again_after_a_load_out_of_memory(C, name, make, opts, after):
    """A load of a larger graph with more labels whose k-th allocation is refused fails; the graph loaded next is
    staged and run as in a new context, also when it has the shape of the one before the failure."""
    first, then, r = make()
    first, then = (W.Graph(g.n, k, g.src, g.lbl, g.dst) for g, k in ((first, 3), (then, 9)))
    g = first if after == "the first graph" else then
    with C.Context(**opts) as ctx:
        want = _run(ctx, g, r)

    def call(ctx, mem, refuse_from_here):
        refuse_from_here()
        ctx.load_graph(then)

    fails = 0
    for ctx, failed in _refused_runs(C, first, r, call, opts):
        fails += failed
        ctx.load_graph(g)
        ctx.run()
        assert all((ctx.reachable_words(b) == want[b]).all() for b in range(r.n_boxes))
    assert fails >= 5


def test_tuning_reports_out_of_memory(C):
    """The autotuner's product of two 8192 x 8192 matrices takes 64 MiB of FP8 bytes a side: without them it keeps the
    built-in choices and says why."""
    mem = Memory(C)
    mem.refuse = lambda i, b: b == 64 << 20
    with mem.context(C) as ctx:
        t = ctx.tune(force=True)
    assert t.tuned == 0 and t.probe_status == C.CFPQ_ERR_OUT_OF_MEMORY
    assert t.gather_gbs > 0  # (the probe query before it ran)
    with C.Context() as ctx:
        assert ctx.tune(force=True).tuned == 1
