"""A graph loaded in the middle of a column-sharded run ends that run: its passes would
mix the two graphs' buffers.  Stepping or applying is refused until the run is begun
again, which gives the new graph's answer."""
import ctypes

import pytest

from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


@pytest.mark.parametrize("how", ["host", "device", "noalloc"])
@pytest.mark.parametrize("query", ["rpq", "dyck"])
def test_load_ends_a_sharded_run(C, query, how):
    import torch
    make = (lambda s: W.rpq_abc(n=1500, out_deg=4, seed=s)) if query == "rpq" else (lambda s: W.dyck_zipf(1500, seed=s))
    (g1, r), (g2, _) = make(1), make(2)
    k = min(g1.m, g2.m)  # (no more edges than the first graph: the load that allocates nothing takes it)
    g2 = W.Graph(g2.n, g2.n_terminals, g2.src[:k], g2.lbl[:k], g2.dst[:k])
    with C.Context(no_single_cta=1) as ctx:
        ctx.load_graph(g2)
        ctx.load_rsm(r)
        ctx.run()
        want = ctx.reachable_words(0)
    with C.Context(no_single_cta=1) as ctx:
        e = C.ColumnShardEngine(ctx, g1, r)
        e.begin(0, 1536)
        full = e.step()
        dev = [torch.from_numpy(a.astype("int32")).cuda() for a in (g2.src, g2.lbl, g2.dst)]
        if how == "host":
            ctx.load_graph(g2)
        elif how == "device":
            ctx.load_graph_device(g2.n, g2.n_terminals, *dev)
        else:
            p = [ctypes.c_void_p(a.data_ptr()) for a in dev]
            assert ctx.lib.cfpq_load_graph_device_noalloc(ctx.h, g2.n, g2.n_terminals, g2.m, *p) == C.CFPQ_OK
        for call in (e.step, lambda: e.apply(full)):
            with pytest.raises(C.CfpqError) as err:
                call()
            assert err.value.status == C.CFPQ_ERR_STATE
        e.begin(0, 1536)
        while not e.apply(e.step()):
            pass
        assert (ctx.reachable_words(0) == want).all()
