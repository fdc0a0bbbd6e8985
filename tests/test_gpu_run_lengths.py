"""Short runs: below the generations that pay for an on-chip launch a run launches
each generation and takes no buffers; whatever the count, the results are those of
single generations, bit for bit (tolerance zero)."""
import gc

import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W

# the fewest generations on the chip: one cluster, rows of one warp and of several, one row per CTA, many
LEAST = [(100, 30, "nec", 0.9, 2), (100, 30, "exp", 0.5, 2), (100, 30, "bin", 0.5, 2), (150, 128, "bin", 0.5, 2),
         (300, 500, "nec", 0.9, 4), (100, 30, "exp", 0.9, 4), (64, 1000, "nec", 0.9, 5), (2000, 64, "nec", 0.1, 3),
         (5000, 30, "exp", 0.9, 5), (5000, 30, "exp", 0.5, 3), (1000, 30, "bin", 0.5, 4), (2000, 128, "bin", 0.5, 3),
         (300, 500, "bin", 0.5, 4), (150, 2000, "bin", 0.5, 4)]


@pytest.mark.parametrize("N,D,xo,cr,least", LEAST)
def test_fewest_generations_on_the_chip(N, D, xo, cr, least):
    kw = dict(F=0.5, CR=cr, xo=xo, obj="rosenbrock", bounds=W.BOXES["rosenbrock"], seed=D)
    for gens in (least - 1, least, least + 1):
        a = DE.Optimizer(N, D, **kw)
        held = len(DE._live_blocks)
        a.run(gens)
        assert (len(DE._live_blocks) > held) == (gens >= least)
        c = DE.Optimizer(N, D, **kw)
        for _ in range(gens):
            c.step()
        for u, v in zip(a.population(), c.population()):
            assert u.tobytes() == v.tobytes()
        assert a.stats() == c.stats()
        a.close()
        c.close()


@pytest.mark.parametrize("N,D", [(100, 30), (300, 500), (64, 3000)])
def test_a_run_without_a_graph_is_refused_under_capture(N, D):
    import torch
    kw = dict(obj="sphere", bounds=(-5.0, 5.0), seed=1)
    o, ref = DE.Optimizer(N, D, **kw), DE.Optimizer(N, D, **kw)
    o.run(3)
    o.synchronize()
    y = torch.zeros(4, device="cuda")
    graph = torch.cuda.CUDAGraph()
    gc.collect()                                 # a graph of an earlier test may not end while this one is captured
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=o.stream):
        y.add_(1)
        for call in (o.run, o.prepare_run):
            with pytest.raises(DE.DEError) as e:
                call(7)
            assert e.value.code == DE.DE_ECUDA
        y.add_(1)
    graph.replay()
    torch.cuda.synchronize()
    assert y.tolist() == [2.0] * 4
    o.run(7)                                     # the context goes on
    ref.run(10)
    for u, v in zip(o.population(), ref.population()):
        assert u.tobytes() == v.tobytes()
    o.close()
    ref.close()
