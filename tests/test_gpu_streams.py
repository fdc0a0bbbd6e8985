"""Runs of several contexts queued on streams of their own at once, from one thread
and from several: kernels whose rows wait for one another, one after the other or
beside others, end with the results of a run alone (bit for bit)."""
import threading

import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W

# populations of a CTA per SM that fill its shared memory, binomial rows of several warps, one cluster, a large one
KINDS = [dict(N=1024, D=1000, xo="nec", obj="rastrigin"), dict(N=1000, D=900, xo="exp", obj="ackley"),
         dict(N=600, D=500, xo="bin", obj="griewank"), dict(N=100, D=30, xo="nec", obj="sphere"),
         dict(N=300, D=3000, xo="nec", obj="rosenbrock")]


def _make(k, seed):
    return DE.Optimizer(F=0.5, CR=0.9, bounds=W.BOXES[KINDS[k]["obj"]], seed=seed, **KINDS[k])


def _out(o):
    o.synchronize()
    res = [v.tobytes() for v in o.population()] + [o.stats()]
    o.close()
    return res


@pytest.mark.parametrize("threads", [False, True])
@pytest.mark.parametrize("which", [(0, 0), (0, 1), (2, 2, 0), (0, 1, 2, 3, 4)])
def test_runs_side_by_side(which, threads):
    counts = (30, 5, 100, 1, 64) * 3
    alone = []
    for n, k in enumerate(which):
        o = _make(k, n)
        for c in counts:
            o.run(c)
        alone.append(_out(o))
    opts = [_make(k, n) for n, k in enumerate(which)]
    for o in opts:
        for c in set(counts):
            o.prepare_run(c)
    if threads:
        todo = [threading.Thread(target=lambda o=o: [o.run(c) for c in counts]) for o in opts]
        for t in todo:
            t.start()
        for t in todo:
            t.join()
    else:
        for c in counts:
            for o in opts:
                o.run(c)
    for o, want in zip(opts, alone):
        assert _out(o) == want
