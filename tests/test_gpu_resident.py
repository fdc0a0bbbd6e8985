"""Whole runs in one launch (gen_resident.cuh; gen_cluster.cu for up to 248 rows
of D <= 128) against one launch per generation.

de_run of a population that fits on the chip makes many generations in one
launch; de_step, and de_run under de_set_kernel(1), launch each generation.
Every value is summed in the same order, so populations, fitness, best and
counters are equal bit for bit (tolerance zero).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W

# edges: the smallest N, one row per CTA and several, a partial last CTA, more
# than 32 rows per CTA (several barrier words), rows of one warp / one slot,
# D % 4 != 0, two slots per thread, the longest rows of the kernel
SHAPES = [(4, 1), (5, 3), (8, 128), (9, 4), (100, 30), (151, 127), (153, 128), (248, 33), (249, 33), (300, 500), (457, 1001), (1024, 1000), (301, 1029),
          (160, 2047), (5000, 30), (4864, 129), (4865, 130), (9000, 61)]


def _state(opt):
    x, f = opt.population()
    bx, bf, bi, bg = opt.best()
    s = opt.stats()
    return x, f, bx, np.float64(bf), bi, bg, s["generation"], s["accepts"], s["masked_genes"], s["best_gen"]


def _same(a, b):
    for u, v in zip(a, b):
        assert np.asarray(u).tobytes() == np.asarray(v).tobytes()


def _pair(N, D, **kw):
    a, b = DE.Optimizer(N, D, **kw), DE.Optimizer(N, D, **kw)
    b.set_kernel(1)
    return a, b


@pytest.mark.parametrize("xo", ["nec", "exp", "bin"])
@pytest.mark.parametrize("N,D", SHAPES)
def test_run_equals_steps(N, D, xo):
    obj = ("sphere", "rastrigin", "ackley", "rosenbrock", "griewank", "elliptic")[(N + D) % 6]
    a, b = _pair(N, D, F=0.5, CR=0.8, xo=xo, obj=obj, bounds=W.BOXES[obj], seed=N + D)
    a.run(7)
    b.run(7)
    _same(_state(a), _state(b))
    a.step()                                     # mixed with single generations, odd and even counts
    a.run(2)
    a.run(12)
    b.run(15)
    _same(_state(a), _state(b))


@pytest.mark.parametrize("obj", ["sphere", "rastrigin", "ackley", "rosenbrock", "griewank", "elliptic"])
@pytest.mark.parametrize("D", [70, 1100])
def test_every_objective(obj, D):
    for xo, cr, repair in (("nec", 0.99, "midpoint"), ("bin", 0.0, "clip"), ("exp", 1.0, "clip"), ("nec", 0.0, "clip")):
        a, b = _pair(200, D, F=0.9, CR=cr, xo=xo, obj=obj, bounds=W.BOXES[obj], seed=3, params={"repair": repair})
        a.run(20)
        b.run(20)
        _same(_state(a), _state(b))


@pytest.mark.parametrize("obj", ["rosenbrock", "ackley"])
@pytest.mark.parametrize("D", [3, 8, 37, 127, 128, 129, 517])
def test_segments_that_wrap(obj, D):
    """Segments of every length up to whole rows, wrapping anywhere."""
    for cr in (0.5, 0.97, 0.999):
        a, b = _pair(2500, D, F=0.7, CR=cr, xo="nec", obj=obj, bounds=W.BOXES[obj], seed=D)
        a.run(12)
        b.run(12)
        _same(_state(a), _state(b))


@pytest.mark.parametrize("xo,cr", [("nec", 0.97), ("exp", 0.4), ("bin", 0.6)])
def test_one_cluster_edges(xo, cr):
    """Rows and slots at the edges of the cluster's CTAs and of what it takes."""
    for N, D in ((4, 2), (7, 31), (8, 4), (9, 5), (64, 127), (160, 128), (161, 65), (241, 64), (248, 61)):
        obj = ("rosenbrock", "ackley", "griewank")[(N + D) % 3]
        a, b = _pair(N, D, F=0.5, CR=cr, xo=xo, obj=obj, bounds=W.BOXES[obj], seed=N)
        for count in (2, 9, 40):
            a.run(count)
            b.run(count)
        _same(_state(a), _state(b))


@pytest.mark.parametrize("base", ["random", "offset", "permutation", "best"])
def test_base_rules_and_long_runs(base):
    a, b = _pair(120, 40, F=0.5, CR=0.9, xo="nec", obj="sphere", bounds=(-100.0, 100.0), seed=9)
    for o in (a, b):
        o.set_base(base)
        o.run(5000)                              # more generations than one launch makes
    _same(_state(a), _state(b))


def test_checkpoint_and_nan():
    """A run resumes from a checkpoint of a stepped run; NaN parents and ties."""
    a, b = _pair(200, 100, F=0.5, CR=0.9, xo="bin", obj="rastrigin", bounds=(-5.12, 5.12), seed=4)
    pop = W.population(200, 100, -5.12, 5.12, 1)
    fit = np.linspace(1000.0, 3000.0, 200).astype(np.float32)
    fit[::7] = np.nan
    fit[5] = fit[6]
    for o in (a, b):
        o.set_population(pop, fit)
        o.run(9)
    _same(_state(a), _state(b))
    blob = b.save()
    b.run(30)
    a.run(100)                                   # a is elsewhere before it loads
    a.load(blob)
    a.run(30)
    _same(_state(a), _state(b))
