"""Runs of a batch that touch only what the segments touch (batch_seg.cu)
against single generations, which read every row: both add in one order, so
populations, fitness, counters and best are equal bit for bit (tolerance zero).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W

OBJ = ("sphere", "rastrigin", "ackley", "rosenbrock", "griewank", "elliptic")
# one slot, fewer and more than 8 and 32 slots, rows that end inside a slot, the longest rows; spans of 1 and 32 rows
SIZES = [(4, 1), (33, 3), (64, 8), (65, 30), (70, 31), (97, 33), (40, 63), (31, 127), (32, 128), (36, 129), (50, 130),
         (64, 257), (35, 1000), (40, 1001), (20, 2047), (37, 2048)]


def _specs(xo, cr, shift):
    return [dict(N=n, D=d, obj=OBJ[(k + shift) % 6], bounds=W.BOXES[OBJ[(k + shift) % 6]], xo=xo, CR=cr, F=0.6)
            for k, (n, d) in enumerate(SIZES)]


def _state(b, k):
    x, f = b.population(k)
    bx, bf, bi, bg = b.best(k)
    s = b.stats(k)
    return [np.asarray(v).tobytes() for v in (x, f, bx, np.float64(bf), bi, bg, s["generation"], s["accepts"],
                                              s["masked_genes"], s["best_gen"])]


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 4, 5])
@pytest.mark.parametrize("xo,cr", [("nec", 0.9), ("nec", 0.0), ("exp", 0.5), ("nec", 0.95)])
def test_run_equals_steps(xo, cr, shift):
    specs = _specs(xo, cr, shift)
    a, b = DE.Batch(specs, seed=3 + shift), DE.Batch(specs, seed=3 + shift)
    for count in (9, 4, 1, 6):                   # several runs, with a single generation between them
        a.run(count)
        for _ in range(count):
            b.step()
        for k in range(len(specs)):
            assert _state(a, k) == _state(b, k), (k, specs[k], count)
    for o in (a, b):                             # new genes and given values, NaN among them, then a run again
        pop = W.population(specs[12]["N"], specs[12]["D"], -1.0, 1.0, 5)
        fit = np.linspace(1.0, 9000.0, specs[12]["N"]).astype(np.float32)
        fit[3] = np.nan
        o.set_population(12, pop, fit)
    a.run(12)
    for _ in range(12):
        b.step()
    for k in range(len(specs)):
        assert _state(a, k) == _state(b, k), (k, specs[k])
    a.close()
    b.close()


@pytest.mark.parametrize("base", ["random", "permutation", "best"])
def test_base_rules(base):
    specs = _specs("nec", 0.9, 1)
    a, b = DE.Batch(specs, seed=8), DE.Batch(specs, seed=8)
    for o in (a, b):
        o.set_base(base)
    a.run(7)
    for _ in range(7):
        b.step()
    for k in range(len(specs)):
        assert _state(a, k) == _state(b, k)
    a.close()
    b.close()
