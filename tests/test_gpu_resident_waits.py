"""Waits of the on-chip runs that give up (gen_resident.cuh), made to by a limit
of a nanosecond: they guard no copy in flight. The launch ends, the error is
reported once and launches are refused from then on; nothing faults.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W

# a warp per row; one row per CTA; several warps per row with a group that has no row in the last CTA (301 rows, two
# per CTA), and with two slots per thread; many rows per CTA, for segments and for binomial rows of one warp
CASES = [(300, 500, "nec", "rastrigin"), (150, 1000, "exp", "rosenbrock"), (301, 500, "bin", "griewank"),
         (301, 500, "bin", "rosenbrock"), (301, 1500, "bin", "ackley"), (5000, 30, "nec", "sphere"),
         (5001, 100, "bin", "rosenbrock")]


def _optimizer(N, D, xo, obj):
    return DE.Optimizer(N, D, F=0.5, CR=0.8, xo=xo, obj=obj, bounds=W.BOXES[obj], seed=N)


@pytest.mark.parametrize("N,D,xo,obj", CASES)
def test_a_wait_that_gives_up_ends_the_run(N, D, xo, obj):
    a = _optimizer(N, D, xo, obj)
    DE.de_set_wait_limit(a.ctx, 1)
    a.run(200)
    for call, code in ((a.synchronize, DE.DE_ETIMEOUT), (a.step, DE.DE_ESTATE), (lambda: a.run(3), DE.DE_ESTATE)):
        with pytest.raises(DE.DEError) as e:
            call()
        assert e.value.code == code
    x, f = a.population()
    lo, hi = W.BOXES[obj]
    assert np.all((x >= lo) & (x <= hi)) and np.all(np.isfinite(f))
    a.close()
    b = _optimizer(N, D, xo, obj)                # the device is as it was: another context runs
    c = _optimizer(N, D, xo, obj)
    c.set_kernel(1)
    DE.de_set_wait_limit(b.ctx, 10**9)           # a limit that is set and not reached
    for o in (b, c):
        o.run(40)
    for u, v in zip(b.population(), c.population()):
        assert u.tobytes() == v.tobytes()
    b.close()
    c.close()


def _generation_and_error(a):
    """Generations counted and the device error, from a checkpoint (the other calls report the error alone)."""
    blob = np.frombuffer(a.save(), np.uint8)
    st = blob[72:]                               # magic .. repair; then best_key, gen, best_gen, 3 counters, done, error
    return int(st[8:16].view(np.int64)[0]), int(st[16:24].view(np.int64)[0]), int(st[52:56].view(np.uint32)[0])


@pytest.mark.parametrize("limit", [1, 3000, 30000])
@pytest.mark.parametrize("N,D,xo,obj", CASES)
def test_what_a_run_that_gave_up_leaves(N, D, xo, obj, limit):
    """Whole rows with their fitness, each of the counted generation or one of the
    three after it (bit for bit), and nothing from what was queued behind it."""
    a, b = _optimizer(N, D, xo, obj), _optimizer(N, D, xo, obj)
    b.set_kernel(1)
    DE.de_set_wait_limit(a.ctx, limit)
    a.run(300)
    a.run(300)                                   # behind a launch that gave up: does nothing
    x, f = a.population()
    g, best_gen, err = _generation_and_error(a)
    assert err == (0 if g == 600 else DE.DE_ETIMEOUT) and best_gen <= g
    assert err or limit > 1
    b.run(g)
    there = np.zeros(N, bool)
    for k in range(4 if err else 1):
        y, fy = b.population()
        there |= np.all(x.view(np.uint32) == y.view(np.uint32), axis=1) & (f.view(np.uint32) == fy.view(np.uint32))
        b.step()
    assert there.all()
    a.close()
    b.close()
