"""Row kernels named by de_batch_set_groups hold for runs: only a batch that was
left to the library, or to its autotuner, keeps partial sums for a run (and takes
their buffers). Every choice gives the same populations, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W

SPECS = [dict(N=40 + 9 * k, D=D, obj=obj, bounds=W.BOXES[obj], xo=xo, CR=0.9, F=0.5)
         for k, (D, xo, obj) in enumerate([(10, "nec", "sphere"), (300, "exp", "ackley"), (2000, "nec", "rosenbrock"),
                                           (33, "nec", "rastrigin")])]


def _run(prepare, gens):
    b = DE.Batch(SPECS, seed=4)
    prepare(b)
    held = len(DE._live_blocks)
    b.run(gens)
    kept = len(DE._live_blocks) > held           # a run that keeps sums takes buffers for them
    out = [x.tobytes() for k in range(len(SPECS)) for x in b.population(k)]
    b.close()
    return kept, out


@pytest.mark.parametrize("gens", [2, 9])
def test_named_kernels_hold_for_runs(gens):
    ref = _run(lambda b: None, gens)
    assert ref[0]
    for groups in ([1] * 4, [2] * 4, [-8, 0, 0, 0], [0, 0, 0, 8], [4, 32, 32, 4]):
        assert _run(lambda b: b.set_groups(groups), gens) == (False, ref[1]), groups

    def back(b):
        b.set_groups([2] * 4)
        b.set_groups([0] * 4)

    def tuned(b):
        b.set_groups([2] * 4)
        b.autotune(reps=1)
    for prepare in (back, tuned):
        assert _run(prepare, gens) == ref
    assert _run(lambda b: b.set_groups(b.autotune(reps=1)), gens) == (False, ref[1])
