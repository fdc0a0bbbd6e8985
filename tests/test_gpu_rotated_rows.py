"""The FP32 rotated product picks its tile height by the number of rows; a row's
value does not depend on it: the fitness of the first n rows of a population is
the same, bit for bit, whatever n (tolerance zero), and within the 1e-5 of the
FP64 oracle that the rotated tests use."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

import oracle as O
from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W


@pytest.mark.parametrize("obj", ["sr_rastrigin", "sr_elliptic"])
@pytest.mark.parametrize("D", [3, 64, 97, 130, 256, 500])
def test_row_values_do_not_depend_on_the_tile(obj, D):
    params = dict(shift=W.shift_vector(D, 5), rotation=W.rotation(D, 6), prec="fp32")
    pop = W.population(9000, D, -100.0, 100.0, 7)
    ref = None
    for n in (9000, 4000, 2300, 1200, 700, 300, 111, 33, 5):
        opt = DE.Optimizer(n, D, obj=obj, bounds=(-100.0, 100.0), seed=1, params=params)
        opt.set_population(pop[:n])
        _, fit = opt.population()
        opt.close()
        if ref is None:
            ref = fit
            f64 = O.evaluate(obj, pop[:64], shift=params["shift"], rot=params["rotation"])
            assert np.all(np.abs(fit[:64] - f64) <= 1e-5 * np.maximum(1, np.abs(f64)))
        assert fit.tobytes() == ref[:n].tobytes()
