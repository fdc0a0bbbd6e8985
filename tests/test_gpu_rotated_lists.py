"""The re-evaluation of uncertain rows takes tiles of 8, 16 or 32 entries by the
length of its list. With a margin that no decision clears every row is on the list,
so its length is N; whatever the tile, decisions and the rows they leave are
the FP32 product's bit for bit (tolerance zero)."""
import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W


# rows of one tile and less, remainders of each tile size, lists that fill the GPU once and several times
@pytest.mark.parametrize("N", [4, 5, 16, 21, 150, 203, 290, 450, 701, 3001])
@pytest.mark.parametrize("D,obj,prec", [(256, "sr_rastrigin", "fp16"), (512, "sr_elliptic", "bf16")])
def test_every_list_length(N, D, obj, prec):
    params = dict(shift=W.shift_vector(D, 5), rotation=W.rotation(D, 6))
    kw = dict(F=0.5, CR=0.9, xo="nec", obj=obj, bounds=(-100.0, 100.0), seed=N)
    a = DE.Optimizer(N, D, params=dict(params, prec=prec, margin_sigmas=1e6), **kw)
    b = DE.Optimizer(N, D, params=dict(params, prec="fp32"), **kw)
    for _ in range(5):
        a.run(2)
        b.run(2)
        x, _ = a.population()
        y, _ = b.population()
        assert x.tobytes() == y.tobytes()
    s, t = a.stats(), b.stats()
    assert s["accepts"] == t["accepts"] and s["reselected"] == 10 * N
    a.close()
    b.close()
