"""Populations to and from the host: a kernel moves them when the buffers are
page-locked and lie on 16-byte boundaries, copies move them otherwise. Either
way the same floats come back, and a run is not disturbed (bit for bit,
tolerance zero)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE

# one gene, totals that are no multiple of four, rows inside one slot, several spans; a pitch that is D, small
# and beyond what the kernel reads
SHAPES = [(4, 1), (5, 1), (300, 30), (65, 63), (40, 65), (33, 127), (9, 255), (51, 1001), (13, 1025), (7, 4097),
          (20, 64), (4096, 4104)]


def _host(n, kind):
    """n floats: page-locked, page-locked but off the boundary, or pageable."""
    import torch
    if kind == "pageable":
        return torch.empty(n)
    return torch.empty(n + 1, pin_memory=True)[1:] if kind == "offset" else torch.empty(n, pin_memory=True)


def _get(o, N, D, kind, inst=None):
    x, f = _host(N * D, kind), _host(N, kind)
    if inst is None:
        DE.de_get_population(o.ctx, x, f)
    else:
        DE.de_batch_get_population(o.ctx, inst, x, f)
    return x.numpy().tobytes(), f.numpy().tobytes()


def _set(o, x, kind, f=None, inst=None):
    hx = _host(x.size, kind)
    hx.numpy()[:] = x.ravel()
    hf = None if f is None else _host(f.size, kind)
    if f is not None:
        hf.numpy()[:] = f
    if inst is None:
        DE.de_set_population(o.ctx, hx, hf)
    else:
        DE.de_batch_set_population(o.ctx, inst, hx, hf)


@pytest.mark.parametrize("N,D", SHAPES)
@pytest.mark.parametrize("kind", ["locked", "offset"])
def test_single(N, D, kind):
    rng = np.random.default_rng(N * 7919 + D)
    x = rng.uniform(-5, 5, (N, D)).astype(np.float32)
    f = rng.uniform(0, 1e3, N).astype(np.float32)
    a, b = [DE.Optimizer(N, D, F=0.6, CR=0.7, obj="rosenbrock", bounds=(-5, 5), seed=3) for _ in range(2)]
    for fit in (None, f):                        # the second one replaces rows that lie in both buffers
        _set(a, x, kind, fit)
        _set(b, x, "pageable", fit)
        assert _get(a, N, D, kind)[0] == x.tobytes()
        for gens in (1, 3, 1, 2):                # a step and a run leave rows in either buffer
            for o in (a, b):
                o.run(gens)
            _get(a, N, D, kind)
        assert _get(a, N, D, kind) == _get(b, N, D, "pageable")
        assert a.best()[0].tobytes() == b.best()[0].tobytes()


def test_batch():
    specs = [dict(N=n, D=d, obj="rastrigin", bounds=(-5, 5), CR=0.8, F=0.5) for n, d in SHAPES if d <= 2048]
    rng = np.random.default_rng(11)
    a, b = DE.Batch(specs, seed=5), DE.Batch(specs, seed=5)
    for k, s in enumerate(specs):
        x = rng.uniform(-5, 5, (s["N"], s["D"])).astype(np.float32)
        f = rng.uniform(0, 1e3, s["N"]).astype(np.float32) if k % 2 else None
        _set(a, x, "locked", f, k)
        _set(b, x, "pageable", f, k)
        assert _get(a, s["N"], s["D"], "locked", k)[0] == x.tobytes()
    for gens in (1, 4, 1, 2):
        for o in (a, b):
            o.run(gens)
        for k in range(0, len(specs), 2):
            _get(a, specs[k]["N"], specs[k]["D"], "locked", k)
    for k, s in enumerate(specs):
        assert _get(a, s["N"], s["D"], "locked", k) == _get(b, s["N"], s["D"], "pageable", k)
