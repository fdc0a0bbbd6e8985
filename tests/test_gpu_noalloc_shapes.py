"""The allocation-free generation at every launch shape of its kernel: slots per
thread 1 to 16, one warp to 16, more rows than the GPU holds CTAs, alone, in chains
and replayed from a captured graph. It sums as the row-per-CTA kernel of a context
does, so rows and values are that kernel's bit for bit (tolerance zero)."""
import gc

import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W

OBJ = ("sphere", "rastrigin", "ackley", "rosenbrock", "griewank", "elliptic")
# edges of 1, 2, 4, 8 and 16 slots per thread, the widest CTA, the longest row; the first ones are several waves of CTAs
SHAPES = [(5000, 40), (3000, 1024), (3000, 1025), (2500, 2048), (2000, 2049), (900, 4096), (700, 4097), (40, 8192),
          (33, 8193), (9, 16384), (8, 16385), (5, 32768), (4, 1), (65, 127)]


def _buffers(torch, pop, fit, pitch):
    N, D = pop.shape
    x = [torch.zeros(N, pitch, device="cuda") for _ in range(2)]
    f = [torch.zeros(N, device="cuda") for _ in range(2)]
    x[0][:, :D] = torch.from_numpy(pop).cuda()
    f[0][:] = torch.from_numpy(fit).cuda()
    return x, f


def _call(x, f, N, D, pitch, cr, obj, box, seed, g, stream):
    a, b = g % 2, (g + 1) % 2
    DE.de_nec_step_noalloc(x[a].data_ptr(), f[a].data_ptr(), x[b].data_ptr(), f[b].data_ptr(), N, D, pitch, 0.6, cr, obj,
                           box, seed, g, stream)


@pytest.mark.parametrize("cr", [0.9, 0.9999])
@pytest.mark.parametrize("N,D", SHAPES)
def test_chain_equals_the_row_kernel(N, D, cr):
    import torch
    obj = OBJ[(N + D) % 6]
    box = W.BOXES[obj]
    opt = DE.Optimizer(N, D, F=0.6, CR=cr, xo="nec", obj=obj, bounds=box, seed=D)
    opt.set_kernel(1)
    pop, fit = opt.population()
    pitch = (D + 3) // 4 * 4 + 4 * (N % 3)
    x, f = _buffers(torch, pop, fit, pitch)
    s = torch.cuda.current_stream().cuda_stream
    for g in range(4):                           # one call behind the other, nothing between them
        _call(x, f, N, D, pitch, cr, obj, box, D, g, s)
        opt.step()
    torch.cuda.synchronize()
    want, wfit = opt.population()
    assert x[0][:, :D].cpu().numpy().tobytes() == want.tobytes()
    assert f[0].cpu().numpy().tobytes() == wfit.tobytes()
    opt.close()


@pytest.mark.parametrize("N,D", [(100, 30), (900, 4097)])
def test_captured_chain(N, D):
    import torch
    obj, box, pitch = "rosenbrock", W.BOXES["rosenbrock"], (D + 3) // 4 * 4
    opt = DE.Optimizer(N, D, F=0.6, CR=0.8, xo="nec", obj=obj, bounds=box, seed=7)
    opt.set_kernel(1)
    pop, fit = opt.population()
    x, f = _buffers(torch, pop, fit, pitch)
    _call(x, f, N, D, pitch, 0.8, obj, box, 7, 0, torch.cuda.current_stream().cuda_stream)   # the thresholds
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    gc.collect()                                 # a graph of an earlier test may not end while this one is captured
    with torch.cuda.graph(graph):
        for g in range(4):
            _call(x, f, N, D, pitch, 0.8, obj, box, 7, g, torch.cuda.current_stream().cuda_stream)
    for k in range(2):                           # new values in the same buffers for the second replay
        for b in x + f:
            b.zero_()
        x[0][:, :D] = torch.from_numpy(pop).cuda()
        f[0][:] = torch.from_numpy(fit).cuda()
        graph.replay()
    opt.run(4)
    torch.cuda.synchronize()
    want, wfit = opt.population()
    assert x[0][:, :D].cpu().numpy().tobytes() == want.tobytes()
    assert f[0].cpu().numpy().tobytes() == wfit.tobytes()
    opt.close()
