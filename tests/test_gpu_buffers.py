"""What contexts take from the allocator: nothing that no kernel reads, and where
it is refused on a run's first use the run goes on with a launch per generation
(the results bit for bit the same) and leaves no block behind."""
import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W


class _Allocator:
    """Torch's blocks with their sizes; requests from the k-th on get nothing."""

    def __init__(self):
        import torch
        self.torch, self.live, self.taken, self.left, self.refused = torch, {}, [], None, False
        self.a, self.f = DE._ALLOC_FN(self._alloc), DE._FREE_FN(self._free)

    def __enter__(self):
        assert DE.load_library().de_set_allocator(self.a, self.f, None) == DE.DE_OK
        return self

    def __exit__(self, *exc):
        DE.use_torch_allocator(True)

    def _alloc(self, n, stream, user):
        if self.left is not None:
            if self.left == 0:
                self.refused = True
                return None
            self.left -= 1
        t = self.torch.empty(int(n), dtype=self.torch.uint8, device="cuda")
        self.live[t.data_ptr()] = t
        self.taken.append(int(n))
        return t.data_ptr()

    def _free(self, ptr, n, stream, user):
        del self.live[ptr]


def _create(N, D, stream, params=None, obj="sphere"):
    return DE.de_create(N, D, 0.5, 0.9, "nec", obj, (-5.0, 5.0), 1, params, stream.cuda_stream)


def test_one_cluster_takes_its_state_alone():
    import torch
    with _Allocator() as al:
        s = torch.cuda.Stream()
        for N, D, held in ((100, 30, 256), (300, 30, 256 + 300 * 128 + 2 * 300 * 32 * 4)):
            h = _create(N, D, s)
            n = len(al.taken)
            DE.de_run(h, 20)
            DE.de_synchronize(h)
            assert sum(al.taken[n:]) == held
            DE.de_destroy(h)
        assert not al.live


@pytest.mark.parametrize("prec,bound,sums", [("fp32", "probabilistic", 1), ("fp32", "worst_case", 1),
                                             ("fp16", "probabilistic", 1), ("bf16", "worst_case", 2)])
def test_rotated_sums_that_nobody_reads(prec, bound, sums):
    import torch
    D, N = 256, 1000
    one = (N * 4 * 4 + 255) // 256 * 256                 # N x (D / 64) floats
    with _Allocator() as al:
        h = _create(N, D, torch.cuda.Stream(), dict(shift=W.shift_vector(D, 1), rotation=W.rotation(D, 2), prec=prec,
                                                    bound=bound), "sr_rastrigin")
        assert al.taken.count(one) == sums
        DE.de_run(h, 3)
        DE.de_synchronize(h)
        DE.de_destroy(h)


@pytest.mark.parametrize("kind", ["cluster", "resident", "batch"])
def test_refused_buffers_leave_a_launch_per_generation(kind):
    import numpy as np
    import torch
    specs = [dict(N=40, D=30, obj="ackley", bounds=(-5.0, 5.0)), dict(N=64, D=700, obj="rosenbrock", bounds=(-5.0, 5.0))]
    N, D = (100, 30) if kind == "cluster" else (300, 500)
    shape = [(s["N"], s["D"]) for s in specs] if kind == "batch" else [(N, D)]

    def out(h):
        res = []
        for k, (n, d) in enumerate(shape):
            x, f = np.empty((n, d), np.float32), np.empty(n, np.float32)
            DE.de_batch_get_population(h, k, x, f) if kind == "batch" else DE.de_get_population(h, x, f)
            res += [x.tobytes(), f.tobytes()]
        return res

    with _Allocator() as al:
        s = torch.cuda.Stream()
        make = lambda: (DE.de_batch_create(specs, 1, s.cuda_stream) if kind == "batch" else _create(N, D, s))
        ref = make()
        for _ in range(12):
            DE.de_step(ref)
        want = out(ref)
        DE.de_destroy(ref)
        for k in range(6):                               # the k-th request of the first run gets nothing
            h = make()
            n = len(al.live)
            al.left, al.refused = k, False
            DE.de_run(h, 12)
            al.left = None
            assert out(h) == want
            assert al.refused == (k < {"cluster": 1, "resident": 3, "batch": 4}[kind])
            # a resident run's 256 bytes of state stay for the next one
            assert not al.refused or len(al.live) == n + (1 if kind == "resident" and k else 0)
            DE.de_destroy(h)
            assert not al.live
