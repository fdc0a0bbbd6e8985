"""Host populations whose buffer is page-locked in pieces: a kernel moves them
only if the pieces cover the whole buffer. With pageable memory between two
pieces the call goes to a copy, which the driver refuses for such a range
(DE_ECUDA) or makes; either way no kernel addresses the gap, and the context
goes on."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2101_06599_gb300 import de as DE

N, D, PAGE = 768, 1024, 1 << 16                  # 3 MB


@pytest.mark.parametrize("pieces,whole", [([(0, 48)], True), ([(0, 16), (16, 32)], True), ([(0, 1), (1, 46), (47, 1)], True),
                                          ([(0, 16), (32, 16)], False), ([(0, 16)], False), ([(32, 16)], False)])
def test_populations_in_pieces(pieces, whole):
    import torch
    torch.cuda.init()
    rt = torch.cuda.cudart()
    raw = np.zeros(N * D * 4 + PAGE, np.uint8)
    off = -raw.ctypes.data % PAGE
    buf = raw[off:off + N * D * 4].view(np.float32)
    a = DE.Optimizer(N, D, obj="sphere", bounds=(-5, 5), seed=3)
    x, f = a.population()
    locked = []
    try:
        for first, n in pieces:
            assert int(rt.cudaHostRegister(buf.ctypes.data + first * PAGE, n * PAGE, 0)) == 0
            locked.append(buf.ctypes.data + first * PAGE)
        for k in range(2):
            try:
                DE.de_get_population(a.ctx, buf, None)
                assert buf.tobytes() == x.tobytes()
                x = np.ascontiguousarray(x[::-1])
                buf[:] = x.ravel()
                DE.de_set_population(a.ctx, buf)
            except DE.DEError as e:
                assert not whole and e.code == DE.DE_ECUDA
            y, g = a.population()                # pageable: as ever
            assert y.tobytes() == x.tobytes()
            f = f[::-1] if whole else f
            assert not whole or g.tobytes() == f.tobytes()
    finally:
        for p in locked:
            rt.cudaHostUnregister(p)
    a.step()
    a.synchronize()
    a.close()
