"""Device scratch of the field reads: min(N, 2^22) cells of four doubles, also
where the cells go through two halves and their number is odd."""
import ctypes as C

import numpy as np
import pytest

from test_fault_injection_gpu import _desc, _FailingAllocator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(64, 33), (1449, 1449), (2049, 1025), (2047, 2049), (2051, 2049)])
def test_macros_scratch(n):
    import torch
    from paper_1407_4524_gb300 import lbm
    lib = lbm.load()
    stream_ptr = int(torch.cuda.current_stream(0).cuda_stream)
    fa = _FailingAllocator(stream_ptr)
    asked = []
    inner = fa.alloc

    def recording(nbytes, ctx):
        asked.append(int(nbytes))
        return inner(nbytes, ctx)

    fa.alloc = lbm.ALLOC_FN(recording)
    d, q, _ = _desc(dict(lattice="D2Q9", n=n, tau=0.7, precision="fp16", u0=(0.03, 0.01)), fa, stream_ptr)
    h = C.c_void_p()
    assert lib.lbm_create_domain(C.byref(d), C.byref(h)) == 0
    assert lib.lbm_step(h, 1) == 0
    del asked[:]
    cells = n[0] * n[1]
    out = np.empty(4 * cells)
    assert lib.lbm_get_macros(h, out.ctypes.data) == 0
    assert asked == [min(cells, 1 << 22) * 32]
    assert np.isfinite(out).all() and abs(out[cells:2 * cells] - 0.03).max() < 1e-3
    assert lib.lbm_destroy_domain(h) == 0
    assert not fa.live
