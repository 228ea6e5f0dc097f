"""xsde_integrate_static_scratch keeps its host tables in the thread's own buffers: a
thread's first call with longer dimensions takes nothing from the heap.

The allocator's counts (mallinfo2, all arenas) include what the CUDA runtime takes for
a call, so the kernels are loaded and the thread has made a short call beforehand,
and the smallest of several threads' growth counts.  2048 factors are 32 KB; 16 KB is
the bound.
"""
import ctypes
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class _MallInfo(ctypes.Structure):
    _fields_ = [(k, ctypes.c_size_t) for k in ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks", "fsmblks",
                                               "uordblks", "fordblks", "keepcost")]


def _in_use():
    libc = ctypes.CDLL(None)
    if not hasattr(libc, "mallinfo2"):
        pytest.skip("no mallinfo2")
    libc.mallinfo2.restype = _MallInfo
    m = libc.mallinfo2()
    return m.uordblks + m.hblkhd


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_a_threads_first_long_call_takes_no_heap(dtype):
    import torch
    from paper_1204_4255_gb300 import xsde

    def setup(shape):
        P = xsde.Problem(shape, (-6.0, -6.0), (6.0, 6.0), dtype)
        P.set_operators(g=1.0)
        psi = torch.ones((1,) + shape, dtype=torch.complex64 if dtype == "c64" else torch.complex128, device="cuda")
        vec = xsde.xsde_vector_wrap(P.grid, xsde.XSDE_C64 if dtype == "c64" else xsde.XSDE_C128, 1, 1, psi.data_ptr())
        return P, psi, vec

    short, long = setup((16, 16)), setup((16, 2048))
    stream = torch.cuda.current_stream().cuda_stream

    def call(s):
        xsde.xsde_integrate_static_scratch(s[0].prob, s[2], 1e-4, 2, 1, 0, 0, stream)
        xsde.xsde_synchronize(s[0].prob, stream)

    call(short)
    call(long)
    grown = []

    def thread():
        torch.cuda.set_device(0)
        call(short)
        call(short)
        before = _in_use()
        call(long)
        grown.append(_in_use() - before)

    for _ in range(4):
        t = threading.Thread(target=thread)
        t.start()
        t.join()
    for s in (short, long):
        xsde.xsde_vector_free(s[2])
        s[0].close()
    assert len(grown) == 4 and min(grown) < 16384, grown
    assert np.isfinite(long[1].cpu().numpy()).all()
