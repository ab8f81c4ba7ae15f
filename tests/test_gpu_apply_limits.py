"""Sizes that the operator apply refuses."""
import ctypes as ct

import numpy as np
import pytest

from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
def test_systems_beyond_32_bit_indices_are_refused_before_any_launch(dtype):
    """N L = 2^31 (cell with projectors, so that a gather would come first): CBS_EINVAL, and no kernel
    has been queued on the vectors, which are far too small here."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    lib = cbs.load()
    g = synth.Grid(256, 256, 128, 0.4, 0.4, 0.4, 2)
    L = 256
    assert g.n * L == 1 << 31
    proj = synth.Projectors(1, 1, np.array([0, 3]), np.array([5, g.n // 2, g.n - 1], np.int32), np.zeros(3, np.int8),
                            np.ones((3, 1)), np.ones((1, 1, 1)))
    H = cbs.Hamiltonian(g, np.zeros(g.n), proj)
    X, Y = torch.zeros(4, dtype=getattr(torch, dtype), device="cuda"), torch.zeros(4, dtype=getattr(torch, dtype), device="cuda")
    dt = {"complex64": cbs.CBS_C64, "complex128": cbs.CBS_C128}[dtype]
    z, E = np.array([[1.5, 0.5]]), np.array([0.1])
    before = lib.cbs_kernel_launches()
    for call in (lib.cbs_apply, lib.cbs_apply_noalloc):
        st = call(H.handle, 1, cbs._dptr(z), cbs._dptr(E), L, ct.c_void_p(X.data_ptr()), ct.c_void_p(Y.data_ptr()), dt,
                  cbs._stream_ptr(torch))
        assert st == cbs.CBS_EINVAL
    assert lib.cbs_kernel_launches() == before
