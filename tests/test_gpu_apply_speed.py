"""The complex128 apply on columns that fixed point does not serve."""
import ctypes as ct

import numpy as np
import pytest

from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["zero", "real", "localised", "decaying", "wide", "every fourth zero"])
def test_columns_of_wide_range_are_no_slower_than_the_fp64_kernels(kind):
    """Such columns go to the FP64 formula, which must not cost more than the FP64 kernels (run with a
    workspace of the coefficients alone).  Fixed point and the formula point by point after it took
    1.4 to 1.7 times their time; a third more leaves room for the passes that find such a column."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    lib = cbs.load()
    wl = synth.workload("c2", with_rhs=False)
    g, L, n = wl.grid, 32, 8
    H = cbs.Hamiltonian(g, wl.vloc, wl.projectors)
    gen = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn((n, g.n, L), dtype=torch.complex128, device="cuda", generator=gen)
    i = torch.arange(g.n, device="cuda")
    if kind == "zero":
        X.zero_()
    elif kind == "real":
        X = X.real.to(X.dtype)
    elif kind == "localised":
        r2 = ((i % g.nx - g.nx / 2) ** 2 + (i // g.nx % g.ny - g.ny / 2) ** 2 + (i // (g.nx * g.ny) - g.nz / 2) ** 2) * g.hx ** 2
        X *= torch.exp(-r2.double() / 2)[None, :, None]
    elif kind == "decaying":
        X *= torch.exp(-60 * i / g.n)[None, :, None]
    elif kind == "wide":
        X *= 10 ** (-14 * torch.rand((1, g.n, 1), dtype=torch.float64, device="cuda", generator=gen))
    else:
        X[:, :, ::4] = 0
    X = X.contiguous()
    Y = torch.empty_like(X)
    z = torch.tensor(2 * np.exp(2j * np.pi * (np.arange(n) + 0.5) / n)).cuda()
    E = torch.linspace(-0.5, 0.5, n, dtype=torch.float64, device="cuda")
    size = int(lib.cbs_apply_workspace_size(H.handle, n, L, cbs.CBS_C128))
    coef = n * wl.projectors.n_atoms * 4 * L * 16
    assert coef < size
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")

    def apply(nbytes):
        p = lambda t: ct.c_void_p(t.data_ptr())  # noqa: E731
        cbs._check(lib.cbs_apply_ws(H.handle, n, p(z), p(E), L, p(X), p(Y), cbs.CBS_C128, p(ws), nbytes,
                                    cbs._stream_ptr(torch)))

    def ms(nbytes):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            apply(nbytes)
        b.record()
        b.synchronize()
        return a.elapsed_time(b)

    ms(size), ms(coef)
    t = sorted(ms(size) for _ in range(7))[3] / sorted(ms(coef) for _ in range(7))[3]
    assert t < 4 / 3, t
