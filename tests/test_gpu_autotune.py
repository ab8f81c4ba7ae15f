"""What the launch-shape search times."""
import pytest

from tests._gpu_common import need_gpu, small_cases

pytestmark = pytest.mark.gpu


def test_complex128_search_runs_the_kernels_that_take_a_shape():
    """Seven applies per shape of the FP64 gather and stencil, two launches each, then seven of the
    fixed-point apply (maxima, scales, gather, stencil) for the time that is reported."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    wl = small_cases()[4]
    H = cbs.Hamiltonian(wl.grid, wl.vloc, wl.projectors)
    L = 16
    shapes = sum(1 for a in range(6) for b in range(5) if 2 ** (a + b) * L <= 256)
    before = cbs.kernel_launches()
    best = cbs.autotune_apply(H, 8, L, torch.complex128)
    assert cbs.kernel_launches() - before == 7 * 2 * shapes + 7 * 4
    assert best["py"] * best["pz"] * L <= 256 and best["ms"] > 0
