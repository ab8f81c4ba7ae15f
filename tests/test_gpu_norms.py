"""Frobenius norms of cells without projectors, whose stencil part has a closed form."""
import numpy as np
import pytest

from oracle.operator import CellOperator
from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu

pytestmark = pytest.mark.gpu


# axes longer than the stencil, as long as it, shorter (arms that meet each other, or their own
# point: the diagonal), one point, and one FD step per cell
@pytest.mark.parametrize("nx,ny,nz,fd", [
    (9, 11, 4, 2), (5, 4, 5, 4), (4, 3, 4, 8), (2, 1, 6, 12), (1, 1, 6, 6), (13, 6, 2, 4), (8, 7, 1, 2), (30, 20, 24, 8),
])
def test_norms_without_projectors(nx, ny, nz, fd):
    need_gpu()
    from paper_1709_09347_gb300 import cbs
    g = synth.Grid(nx, ny, nz, 0.41, 0.37, 0.45, fd)
    v = np.random.default_rng(3).standard_normal(g.n)
    H = cbs.Hamiltonian(g, v)
    op = CellOperator(g, v, None)
    for E in (0.0, 0.37):
        assert np.allclose(H.norms(E), op.frobenius(E), rtol=1e-12, atol=0)
