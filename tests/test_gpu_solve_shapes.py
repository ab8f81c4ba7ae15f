"""Shapes at which the solver's reductions and the Hankel SVD change their launch form."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from oracle import ss
from oracle.contour import ring_contour
from oracle.dense import match
from oracle.operator import CellOperator
from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu, rel_err

pytestmark = pytest.mark.gpu


# one column (256 lanes share it) to 256 columns (one lane each), widths that leave lanes over,
# cells of one and of many chunks, one point and several
@pytest.mark.parametrize("L,points,cell", [
    (1, 1, (6, 5, 4)), (1, 3, (13, 10, 6)), (2, 5, (13, 10, 6)), (31, 2, (6, 5, 4)), (40, 1, (13, 10, 6)),
    (64, 2, (6, 5, 4)), (130, 1, (6, 5, 4)), (256, 2, (6, 5, 4)),
])
def test_shifted_solves_over_column_counts(L, points, cell):
    """Primal and dual solutions against sparse direct solves: residuals of 1e-12 times a condition
    number of a few hundred."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    wl = synth.tiny_workload(nx=cell[0], ny=cell[1], nz=cell[2], h=0.45, fd_order=4, n_atoms=2, r_c=0.8, sigma=0.3, L=L)
    H = cbs.Hamiltonian(wl.grid, wl.vloc, wl.projectors)
    op = CellOperator(wl.grid, wl.vloc, wl.projectors)
    z1, _, _, _ = ring_contour(0.5, 8)
    zs, E = z1[:points], 0.2
    B = torch.from_numpy(wl.V).to("cuda").contiguous()
    Y, Yd, iters, _ = cbs.solve_shifted(H, zs, E, B, cbs.options(tol=1e-12))
    Y, Yd = Y.cpu().numpy(), Yd.cpu().numpy()
    for s, z in enumerate(zs):
        P = op.P_matrix(z, E)
        assert rel_err(Y[s], spla.spsolve(P, wl.V).reshape(Y[s].shape)) < 1e-9
        assert rel_err(Yd[s], spla.spsolve(P.conj().T.tocsc(), wl.V).reshape(Y[s].shape)) < 1e-9
    assert (iters > 0).all()


# Hankel orders LM of 6 (fewer than the blocks of a cluster) to 184, odd and even; two energies
# (a block per Jacobi pair) and four of order 184 (a warp per pair)
@pytest.mark.parametrize("L,M,energies", [
    (2, 3, (0.2, -0.3)), (3, 7, (0.2, -0.3)), (11, 3, (0.2,)), (23, 8, (0.2, -0.3)), (23, 8, (0.2, -0.3, 0.2, -0.3)),
])
def test_hankel_extraction_over_orders(L, M, energies):
    """Eigenvalues of Algorithm 1 against the oracle's.  The oracle's own move by up to 3e-12
    between solve tolerances of 1e-12 and 1e-13; 1e-9 leaves room for another rounding."""
    need_gpu()
    from paper_1709_09347_gb300 import cbs
    wl = synth.tiny_workload(nx=6, ny=5, nz=4, h=0.45, fd_order=4, n_atoms=2, r_c=0.8, sigma=0.3, L=L, M=M, n_int=32,
                             energies=energies)
    H = cbs.Hamiltonian(wl.grid, wl.vloc, wl.projectors)
    res = cbs.solve(H, wl.energies, wl.lambda_min, wl.n_int, L, M, wl.V, cbs.options(tol=1e-12))
    op = CellOperator(wl.grid, wl.vloc, wl.projectors)
    for e, E in enumerate(wl.energies):
        ref = ss.ss_hankel(op, float(E), wl.lambda_min, wl.n_int, wl.V, M, tol=1e-12)
        got = res.energies[e]
        assert len(got["lam"]) == len(ref.lam) == 2
        worst, un_f, un_r = match(got["lam"], ref.lam, 1e-9)
        assert not un_f and not un_r, worst
        assert np.all(got["residual"] <= 1e-8)
