"""The fixed-point complex128 apply: against the oracle's explicit operator, component by
component, and against the FP64 kernels (which serve a workspace of only the coefficients)."""
import ctypes as ct
import dataclasses

import numpy as np
import pytest

from oracle.operator import CellOperator
from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
ZS = np.array([2 * np.exp(0.3j), 0.5 * np.exp(-1.2j), np.exp(2.0j), 1.7 - 0.2j])
ES = np.array([0.3, -0.45, 0.0, 1.1])


def _apply(H, n_atoms, z, E, X, fp64_kernels=False):
    """cbs_apply_ws with the full workspace, or with one that holds the coefficients alone."""
    torch = need_gpu()
    from paper_1709_09347_gb300 import cbs
    lib = cbs.load()
    n, _, L = X.shape
    Xd = torch.from_numpy(np.ascontiguousarray(X)).cuda()
    zd, Ed = torch.tensor(np.asarray(z, complex)).cuda(), torch.tensor(np.asarray(E, float)).cuda()
    size = int(lib.cbs_apply_workspace_size(H.handle, n, L, cbs.CBS_C128))
    coef = n * max(n_atoms, 1) * 4 * L * 16
    ws = torch.empty(coef if fp64_kernels else size, dtype=torch.uint8, device="cuda")
    Y = torch.full_like(Xd, float("nan"))
    p = lambda t: ct.c_void_p(t.data_ptr())  # noqa: E731
    cbs._check(lib.cbs_apply_ws(H.handle, n, p(zd), p(Ed), L, p(Xd), p(Y), cbs.CBS_C128, p(ws), ws.numel(),
                                cbs._stream_ptr(torch)))
    torch.cuda.synchronize()
    return Y.cpu().numpy()


def _cell(nx, ny, nz, fd, atoms, h=(0.4, 0.4, 0.4), r_c=0.75, seed=3):
    wl = synth.tiny_workload(nx=nx, ny=ny, nz=nz, h=0.4, fd_order=fd, n_atoms=max(atoms, 1), r_c=r_c, sigma=0.3,
                             projectors=atoms > 0, L=1, seed=seed)
    return dataclasses.replace(wl.grid, hx=h[0], hy=h[1], hz=h[2]), wl.vloc, wl.projectors


def _handle(cell):
    need_gpu()
    from paper_1709_09347_gb300 import cbs
    return cbs.Hamiltonian(*cell)


def _within(cell, z, E, X, Y):
    """|Y - P X| <= 200 eps |P| |X| per component: a row has 6 m + 1 stencil terms and at most a
    few projector rows of some 30 entries in these cells, each product and sum rounding once."""
    op = CellOperator(*cell)
    for s in range(len(z)):
        P = op.P_matrix(z[s], E[s])
        err = np.abs(Y[s] - P @ X[s])
        assert np.all(err <= 200 * EPS * (abs(P) @ np.abs(X[s])) + 1e-300), (s, err.max())


def _random(shape, seed=5):
    rng = np.random.default_rng(seed)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


# edges of the 8 x 8 x 4 tiles, one line, short and long marches, every half-width, few and many
# systems (planes are split between blocks when there are few), unequal spacings
@pytest.mark.parametrize("nx,ny,nz,fd,atoms,L,n,h", [
    (8, 8, 4, 4, 2, 4, 4, None), (9, 7, 5, 8, 3, 5, 4, None), (16, 17, 4, 2, 1, 3, 1, None),
    (5, 5, 12, 12, 2, 1, 4, None), (1, 3, 6, 6, 0, 2, 4, None), (13, 10, 6, 10, 4, 33, 2, None),
    (7, 9, 70, 4, 2, 2, 1, None), (9, 8, 6, 8, 3, 6, 4, (0.41, 0.37, 0.43)), (6, 6, 4, 8, 2, 64, 4, None),
])
def test_against_the_explicit_operator(nx, ny, nz, fd, atoms, L, n, h):
    cell = _cell(nx, ny, nz, fd, atoms, h or (0.4, 0.4, 0.4))
    X = _random((n, nx * ny * nz, L))
    _within(cell, ZS[:n], ES[:n], X, _apply(_handle(cell), atoms, ZS[:n], ES[:n], X))


def test_many_atoms_on_one_point():
    """20 atoms on one centre: more entries per point than the scatter adds between carries."""
    g = synth.Grid(8, 8, 6, 0.4, 0.4, 0.4, 4)
    centres = np.tile(np.array([[1.5, 1.4, 1.3]]), (20, 1)) + np.arange(20)[:, None] * 0.01
    cell = (g, synth.gaussian_wells(g, centres[:2], [-0.5, -0.2], 0.6),
            synth.make_projectors(g, centres, r_c=1.1, sigma=0.4))
    X = _random((4, g.n, 4))
    _within(cell, ZS, ES, X, _apply(_handle(cell), 20, ZS, ES, X))


@pytest.mark.parametrize("kind", ["points", "decay", "one point", "columns", "twists", "energies"])
def test_ranges_that_fixed_point_does_not_serve(kind):
    """Components of very different magnitude in a column, columns that are zero, tiny or huge, and
    twists and energies out of range: FP64 accuracy per component all the same."""
    cell = _cell(9, 10, 6, 8, 3)
    n, z, E = cell[0].n, ZS, ES
    X = _random((4, n, 4))
    rng = np.random.default_rng(8)
    if kind == "points":
        X *= 10.0 ** rng.uniform(-14, 0, (1, n, 1))
    elif kind == "decay":
        X *= np.exp(-np.linspace(0, 60, n))[None, :, None]
    elif kind == "one point":
        X[:, np.arange(n) != 100] = 0
    elif kind == "columns":
        X *= np.array([1e-200, 0.0, 1e200, 1.0])
    elif kind == "twists":
        z = np.array([300 * np.exp(1j), 0.05 * np.exp(2j), 5j, 1e5])
    else:
        E = np.array([1e6, -300.0, 40.0, 1e15])
    _within(cell, z, E, X, _apply(_handle(cell), 3, z, E, X))


def test_nonfinite_components():
    """NaN and infinities reach the outputs that the FP64 kernels give them to."""
    cell = _cell(9, 10, 6, 8, 3)
    H = _handle(cell)
    X = _random((2, cell[0].n, 5))
    X[0, 17, 1], X[1, 5, 2], X[1, 40, 0] = np.nan, np.inf, complex(0, -np.inf)
    a, b = _apply(H, 3, ZS[:2], ES[:2], X), _apply(H, 3, ZS[:2], ES[:2], X, fp64_kernels=True)
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
    z = np.array([0.0, np.nan])
    a, b = _apply(H, 3, z, ES[:2], X[:1].repeat(2, 0)), _apply(H, 3, z, ES[:2], X[:1].repeat(2, 0), fp64_kernels=True)
    assert np.array_equal(np.isfinite(a), np.isfinite(b))


def test_error_not_above_the_fp64_kernels():
    """Against extended precision where the host has it: the fixed-point apply's error in the
    2-norm is no larger than the FP64 kernels' on Gaussian columns."""
    if np.finfo(np.longdouble).nmant <= 52:
        pytest.skip("no extended precision on this host")
    cell = _cell(9, 10, 6, 8, 3)
    H, X = _handle(cell), _random((1, cell[0].n, 4))
    z, E = ZS[:1], ES[:1]
    op = CellOperator(*cell)
    P = op.P_matrix(z[0], E[0]).toarray().astype(np.clongdouble)
    ref = P @ X[0].astype(np.clongdouble)
    err = [float(np.sqrt((np.abs(_apply(H, 3, z, E, X, k)[0] - ref) ** 2).sum())) for k in (False, True)]
    assert err[0] <= err[1]


def test_constant_field_keeps_the_weights_of_the_fp64_kernels():
    """On a constant column the neighbours' coefficients must not add up to another energy than the
    FP64 weights: mean difference to the FP64 kernels below one rounding of E minus the kinetic
    diagonal (23.4, half an ulp 1.8e-15) and the mean of the 840 points' own roundings (exact
    coefficients beside the rounded diagonal: 5.8e-15)."""
    cell = _cell(12, 10, 7, 4, 0)
    X = np.ones((1, cell[0].n, 1), complex)
    H, z = _handle(cell), np.array([1.0])
    a, b = (_apply(H, 0, z, ES[:1], X, k) for k in (False, True))
    assert abs((a - b).real.mean()) < 3e-15
