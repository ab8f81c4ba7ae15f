"""The complex128 apply's real and imaginary parts, each against its own terms."""
import numpy as np
import pytest

from oracle.operator import CellOperator
from paper_1709_09347_gb300 import synth
from tests._gpu_common import need_gpu
from tests.test_gpu_apply_fixed import EPS, _apply, _cell, _handle, _random

pytestmark = pytest.mark.gpu


def _parts_within(cell, z, E, X, Y):
    """Each part of Y - P X within 200 eps of the sum of the magnitudes of its terms: a row has 6 m + 1
    stencil terms and at most a few projector rows of some 30 entries in these cells, each product
    and sum rounding once."""
    op = CellOperator(*cell)
    for s in range(len(z)):
        P = op.P_matrix(z[s], E[s])
        err = Y[s] - P @ X[s]
        a, b, x, y = abs(P.real), abs(P.imag), np.abs(X[s].real), np.abs(X[s].imag)
        for got, bound in ((err.real, a @ x + b @ y), (err.imag, a @ y + b @ x)):
            assert np.all(np.abs(got) <= 200 * EPS * bound + 1e-300), (s, np.max(np.abs(got) / (EPS * bound + 1e-290)))


REAL, COMPLEX = np.array([1.7, 0.6, -1.0]), np.array([2 * np.exp(0.3j), 0.5 * np.exp(-1.2j), np.exp(2.0j)])
ES = np.array([0.3, -0.45, 0.1])


@pytest.mark.parametrize("z", [REAL, COMPLEX], ids=["real twists", "complex twists"])
@pytest.mark.parametrize("kind", ["tiny imaginary", "tiny real", "real", "imaginary", "holes", "one tiny column"])
def test_small_parts_keep_their_digits(kind, z):
    """A small part beside a large one, in whole columns or at a few points."""
    cell = _cell(9, 10, 16, 8, 3)
    n = cell[0].n
    X = _random((3, n, 6))
    if kind == "tiny imaginary":
        X = X.real + 1e-10j * X.imag
    elif kind == "tiny real":
        X = 1e-10 * X.real + 1j * X.imag
    elif kind == "real":
        X = X.real.astype(complex)
    elif kind == "imaginary":
        X = 1j * X.imag
    elif kind == "one tiny column":
        X[:, :, 2] = X[:, :, 2].real + 1e-10j * X[:, :, 2].imag
    else:
        x = X.reshape(3, 16, 10, 9, 6)
        for k, (iz, iy, ix) in enumerate([(3, 4, 5), (0, 0, 0), (15, 9, 8), (9, 5, 0), (12, 0, 4)]):
            for d in [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]:
                p = (iz + d[0]) % 16, (iy + d[1]) % 10, (ix + d[2]) % 9
                v = x[:, p[0], p[1], p[2]]
                x[:, p[0], p[1], p[2]] = v.real * (1e-9 if k % 2 else 1) + 1j * v.imag * (1 if k % 2 else 1e-9)
    Y = _apply(_handle(cell), 3, z, ES, X)
    _parts_within(cell, z, ES, X, Y)
    if kind == "real" and z is REAL:
        assert not Y.imag.any()
    if kind == "imaginary" and z is REAL:
        assert not Y.real.any()


@pytest.mark.parametrize("kind", ["strong entries tiny", "weak entries only", "one projector's entries only"])
def test_projector_sums_of_small_terms(kind):
    """Columns that are ordinary but over one atom's support: nothing but small terms in its sums, or
    large components where its projectors (some of them) are small.  The sums are then no better than
    their terms, not than the column."""
    cell = _cell(16, 16, 12, 4, 4, r_c=1.1)
    P = cell[2]
    X = _random((3, cell[0].n, 5))
    t = slice(P.sup_ptr[0], P.sup_ptr[1])
    idx, val = P.sup_idx[t], np.abs(P.sup_val[t])
    strong = (val >= val.max(0) / 4)
    assert strong.any(0).all() and not strong.all(0).any()
    if kind == "strong entries tiny":
        X[:, idx[strong.any(1)]] *= 1e-9
    elif kind == "weak entries only":
        weak = ~strong.any(1)
        assert weak.any()
        X[:, idx[~weak]] *= 1e-9
    else:
        X[:, idx[val[:, 1] > 1e-3 * val[:, 1].max()]] *= 1e-9
    Y = _apply(_handle(cell), 4, COMPLEX, ES, X)
    _parts_within(cell, COMPLEX, ES, X, Y)


@pytest.mark.parametrize("modulus", [1.0, 2.0, 3.2, 3.5, 4.0, 4.2, 4.4])
def test_widest_stencil_on_an_alternating_column(modulus):
    """All terms of a row of one sign, the twisted arms aligned with them: the largest sums that the
    fixed-point words have to hold (order 12; |z| and |1/z|)."""
    need_gpu()
    g = synth.Grid(8, 8, 8, 0.4, 0.4, 0.4, 12)
    cell = (g, np.zeros(g.n), None)
    i = np.arange(g.n)
    x = (-1.0) ** (i % 8 + i // 8 % 8 + i // 64) * (1 + 1j) * 0.999
    z = np.concatenate([modulus * np.exp(1j * np.pi / 4 * k) * np.array([1, modulus ** -2]) for k in range(8)])
    X = np.repeat(np.stack([x, x.conj(), x.real, 1j * x.imag], 1)[None], len(z), 0)
    E = np.zeros(len(z))
    _parts_within(cell, z, E, X, _apply(_handle(cell), 0, z, E, X))


@pytest.mark.parametrize("L,systems,nx,ny,nz,fd,launches", [
    (1, 14, 62, 9, 16, 2, 1), (16, 1, 8, 8, 4, 4, 1), (1, 8, 9, 32, 5, 8, 1),
    (14, 1, 47, 14, 6, 8, 3), (16, 8, 30, 20, 16, 4, 3),
])
def test_short_marches_of_few_columns_stay_on_one_launch(L, systems, nx, ny, nz, fd, launches):
    """Without projectors the FP64 stencil is a single launch, and quicker where there is little to do
    or where tiles of 8 x 8 lines and 4 columns would be mostly padding; both against the oracle."""
    need_gpu()
    from paper_1709_09347_gb300 import cbs
    cell = _cell(nx, ny, nz, fd, 0)
    X = _random((systems, cell[0].n, L))
    z, E = 1.8 * np.exp(1j * np.arange(systems)), np.linspace(-0.5, 0.5, systems)
    H = _handle(cell)
    before = cbs.kernel_launches()
    Y = _apply(H, 0, z, E, X)
    assert cbs.kernel_launches() - before == launches
    _parts_within(cell, z, E, X, Y)


def test_constant_field_on_a_long_march():
    """On a constant column the neighbours' coefficients add up to the energy of the FP64 weights (on a
    cell whose apply runs in fixed point): mean difference to the FP64 kernels below one rounding of
    E minus the kinetic diagonal (about 30, half an ulp 1.8e-15) and the mean of the 3600 points' own."""
    cell = _cell(12, 10, 30, 8, 0)
    X = np.ones((1, cell[0].n, 1), complex)
    X.imag = 1
    H, z = _handle(cell), np.array([1.0])
    a, b = (_apply(H, 0, z, ES[:1], X, k) for k in (False, True))
    assert not np.array_equal(a, b)
    assert abs((a - b).real.mean()) < 3e-15 and abs((a - b).imag.mean()) < 3e-15
