"""FP64 products over FP64's whole exponent range.

Every row and every vector has its own power of two, so scaling a right-hand
side or a row by a power of two scales the product by it, bit for bit, as long
as nothing around the digits (the transforms) leaves FP64's normal range.  A
sum that is zero stays zero however large the row and the vector are.  Columns
and vector entries of very different size keep the bound of the digits: the
error of an output is below n 2^-48 of its row's maximum times the vector's
maximum (n sources; tests of the tile edges derive it) plus one rounding.
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H
COEF = (1j * W.K0, 0.9 - 0.2j, -1.1, 0.5 + 1j * W.K0)


def product(B, h, x):
    import torch
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    y = torch.full_like(xd, float("nan"))
    B.emsurf_matvec(h, xd, y, B.FP64)
    return y.cpu().numpy()


def single_cell(B, n, Z):
    """One box without coupling: y = Z x."""
    E = 18 * n * n
    idx, sgn, nu = B.emsurf_setup_overlap(n, 1, 1)
    assert nu == 2 * E and (sgn == 1).all() and (idx == np.arange(nu)).all()
    T = np.zeros((1, 1, E, E), complex)
    return B.emsurf_create(1, 1, E, nu, np.zeros(1, np.int32), Z[None], T, T, COEF, idx, sgn, precision=B.FP64)


@pytest.mark.parametrize("s", [-930, -905, -400, 0, 500, 900])
def test_rhs_scaled_by_powers_of_two(emsurf_lib, s):
    from paper_1911_04576_gb300 import binding as B
    n, nx, ny = 2, 3, 2
    E = 18 * n * n
    idx, sgn, nu = lattice.overlap_map(box_mesh(A, A, H, n), nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, 3)
    h = B.emsurf_create(nx, ny, E, nu, np.arange(6, dtype=np.int32) % 2, W.random_macromodels(2, 2 * E, 4), Lt, Kt, COEF,
                        idx, sgn, precision=B.FP64, max_rhs=2)
    x = W.random_vectors(2, nu, 5)
    y = product(B, h, x)
    f = np.ldexp(1.0, s)
    assert (product(B, h, x * np.array([[f], [1.0]])) == y * np.array([[f], [1.0]])).all()
    h.close()


def test_rows_scaled_by_powers_of_two(emsurf_lib):
    from paper_1911_04576_gb300 import binding as B
    n, K = 2, 144
    Z = W.random_macromodels(1, K, 4)[0]
    x = W.random_vectors(1, K, 5)
    h = single_cell(B, n, Z)
    y = product(B, h, x)[0]
    h.close()
    r = np.random.default_rng(6).integers(-960, 900, K)
    h = single_cell(B, n, Z * np.ldexp(1.0, r)[:, None])
    ys = y * np.ldexp(1.0, r)
    assert (product(B, h, x)[0] == ys).all()
    # a small vector against large rows: the powers meet before they leave the range
    yb = product(B, h, x * np.ldexp(1.0, -940))[0]
    assert (yb[r > 0] == (ys * np.ldexp(1.0, -940))[r > 0]).all()
    h.close()


def test_zero_sums_of_large_rows_and_vectors(emsurf_lib):
    from paper_1911_04576_gb300 import binding as B
    n, K = 2, 144
    Z = np.zeros((K, K), complex)
    Z[:, 3] = 2.0 ** 600
    h = single_cell(B, n, Z)
    x = np.zeros((1, K), complex)
    x[0, 7] = 2.0 ** 600
    assert (product(B, h, x) == 0).all()
    h.close()


@pytest.mark.parametrize("decades", [6, 30, 120])
def test_columns_and_entries_of_very_different_size(emsurf_lib, decades):
    from paper_1911_04576_gb300 import binding as B
    n, K = 2, 144
    g = np.random.default_rng(decades)
    Z = W.random_macromodels(1, K, 4)[0] * 10.0 ** g.uniform(-decades, 0, K) * 10.0 ** g.uniform(-decades, decades, K)[:, None]
    x = W.random_vectors(1, K, 5)[0] * 10.0 ** g.uniform(-decades, 0, K)
    h = single_cell(B, n, Z)
    y = product(B, h, x[None])[0]
    ref = Z.astype(np.clongdouble) @ x.astype(np.clongdouble)
    big = np.abs(Z).max(1) * np.abs(x).max()
    assert (np.abs(y - ref) <= K * 2.0 ** -48 * big + 2.0 ** -52 * np.abs(ref)).all()
    h.close()
