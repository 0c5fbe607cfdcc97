"""FP64 products on the digit planes at the edges of their tiles: 4E and 2K
rows around 128, sources around 16 and 32, 1 to 6 rhs per launch and several
launches, cells of a type that do not fill an entry, rows and vectors of very
different size, non-finite entries, handles that share planes and budgets that
have no room for them.

Tolerance: the digits hold 55 bits below the largest component of a row or a
vector and the dropped products weigh less than n 2^-48 of row maximum times
vector maximum (n sources); with random entries a sum is about sqrt(n) of that
maximum, so n <= 2304 sources give errors below 48 * 2^-48 = 2e-13 (the most
with more than 990, which take a bit less) and the transforms around them a
few 1e-16: 1e-12 bounds both.
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H
COEF = (1j * W.K0, 0.9 - 0.2j, -1.1, 0.5 + 1j * W.K0)
TOL = 1e-12


def build(n, nx, ny, T, seed):
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, seed)
    Z = W.random_macromodels(T, 2 * E, seed + 1)
    tmap = np.random.default_rng(seed + 2).integers(0, T, nx * ny).astype(np.int32)
    return E, idx, sgn, nu, Lt, Kt, Z, tmap


def product(B, h, x):
    import torch
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    y = torch.full_like(xd, float("nan"))
    B.emsurf_matvec(h, xd, y, B.FP64)
    return y.cpu().numpy()


@pytest.mark.parametrize("n,nx,ny,T,R,mx", [
    (1, 1, 1, 1, 1, 1), (1, 2, 1, 2, 2, 13), (1, 4, 3, 1, 13, 13), (2, 3, 2, 6, 3, 7), (2, 1, 3, 2, 4, 4),
    (2, 3, 3, 1, 5, 5), (3, 2, 1, 2, 6, 6), (3, 1, 2, 1, 7, 8), (3, 3, 3, 2, 1, 2), (4, 2, 1, 1, 2, 2), (4, 1, 1, 1, 12, 12),
    (6, 1, 1, 1, 2, 2), (8, 1, 1, 1, 1, 1),
])
def test_products_at_tile_edges(emsurf_lib, n, nx, ny, T, R, mx):
    from paper_1911_04576_gb300 import binding as B
    E, idx, sgn, nu, Lt, Kt, Z, tmap = build(n, nx, ny, T, 31 * n + nx + R)
    h = B.emsurf_create(nx, ny, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=mx)
    # rhs of very different size: each has its own exponents
    x = W.random_vectors(R, nu, 5) * 10.0 ** np.linspace(-150, 90, R)[:, None]
    ref = lattice.matvec_direct(x, Lt, Kt, COEF, Z, tmap, idx, sgn, nu, nx, ny)
    y = product(B, h, x)
    for r in range(R):
        assert np.linalg.norm(y[r] - ref[r]) <= TOL * np.linalg.norm(ref[r]), r
    assert (product(B, h, 0 * x) == 0).all()
    B.emsurf_check(h)
    h.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, complex(0, -np.inf)])
def test_non_finite_entries_show_in_every_rhs_they_reach(emsurf_lib, bad):
    from paper_1911_04576_gb300 import binding as B
    E, idx, sgn, nu, Lt, Kt, Z, tmap = build(2, 2, 2, 2, 3)
    h = B.emsurf_create(2, 2, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=3)
    x = W.random_vectors(3, nu, 5)
    ref = lattice.matvec_direct(x, Lt, Kt, COEF, Z, tmap, idx, sgn, nu, 2, 2)
    x[1, nu // 2] = bad
    y = product(B, h, x)
    assert not np.isfinite(y[1]).any()
    for r in (0, 2):
        assert np.linalg.norm(y[r] - ref[r]) <= TOL * np.linalg.norm(ref[r]), r
    B.emsurf_check(h)
    h.close()


def test_shared_and_budgeted_handles(emsurf_lib):
    """A sharer takes the planes over; every budget that a handle is built in
    gives the same products."""
    from paper_1911_04576_gb300 import binding as B
    E, idx, sgn, nu, Lt, Kt, Z, tmap = build(2, 4, 3, 2, 9)
    x = W.random_vectors(7, nu, 5)
    ref = lattice.matvec_direct(x, Lt, Kt, COEF, Z, tmap, idx, sgn, nu, 4, 3)
    kw = dict(precision=B.MIXED, max_rhs=7)
    h = B.emsurf_create(4, 3, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, **kw)
    full = B.emsurf_query(h)[2]
    hs = [h, B.emsurf_create(4, 3, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, share=h, **kw)]
    for part in (2.5, 2.0, 1.8, 1.6, 1.5, 1.4, 1.3, 1.2, 1.1, 1.0, 0.9):
        try:
            hs.append(B.emsurf_create(4, 3, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, device_mem_budget=int(full * part),
                                      **kw))
        except B.EmsurfError as e:
            assert e.status == B.EMSURF_ENOMEM
    assert len(hs) >= 3
    hs.append(B.emsurf_create(4, 3, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, share=h,
                              device_mem_budget=B.emsurf_query(hs[1])[2] - (1 << 18), **kw))
    for k, g in enumerate(hs):
        y = product(B, g, x)
        for r in range(7):
            assert np.linalg.norm(y[r] - ref[r]) <= TOL * np.linalg.norm(ref[r]), (k, r)
        B.emsurf_check(g)
    for g in reversed(hs):
        g.close()
