"""Products of lattices of a few cells with many right-hand sides: transforms
whose CTAs hold up to 32 lanes of a small grid, operand splits whose blocks share
a bin or a tile.  Lane counts that are not a multiple of a CTA's, lengths of one
stage, one row.  The products' tolerances: 3e-5 (FP32, with and without tensor
cores) and 1e-12 (FP64) against the oracle's direct sum.
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H
COEF = (1j * W.K0, 0.9, -1.1, 1j * W.K0)


@pytest.mark.parametrize("n,nx,ny,R", [
    (1, 1, 1, 1), (2, 1, 1, 33), (3, 1, 1, 64), (2, 2, 1, 17), (2, 3, 3, 20), (3, 11, 1, 9), (2, 1, 5, 31), (4, 2, 2, 13),
    (3, 4, 3, 8), (2, 6, 5, 21), (1, 7, 2, 40),
])
def test_products_with_many_rhs(emsurf_lib, n, nx, ny, R):
    import torch
    from paper_1911_04576_gb300 import binding as B
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, n + R)
    T = min(2, nx * ny)
    Z = W.random_macromodels(T, 2 * E, R)
    tmap = np.arange(nx * ny, dtype=np.int32) % T
    x = W.random_vectors(R, nu, 2)
    ref = lattice.matvec_direct(x, Lt, Kt, COEF, Z, tmap, idx, sgn, nu, nx, ny)
    xd = torch.from_numpy(x).cuda()
    for tc, prec, tol in ((False, B.FP64, 1e-12), (False, B.FP32, 3e-5), (True, B.FP32, 3e-5)):
        h = B.emsurf_create(nx, ny, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=R, tensor_cores=tc)
        y = torch.full_like(xd, float("nan"))
        B.emsurf_matvec(h, xd, y, prec)
        y = y.cpu().numpy()
        for r in range(R):
            assert np.linalg.norm(y[r] - ref[r]) <= tol * np.linalg.norm(ref[r]), (tc, prec, r)
        B.emsurf_check(h)
        h.close()
