"""Products on grids of every kind of length: single-stage ones (1 to 8
points), two- and three-stage ones with radices 2 to 16, factors 7, unequal
sides, grids that fit the fused 2-D transforms and grids that take the
pass-based ones.  Every grid >= 2N - 1 embeds the lattice exactly, so each
product equals the oracle's direct sum: FP64 1e-10, FP32 3e-5 (the products'
tolerances).
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H
COEF = (1j * W.K0, 1.0, -1.0, 1j * W.K0)


@pytest.mark.parametrize("nx,ny,grid,R", [
    (1, 1, (1, 1), 1), (1, 3, (2, 5), 2), (3, 1, (5, 1), 1), (2, 2, (3, 4), 3), (4, 4, (7, 8), 1),
    (4, 3, (10, 9), 5), (6, 5, (12, 14), 1), (7, 8, (15, 16), 9), (9, 4, (18, 20), 1), (10, 6, (21, 25), 2),
    (5, 4, (27, 28), 1), (3, 3, (35, 49), 1), (3, 2, (63, 45), 2), (2, 3, (64, 60), 4), (2, 2, (30, 36), 1),
    (3, 3, (96, 100), 1), (2, 3, (200, 6), 3), (2, 2, (343, 3), 1), (2, 2, (128, 144), 1), (2, 1, (108, 1), 2),
])
def test_products_on_every_grid_length(emsurf_lib, nx, ny, grid, R):
    import torch
    from paper_1911_04576_gb300 import binding as B
    n, seed = 1, 17 * grid[0] + grid[1]
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, seed)
    Z = W.random_macromodels(2, 2 * E, seed + 1)
    tmap = np.arange(nx * ny, dtype=np.int32) % 2
    x = W.random_vectors(R, nu, seed + 2)
    h = B.emsurf_create(nx, ny, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=R, grid=grid)
    ref = lattice.matvec_direct(x, Lt, Kt, COEF, Z, tmap, idx, sgn, nu, nx, ny)
    xd = torch.from_numpy(x).cuda()
    for prec, tol in ((B.FP64, 1e-10), (B.FP32, 3e-5)):
        y = torch.full_like(xd, float("nan"))
        B.emsurf_matvec(h, xd, y, prec)
        y = y.cpu().numpy()
        for r in range(R):
            assert np.linalg.norm(y[r] - ref[r]) <= tol * np.linalg.norm(ref[r]), (prec, r)
    B.emsurf_check(h)
    h.close()
