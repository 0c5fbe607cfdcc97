"""FP32 products of 2 to 13 rhs without tensor cores: every count that one
pass over the spectrum takes, equal groups above, more bins than resident
blocks and fewer, handles whose max_rhs is larger than the call's.  The
products' tolerance: 3e-5 against the oracle's direct sum.
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H
COEF = (1j * W.K0, 0.9, -1.1, 1j * W.K0)


@pytest.mark.parametrize("n,nx,ny,R,mx", [
    (2, 3, 2, 2, 2), (2, 20, 13, 3, 3), (2, 4, 4, 4, 5), (3, 2, 3, 5, 5), (2, 3, 3, 6, 8), (2, 2, 5, 7, 7),
    (4, 2, 1, 8, 8), (2, 3, 3, 9, 9), (3, 2, 2, 13, 13), (4, 1, 2, 3, 4), (1, 3, 3, 6, 6),
])
def test_products_of_a_few_rhs(emsurf_lib, n, nx, ny, R, mx):
    import torch
    from paper_1911_04576_gb300 import binding as B
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, n + R)
    Z = W.random_macromodels(2, 2 * E, R)
    tmap = np.arange(nx * ny, dtype=np.int32) % 2
    x = W.random_vectors(R, nu, 2)
    h = B.emsurf_create(nx, ny, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=mx)
    ref = lattice.matvec_direct(x, Lt, Kt, COEF, Z, tmap, idx, sgn, nu, nx, ny)
    xd = torch.from_numpy(x).cuda()
    y = torch.full_like(xd, float("nan"))
    B.emsurf_matvec(h, xd, y, B.FP32)
    y = y.cpu().numpy()
    for r in range(R):
        assert np.linalg.norm(y[r] - ref[r]) <= 3e-5 * np.linalg.norm(ref[r]), r
    B.emsurf_check(h)
    h.close()
