"""Tensor-core products and preconditioner applies where the operand copies
hold only the live rows: 8, 9, 16, 17, 32, 33 and 40 rhs (boxes of 32, 64 and
128 rows, two groups), fewer rhs than the handle's max_rhs after a call with
all of them, sizes that are no multiple of eight sources.  Tolerances of the
tensor-core tests: products 3 * 2^-18 * sqrt(2E) against the oracle; the
preconditioner against its own one-rhs applies, 3 * 2^-18 * sqrt(n) with
subdomains of n <= 1100: 4e-4.
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H
COEF = (1j * W.K0, 1.0, -1.0, 1j * W.K0)


@pytest.mark.parametrize("n,nx,ny,mx,rhs", [(2, 3, 2, 40, (40, 33, 8, 32, 17)), (3, 2, 2, 16, (16, 9, 8)), (2, 2, 3, 64, (64, 10))])
def test_live_rows(emsurf_lib, n, nx, ny, mx, rhs):
    import torch
    from paper_1911_04576_gb300 import binding as B
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, n)
    Z = W.random_macromodels(2, 2 * E, 3)
    tmap = np.arange(nx * ny, dtype=np.int32) % 2
    h = B.emsurf_create(nx, ny, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=mx, tensor_cores=True)
    tol = 3 * 2.0 ** -18 * np.sqrt(2 * E)
    for R in rhs:
        x = W.random_vectors(R, nu, R)
        ref = lattice.matvec_direct(x, Lt, Kt, COEF, Z, tmap, idx, sgn, nu, nx, ny)
        xd = torch.from_numpy(x).cuda()
        y = torch.full_like(xd, float("nan"))
        B.emsurf_matvec(h, xd, y, B.FP32)
        y = y.cpu().numpy()
        for r in range(R):
            assert np.linalg.norm(y[r] - ref[r]) <= tol * np.linalg.norm(ref[r]), (R, r)
    B.emsurf_check(h)
    h.close()


def test_preconditioner_live_rows(emsurf_lib):
    import torch
    from paper_1911_04576_gb300 import binding as B
    n, nx, ny, mx = 3, 3, 3, 64
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, n)
    Z = W.random_macromodels(1, 2 * E, 3)
    Z += 50 * np.eye(2 * E) * np.abs(Z).max()          # well conditioned subdomains
    xy = B.emsurf_setup_unknown_xy(A, A, H, n, nx, ny, idx, nu)
    h = B.emsurf_create(nx, ny, E, nu, np.zeros(nx * ny, np.int32), Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=mx,
                        tensor_cores=True, unknown_xy=xy, cell=(A, A), precond_overlap=1.01 * A / n)
    x = torch.from_numpy(W.random_vectors(mx, nu, 5)).cuda()
    one = torch.empty_like(x)
    for r in range(mx):
        B.emsurf_precond_apply(h, x[r:r + 1].contiguous(), one[r:r + 1])
    for R in (64, 33, 32, 17, 16, 8):
        y = torch.full_like(x[:R], float("nan"))
        B.emsurf_precond_apply(h, x[:R].contiguous(), y)
        for r in range(R):
            assert float((y[r] - one[r]).norm()) <= 4e-4 * float(one[r].norm()), (R, r)
    B.emsurf_check(h)
    h.close()
