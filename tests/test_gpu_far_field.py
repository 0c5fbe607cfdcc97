"""Far field against the oracle on ragged lattices and direction counts.

The lattice sum works on tiles of 32 or 64 directions, 96 columns and 16
cells; the box integrals on translated triangle shapes (uniform and slab rows,
odd and even face meshes, rectangular cells).  FP64 handles: 1e-11 of the
largest |F|, the setup rows' tolerance.  MIXED handles sum the cells in FP32:
products and sums of M terms with phases rounded to FP32, (M + 8) 2^-24 of
sum_m |X_m|, which for random currents is about sqrt(M) times the largest
|F|: M = 35 gives 1.5e-5.
"""
import numpy as np
import pytest

from oracle import lattice, operators
from oracle.mesh import box_mesh, slab_zlevels
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H, K0 = W.PERIOD, W.BOX_H, W.K0
COEF = (1j * K0, 1.0, -1.0, 1j * K0)


@pytest.mark.parametrize("prec,n,nx,ny,b,slab,R,nd", [
    ("FP64", 2, 1, 1, A, False, 1, 1), ("FP64", 3, 5, 4, 1.25 * A, True, 2, 67),
    ("MIXED", 3, 5, 7, A, True, 1, 130), ("MIXED", 2, 2, 9, 0.8 * A, False, 3, 33), ("MIXED", 4, 1, 2, A, True, 1, 64),
])
def test_far_field_matches_oracle(emsurf_lib, prec, n, nx, ny, b, slab, R, nd):
    import torch
    from paper_1911_04576_gb300 import binding as B
    zl = slab_zlevels(H, n, W.SLAB_T) if slab else None
    box = box_mesh(A, b, H, n, zl)
    E = box.n_rwg
    idx, sgn, nu = B.emsurf_setup_overlap(n, nx, ny)
    Lt, Kt = W.random_tables(nx, ny, E, 3)
    h = B.emsurf_create(nx, ny, E, nu, np.zeros(nx * ny, np.int32), W.random_macromodels(1, 2 * E, 4), Lt, Kt, COEF,
                        idx, sgn, precision=getattr(B, prec), max_rhs=R)
    rng = np.random.default_rng(nd)
    Y = rng.standard_normal((R, nu)) + 1j * rng.standard_normal((R, nu))
    th, ph = rng.uniform(0, np.pi, nd), rng.uniform(0, 2 * np.pi, nd)
    rhat = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], -1)
    F = torch.full((R, nd, 3), float("nan"), dtype=torch.complex128, device="cuda")
    rcs = torch.full((R, nd), float("nan"), dtype=torch.float64, device="cuda")
    B.emsurf_far_field(h, A, b, H, n, K0, torch.from_numpy(Y).cuda(), rhat, F, rcs, zlevels=zl)
    F = F.cpu().numpy()
    tol = 1e-11 if prec == "FP64" else (nx * ny + 8) * 2.0 ** -24 * np.sqrt(nx * ny)
    for r in range(R):
        Yl = lattice.gather(Y[r], idx, sgn, nx * ny, 2 * E)
        ref = 0
        for m in range(nx * ny):
            rad = operators.radiation_vectors(box, lattice.cell_shift(m % nx, m // nx, A, b), K0, rhat)
            ref = ref + operators.far_field(rad, rhat, K0, Yl[m, :E], Yl[m, E:])
        assert np.abs(F[r] - ref).max() <= tol * np.abs(ref).max()
        np.testing.assert_allclose(rcs[r].cpu().numpy(), 4 * np.pi * np.sum(np.abs(F[r]) ** 2, -1), rtol=1e-12)
    h.close()
