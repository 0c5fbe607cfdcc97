"""Offset tables against the general tabulation of the same blocks.

emsurf_tabulate_offsets integrates one offset of each orbit of the box's
mirrors and reciprocity and fills the others with signed permutations;
emsurf_tabulate integrates every block it is given.  Both use the same
quadrature, so the tables agree to rounding: 1e-11 of the largest entry, the
setup rows' tolerance.  Square and rectangular cells, odd and even face
meshes, uniform and slab rows, lattices with one row and with unequal sides.
"""
import numpy as np
import pytest

from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H


@pytest.mark.parametrize("n,b,nx,ny,slab", [
    (1, A, 2, 3, False), (2, A, 4, 3, True), (2, 1.25 * A, 3, 4, False), (3, A, 3, 3, True),
    (3, 0.8 * A, 4, 2, True), (4, A, 5, 1, False), (2, A, 1, 1, False),
])
def test_offset_tables_equal_general_blocks(emsurf_lib, n, b, nx, ny, slab):
    import torch
    from paper_1911_04576_gb300 import binding as B
    zl = B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T) if slab else None
    E = 18 * n * n
    shape = (2 * ny - 1, 2 * nx - 1, E, E)
    L, K, L1, K1 = (torch.full(shape, float("nan"), dtype=torch.complex128, device="cuda") for _ in range(4))
    B.emsurf_tabulate_offsets(A, b, H, n, nx, ny, W.K0, L, K, zlevels=zl)
    box = B.emsurf_setup_box_mesh(A, b, H, n, zlevels=zl)
    d = [(dx, dy) for dy in range(-(ny - 1), ny) for dx in range(-(nx - 1), nx)]
    shifts = np.array([(dx * A, dy * b, 0.0) for dx, dy in d])
    near = np.array([abs(dx) <= 1 and abs(dy) <= 1 for dx, dy in d])
    B.emsurf_tabulate(box, box, shifts, near, W.K0, L1, K1)
    for T, T1 in ((L, L1), (K, K1)):
        T1 = T1.reshape(-1, E, E)
        ref = 0.5 * (T1 + T1.flip(0).transpose(1, 2))
        T = T.reshape(-1, E, E)
        assert float((T - ref).abs().max()) <= 1e-11 * float(ref.abs().max())
        # reciprocity holds entry by entry
        assert torch.equal(T.flip(0).transpose(1, 2), T)
