"""Offset tables of lattices whose pair classes take several chunks of the
table of slot integrals (5 x 5 quads per face; many offsets) or are few (one
row, one box), square and rectangular cells, against the general tabulation of
each block: both integrate with the same quadrature, so 1e-11 of the largest
entry, the setup rows' tolerance.
"""
import numpy as np
import pytest

from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H


@pytest.mark.parametrize("n,b,nx,ny,slab", [
    (5, 0.9 * A, 7, 5, True), (4, A, 12, 12, True), (4, 1.1 * A, 1, 9, False), (3, A, 6, 6, False), (5, A, 1, 1, True),
])
def test_offset_tables_from_pair_classes(emsurf_lib, n, b, nx, ny, slab):
    import torch
    from paper_1911_04576_gb300 import binding as B
    zl = B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T) if slab else None
    E = 18 * n * n
    L, K = (torch.full((2 * ny - 1, 2 * nx - 1, E, E), float("nan"), dtype=torch.complex128, device="cuda") for _ in range(2))
    B.emsurf_tabulate_offsets(A, b, H, n, nx, ny, W.K0, L, K, zlevels=zl)
    box = B.emsurf_setup_box_mesh(A, b, H, n, zlevels=zl)
    r = np.random.default_rng(n + nx)
    d = [(0, 0), (nx - 1, ny - 1), (1 - nx, ny - 1), (min(1, nx - 1), 0)]
    d += [(int(r.integers(1 - nx, nx)), int(r.integers(1 - ny, ny))) for _ in range(12)]
    d += [(-x, -y) for x, y in d]
    shifts = np.array([(x * A, y * b, 0.0) for x, y in d])
    near = np.array([abs(x) <= 1 and abs(y) <= 1 for x, y in d])
    L1, K1 = (torch.empty((len(d), E, E), dtype=torch.complex128, device="cuda") for _ in range(2))
    B.emsurf_tabulate(box, box, shifts, near, W.K0, L1, K1)
    for T, T1 in ((L, L1), (K, K1)):
        m = len(d) // 2
        ref = 0.5 * (T1[:m] + T1[m:].transpose(1, 2))
        for q in range(m):
            got = T[d[q][1] + ny - 1, d[q][0] + nx - 1]
            assert float((got - ref[q]).abs().max()) <= 1e-11 * float(ref.abs().max()), d[q]
        assert torch.equal(T.flip(0, 1).transpose(2, 3), T)
