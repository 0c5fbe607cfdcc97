"""Macromodels of a cell library against the same cells one at a time: types
of equal mesh size are tabulated and eliminated together (several scratch
chunks at n = 4), empty boxes in between break the runs.  Every type goes
through the same quadrature and elimination: 1e-12 in norm covers a
difference in the order of sums.
"""
import numpy as np
import pytest

from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H, K0 = W.PERIOD, W.BOX_H, W.K0


@pytest.mark.parametrize("n,patch_n,layers,sides,eps", [
    (2, 3, 2, (0.2, 0.3, 0.0, 0.0, 0.41), 3.0 * (1 - 0.001j)),
    (3, 4, 1, (0.0, 0.15, 0.45), 2.2 * (1 - 0.3j)),
    (4, 4, 3, tuple(np.linspace(0.15, 0.45, 17)), 3.0 * (1 - 0.001j)),
    (2, 5, 4, (0.33,), 1.0),
])
def test_library_equals_single_cells(emsurf_lib, n, patch_n, layers, sides, eps):
    import torch
    from paper_1911_04576_gb300 import binding as B
    z = B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T)
    K = 36 * n * n

    def models(s):
        Z = torch.full((len(s), K, K), float("nan"), dtype=torch.complex128, device="cuda")
        B.emsurf_macromodel_slab_patch(A, A, H, n, z, np.array(s) * W.LAMBDA, patch_n, layers, eps, K0, Z)
        return Z

    Z = models(sides)
    for t in sorted({0, 1 % len(sides), len(sides) // 2, len(sides) - 1}):
        one = models(sides[t:t + 1])[0]
        assert float((Z[t] - one).norm()) <= 1e-12 * float(one.norm()), t


@pytest.mark.parametrize("n,patch_n,layers,side", [(2, 1, 1, 0.3), (2, 5, 4, 0.2), (2, 6, 5, 0.4)])
def test_elimination_of_few_and_many_interior_unknowns(emsurf_lib, n, patch_n, layers, side):
    """Panels of less than 32 columns, remainders, and interior blocks too
    large for shared memory, against the oracle (same quadrature: the slab
    tests' 1e-10 in norm); the second type is an empty cell."""
    import torch
    from oracle import macromodel
    from oracle.mesh import box_mesh, slab_zlevels
    from paper_1911_04576_gb300 import binding as B
    K = 36 * n * n
    sides = np.array([side * W.LAMBDA, 0.0])
    Z = torch.full((2, K, K), float("nan"), dtype=torch.complex128, device="cuda")
    B.emsurf_macromodel_slab_patch(A, A, H, n, B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T), sides, patch_n, layers,
                                   W.EPS_SLAB, K0, Z)
    box = box_mesh(A, A, H, n, slab_zlevels(H, n, W.SLAB_T))
    for t, s in enumerate(sides):
        ref = macromodel.slab_patch(box, n, s, patch_n, W.EPS_SLAB, K0, W.SLAB_T, ring_layers=layers)
        assert np.linalg.norm(Z[t].cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref), t
