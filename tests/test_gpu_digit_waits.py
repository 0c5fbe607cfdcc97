"""Waits of the digit kernels that run out: emsurf_selftest_wait runs the
FP64-accuracy product and the macromodels' trailing update with operands that
never arrive, and reports only when every kernel has given up.  The limits go
from a single try to far more than the kernels' first copies need; afterwards
the same handle's product and a macromodel are bit for bit what they were.
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H, K0 = W.PERIOD, W.BOX_H, W.K0
COEF = (1j * K0, 1.0, -1.0, 1j * K0)


@pytest.mark.parametrize("n,nx,ny,R", [(1, 1, 1, 1), (2, 3, 2, 1), (3, 12, 13, 1), (2, 3, 2, 7)])
@pytest.mark.parametrize("limit", [1, 300, 5000])
def test_expired_waits_are_reported_and_leave_no_trace(emsurf_lib, n, nx, ny, R, limit):
    import torch
    from paper_1911_04576_gb300 import binding as B
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    g = torch.Generator(device="cuda").manual_seed(n)
    rnd = lambda *s: torch.randn(s, dtype=torch.complex128, device="cuda", generator=g)  # noqa: E731
    h = B.emsurf_create(nx, ny, E, nu, np.arange(nx * ny, dtype=np.int32) % 2, rnd(2, 2 * E, 2 * E),
                        rnd(2 * ny - 1, 2 * nx - 1, E, E), rnd(2 * ny - 1, 2 * nx - 1, E, E), COEF, idx, sgn,
                        precision=B.FP64, max_rhs=R, tables_on_device=True)
    x = rnd(R, nu)
    z = B.emsurf_setup_slab_zlevels(H, 2, W.SLAB_T)

    def outputs():
        y = torch.full_like(x, float("nan"))
        B.emsurf_matvec(h, x, y, B.FP64)
        Z = torch.empty((1, 144, 144), dtype=torch.complex128, device="cuda")
        B.emsurf_macromodel_slab_patch(A, A, H, 2, z, np.array([0.3 * W.LAMBDA]), 3, 2, W.EPS_SLAB, K0, Z)
        return y, Z

    before = outputs()
    assert torch.isfinite(torch.view_as_real(before[0])).all()
    for _ in range(2):
        B.emsurf_selftest_wait(h, limit)
        with pytest.raises(B.EmsurfError) as e:
            B.emsurf_check(h)
        assert e.value.status == B.EMSURF_ETIMEDOUT
        B.emsurf_check(h)
        for a, b in zip(outputs(), before):
            assert torch.equal(a, b)
    B.emsurf_check(h)
    h.close()
