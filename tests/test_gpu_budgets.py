"""Device-memory budgets: whatever a handle of a smaller budget can do, one of a
larger budget can (digit planes that fit now must not take the room of what is
allocated after them), and every handle gives the same FP64 product (1e-12 against
the handle without a limit, the tile edges' bound).
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H, K0 = W.PERIOD, W.BOX_H, W.K0
COEF = (1j * K0, 0.9, -1.1, 1j * K0)


@pytest.mark.parametrize("n,nx,ny,R,prec,extra", [
    (1, 3, 2, 1, "FP64", ""), (2, 3, 2, 4, "FP64", "share"), (2, 3, 2, 4, "MIXED", "share"), (2, 4, 4, 1, "MIXED", ""),
    (2, 3, 3, 13, "FP64", ""), (3, 5, 4, 9, "FP64", "precond"), (3, 3, 2, 1, "MIXED", "precond"),
])
def test_every_budget_above_the_smallest_serves(emsurf_lib, n, nx, ny, R, prec, extra):
    import torch
    from paper_1911_04576_gb300 import binding as B
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    g = torch.Generator(device="cuda").manual_seed(n)
    rnd = lambda *s: torch.randn(s, dtype=torch.complex128, device="cuda", generator=g)  # noqa: E731
    # no reciprocity, so that MIXED handles keep the whole FP32 spectrum
    L, K, Z = rnd(2 * ny - 1, 2 * nx - 1, E, E), rnd(2 * ny - 1, 2 * nx - 1, E, E), rnd(2, 2 * E, 2 * E)
    Z += 30 * torch.eye(2 * E, device="cuda")
    kw = dict(precision=getattr(B, prec), max_rhs=R, tables_on_device=True)
    if extra == "precond":
        kw.update(unknown_xy=B.emsurf_setup_unknown_xy(A, A, H, n, nx, ny, idx, nu), cell=(A, A), precond_overlap=A / n)

    def create(budget):
        return B.emsurf_create(nx, ny, E, nu, np.arange(nx * ny, dtype=np.int32) % 2, Z, L, K, COEF, idx, sgn,
                               device_mem_budget=int(budget), **kw)

    full = create(0)
    x = rnd(R, nu)
    ref = torch.empty_like(x)
    B.emsurf_matvec(full, x, ref, B.FP64)
    if extra == "share":
        kw["share"] = full
    lo, hi = 1 << 10, 1 << 34
    while hi > 1.02 * lo:
        mid = (lo * hi) ** 0.5
        try:
            create(mid).close()
            hi = mid
        except B.EmsurfError as e:
            assert e.status == B.EMSURF_ENOMEM
            lo = mid
    for b in np.geomspace(hi, 4 * hi, 24):
        h = create(b)
        y = torch.full_like(x, float("nan"))
        B.emsurf_matvec(h, x, y, B.FP64)
        assert float((y - ref).norm()) <= 1e-12 * float(ref.norm()), b / hi
        assert B.emsurf_query(h)[2] <= b
        h.close()
    full.close()
