"""Chains of products without a host wait between them: kernels that start
while the one before them drains must still see its results and leave its
inputs alone.  The same chain with a synchronisation after every product is
bitwise equal (every kernel of these products is deterministic).
"""
import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H
COEF = (1j * W.K0, 1.0, -1.0, 1j * W.K0)


@pytest.mark.parametrize("n,nx,ny,R,mx,prec", [
    (2, 5, 4, 1, 1, "FP32"), (2, 12, 12, 1, 1, "FP32"), (2, 5, 4, 3, 3, "FP32"), (2, 4, 3, 9, 9, "FP32"),
    (2, 5, 4, 1, 1, "FP64"), (2, 12, 12, 1, 1, "FP64"), (2, 4, 3, 7, 7, "FP64"), (1, 2, 2, 2, 2, "FP64"),
])
def test_chain_equals_synchronised_chain(emsurf_lib, n, nx, ny, R, mx, prec):
    import torch
    from paper_1911_04576_gb300 import binding as B
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, n)
    if mx == 1:        # reciprocal tables: the half spectrum of one rhs
        Lt = 0.5 * (Lt + Lt[::-1, ::-1].swapaxes(2, 3))
        Kt = 0.5 * (Kt + Kt[::-1, ::-1].swapaxes(2, 3))
    Z = W.random_macromodels(3, 2 * E, 3)
    tmap = (np.arange(nx * ny) % 3).astype(np.int32)
    h = B.emsurf_create(nx, ny, E, nu, tmap, Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=mx)
    p = getattr(B, prec)
    x0 = torch.from_numpy(W.random_vectors(R, nu, 7)).cuda()

    def chain(sync):
        v = [x0.clone(), torch.empty_like(x0)]
        for s in range(24):
            B.emsurf_matvec(h, v[s & 1], v[~s & 1], p)
            if sync:
                torch.cuda.synchronize()
            v[~s & 1] /= v[~s & 1].abs().max()      # keeps the chain in range
        torch.cuda.synchronize()
        return v[0]

    ref = chain(True)
    assert torch.isfinite(torch.view_as_real(ref)).all()
    for _ in range(3):
        assert torch.equal(chain(False), ref)
    B.emsurf_check(h)
    h.close()


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_captured_product_equals_direct_one(emsurf_lib, prec):
    import torch
    from paper_1911_04576_gb300 import binding as B
    n, nx, ny = 2, 4, 3
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, n)
    Z = W.random_macromodels(1, 2 * E, 3)
    h = B.emsurf_create(nx, ny, E, nu, np.zeros(nx * ny, np.int32), Z, Lt, Kt, COEF, idx, sgn, precision=B.MIXED, max_rhs=2)
    x = torch.from_numpy(W.random_vectors(2, nu, 7)).cuda()
    y, z = torch.empty_like(x), torch.empty_like(x)
    p = getattr(B, prec)
    B.emsurf_matvec(h, x, y, p)
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=st):
        B.emsurf_matvec(h, x, z, p)
    for _ in range(3):
        z.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, z)
    h.close()
