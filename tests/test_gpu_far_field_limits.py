"""Far fields at the limits of their launch rules, against the sum over the
cells of one box's radiation integrals times e^{jk rhat . c_m}: few directions
with more right-hand sides than a warp has lanes, many of both (32 rhs at a time,
one per lane), a lattice whose phase tables
leave room for 8 cells per stage only (nx + ny from 391 to 422 in FP64), a box
whose triangle phases are formed per member, and a nearly full device.

FP64 handles: 1e-11 of the largest |F| (the setup rows' tolerance).  MIXED and
FP32 handles sum M cells in FP32: (M + 8) 2^-24 sqrt(M) of the largest |F| as in
the ragged lattices' test, with sums of one box to single precision.
"""
import numpy as np
import pytest

from oracle import lattice, operators
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H, K0 = W.PERIOD, W.BOX_H, W.K0
COEF = (1j * K0, 1.0, -1.0, 1j * K0)


def zeros(*shape):
    import torch
    return torch.zeros(shape, dtype=torch.complex128, device="cuda")


def handle(B, n, nx, ny, prec):
    """A handle without coupling (the far field reads its lattice only)."""
    E = 18 * n * n
    idx, sgn, nu = B.emsurf_setup_overlap(n, nx, ny)
    T = zeros(2 * ny - 1, 2 * nx - 1, E, E)
    h = B.emsurf_create(nx, ny, E, nu, np.zeros(nx * ny, np.int32), zeros(1, 2 * E, 2 * E), T, T, COEF, idx, sgn,
                        precision=prec, max_rhs=1, tables_on_device=True)
    return h, idx, sgn, nu


def directions(nd, seed):
    rng = np.random.default_rng(seed)
    th, ph = rng.uniform(0, np.pi, nd), rng.uniform(0, 2 * np.pi, nd)
    return np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], -1)


def reference(box, nx, ny, Y, idx, sgn, rhat):
    E = box.n_rwg
    rad = operators.radiation_vectors(box, np.zeros(3), K0, rhat)
    c = np.array([lattice.cell_shift(m % nx, m // nx, A, A) for m in range(nx * ny)])
    ph = np.exp(1j * K0 * rhat @ c.T)
    out = []
    for y in Y:
        S = ph @ lattice.gather(y, idx, sgn, nx * ny, 2 * E)                  # [D, 2E]
        N, L = (np.einsum("dm,dmx->dx", s, rad) for s in (S[:, :E], S[:, E:]))
        Np = N - np.sum(rhat * N, -1, keepdims=True) * rhat
        out.append(-(1j * K0 / (4 * np.pi)) * (Np - np.cross(rhat, L)))
    return np.array(out)


@pytest.mark.parametrize("prec,n,nx,ny,R,nd", [
    ("FP64", 1, 3, 2, 33, 3), ("MIXED", 2, 2, 2, 70, 1), ("MIXED", 1, 4, 3, 32, 130), ("FP64", 2, 1, 1, 31, 2),
    ("MIXED", 1, 2, 2, 70, 1300), ("FP64", 2, 2, 1, 33, 2600), ("MIXED", 3, 1, 1, 64, 1300),
    ("FP64", 1, 390, 1, 1, 40), ("FP64", 1, 391, 1, 2, 33), ("FP64", 1, 400, 1, 1, 1),
])
def test_many_rhs_and_long_lattices(emsurf_lib, prec, n, nx, ny, R, nd):
    import torch
    from paper_1911_04576_gb300 import binding as B
    h, idx, sgn, nu = handle(B, n, nx, ny, getattr(B, prec))
    rng = np.random.default_rng(nd + R)
    Y = rng.standard_normal((R, nu)) + 1j * rng.standard_normal((R, nu))
    rhat = directions(nd, R)
    F = torch.full((R, nd, 3), float("nan"), dtype=torch.complex128, device="cuda")
    rcs = torch.full((R, nd), float("nan"), dtype=torch.float64, device="cuda")
    B.emsurf_far_field(h, A, A, H, n, K0, torch.from_numpy(Y).cuda(), rhat, F, rcs)
    F, rcs = F.cpu().numpy(), rcs.cpu().numpy()
    ref = reference(box_mesh(A, A, H, n), nx, ny, Y, idx, sgn, rhat)
    M = nx * ny
    tol = 1e-11 if prec == "FP64" else (M + 8) * 2.0 ** -24 * np.sqrt(M)
    for r in range(R):
        assert np.abs(F[r] - ref[r]).max() <= tol * np.abs(ref).max(), r
    np.testing.assert_allclose(rcs, 4 * np.pi * np.sum(np.abs(F) ** 2, -1), rtol=1e-12)
    h.close()


def test_box_of_many_triangles_and_shapes(emsurf_lib):
    """13 x 13 quads per face in rows of 13 different heights: the phases of four
    warps do not fit in shared memory."""
    import torch
    from paper_1911_04576_gb300 import binding as B
    n = 13
    zl = H * (np.arange(n + 1) / n) ** 1.3
    h, idx, sgn, nu = handle(B, n, 1, 1, B.FP32)
    rng = np.random.default_rng(3)
    Y = rng.standard_normal((2, nu)) + 1j * rng.standard_normal((2, nu))
    rhat = directions(5, 4)
    F = torch.full((2, 5, 3), float("nan"), dtype=torch.complex128, device="cuda")
    B.emsurf_far_field(h, A, A, H, n, K0, torch.from_numpy(Y).cuda(), rhat, F, zlevels=zl)
    ref = reference(box_mesh(A, A, H, n, zl), 1, 1, Y, idx, sgn, rhat)
    assert np.abs(F.cpu().numpy() - ref).max() <= 9 * 2.0 ** -24 * np.abs(ref).max()
    h.close()


def test_lattice_beyond_the_phase_tables_is_refused(emsurf_lib):
    import torch
    from paper_1911_04576_gb300 import binding as B
    h, _, _, nu = handle(B, 1, 211, 212, B.FP32)
    F = torch.zeros((1, 1, 3), dtype=torch.complex128, device="cuda")
    B.emsurf_far_field(h, A, A, H, 1, K0, zeros(1, nu), directions(1, 0), F)      # 423 columns and rows fit in FP32
    h.close()
    h, _, _, nu = handle(B, 1, 400, 23, B.FP64)
    with pytest.raises(B.EmsurfError) as e:
        B.emsurf_far_field(h, A, A, H, 1, K0, zeros(1, nu), directions(1, 0), F)
    assert e.value.status == B.EMSURF_EINVAL
    h.close()


def test_many_rhs_on_a_nearly_full_device(emsurf_lib):
    """The column sums and phase tables of a chunk of directions stay below
    512 MB: 100 rhs of K = 576 in FP64 work with 1 GB left on the device."""
    import torch
    from paper_1911_04576_gb300 import binding as B
    n, R, nd = 4, 100, 4096
    h, idx, sgn, nu = handle(B, n, 2, 1, B.FP64)
    rng = np.random.default_rng(1)
    Y = rng.standard_normal((R, nu)) + 1j * rng.standard_normal((R, nu))
    rhat = directions(nd, 2)
    Yd = torch.from_numpy(Y).cuda()
    F = torch.empty((R, nd, 3), dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")
    try:
        B.emsurf_far_field(h, A, A, H, n, K0, Yd, rhat, F)
    finally:
        del fill
        torch.cuda.empty_cache()
    pick = [0, 1, 2047, 4000, 4095]
    ref = reference(box_mesh(A, A, H, n), 2, 1, Y[[0, 57, 99]], idx, sgn, rhat[pick])
    got = F[[0, 57, 99]][:, pick].cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-11 * np.abs(ref).max()
    h.close()
