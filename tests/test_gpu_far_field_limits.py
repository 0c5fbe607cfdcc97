"""Far fields at the limits of their launch rules, against the sum over the
cells of one box's radiation integrals times e^{jk rhat . c_m}.  FP64 handles:
1e-11 of the largest |F| (the setup rows' tolerance).
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
