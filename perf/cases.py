"""The work whose speed counts: products, preconditioner applies, solves, setup and far
fields of patch-on-slab lattices, as a program that uses the library calls them.

A case is one public call (or, for `solve`, one whole solve) on one lattice.  Sizes are
those of the repository's workloads and of its serving stream (lattices 8 to 64 cells wide,
boxes meshed 3 x 3 or 4 x 4 per face, 1 to 32 right-hand sides) with rectangular and odd
lattices among them.  Every input comes from the seed: patch sides, type map, vectors,
incidence angle, frequency of a tabulation.

Results of the FP32 operator are kept in 32 bits (complex64, float32), the precision they
are computed in; those of the FP64 operator and of the setup stay in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1911_04576_gb300 import binding as B
from paper_1911_04576_gb300 import workloads as W

A, H, K0 = W.PERIOD, W.BOX_H, W.K0
COEF = (1j * K0, 1.0, -1.0, 1j * K0)
PRECISION = {"fp32": B.FP32, "fp64": B.FP64, "mixed": B.MIXED}
DEV = "cuda"


def listed():
    return [
        # the smallest lattice of the serving stream, one right-hand side: launches and latency
        dict(name="product_fp32_8x8_k324", kind="product", nx=8, ny=8, n=3, types=9, rhs=1, operator="fp32", tc=False, mirrors=False),
        # the product inside every iteration of the headline solve
        dict(name="product_fp32_16x16_k576", kind="product", nx=16, ny=16, n=4, types=32, rhs=1, operator="fp32", tc=False, mirrors=False),
        # the same with one stored bin per mirror orbit
        dict(name="product_fp32_mirrors_16x16_k576", kind="product", nx=16, ny=16, n=4, types=32, rhs=1, operator="fp32", tc=False, mirrors=True),
        # a few right-hand sides of a rectangular lattice whose grid sides are not powers of two
        dict(name="product_fp32_r3_20x13_k324", kind="product", nx=20, ny=13, n=3, types=16, rhs=3, operator="fp32", tc=False, mirrors=False),
        # many plane waves at once, on the tensor cores
        dict(name="product_fp32_r32_24x24_k576", kind="product", nx=24, ny=24, n=4, types=32, rhs=32, operator="fp32", tc=True, mirrors=False),
        # the FP64-accuracy product: refinement residuals, every iteration of the plain FP64 solve
        dict(name="product_fp64_16x16_k576", kind="product", nx=16, ny=16, n=4, types=32, rhs=1, operator="fp64", tc=False, mirrors=False),
        # the same for several right-hand sides of a ragged lattice
        dict(name="product_fp64_r6_12x9_k576", kind="product", nx=12, ny=9, n=4, types=16, rhs=6, operator="fp64", tc=False, mirrors=False),
        # the preconditioner apply of a solve with 16 right-hand sides
        dict(name="precond_r16_12x12_k324", kind="precond", nx=12, ny=12, n=3, types=16, rhs=16, tc=True),
        # the headline: a whole mixed-precision solve to 1e-6
        dict(name="solve_16x16_k576", kind="solve", nx=16, ny=16, n=4, types=32, rhs=1, tc=False),
        # setup of a new lattice or frequency: offset tables
        dict(name="tabulate_16x16_k576", kind="tabulate", nx=16, ny=16, n=4),
        # setup of a new cell library: macromodels
        dict(name="macromodels_32_k576", kind="macromodel", n=4, types=32),
        # bistatic RCS of a solved array on a 1 degree grid
        dict(name="far_field_16x16_k576", kind="far_field", nx=16, ny=16, n=4, rhs=1, step=1.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "product", "product", "product", "precond", "solve", "tabulate", "macromodel", "far_field"])
    n = rng.choice([2, 3, 3, 4, 4])
    nx, ny = _log(rng, 3, 22), _log(rng, 3, 22)
    if rng.random() < 0.4:
        ny = nx
    case = dict(kind=kind, nx=nx, ny=ny, n=n, types=_log(rng, 2, 32))
    if kind == "product":
        case["rhs"] = rng.choice([1, 1, 1, _log(rng, 2, 7), _log(rng, 2, 7), _log(rng, 8, 32)])
        case["operator"] = rng.choice(["fp32", "fp32", "fp64"]) if case["rhs"] < 8 else "fp32"
        case["tc"] = case["rhs"] >= 8
        case["mirrors"] = case["rhs"] == 1 and case["operator"] == "fp32" and n % 2 == 0 and rng.random() < 0.5
    elif kind == "precond":
        case["n"] = rng.choice([3, 4])          # the overlap of one mesh cell has to stay below half a period
        case["rhs"] = rng.choice([1, 1, _log(rng, 2, 7), _log(rng, 8, 32)])
        case["tc"] = case["rhs"] >= 8
    elif kind == "solve":
        case["nx"], case["ny"], case["n"] = _log(rng, 3, 14), _log(rng, 3, 14), rng.choice([3, 4])
        case["rhs"] = rng.choice([1, 1, _log(rng, 2, 16)])
        case["tc"] = case["rhs"] >= 8
    elif kind == "tabulate":
        case["nx"], case["ny"] = min(nx, 16), min(ny, 16)
        del case["types"]
    elif kind == "macromodel":
        del case["nx"], case["ny"]
    else:
        del case["types"]
        case["rhs"] = _log(rng, 1, 8)
        case["step"] = rng.choice([1.0, 2.0, 3.0])
    return case


# ---------------------------------------------------------------- inputs
def _rng(seed):
    return np.random.default_rng([seed, 1911])


def _random(shape, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn(shape, dtype=torch.complex128, device=DEV, generator=g)


def _cells(case, seed):
    """The lattice's cell library and map: patch sides (m), type of each cell."""
    r = _rng(seed)
    sides = r.uniform(0.15, 0.45, case["types"]) * W.LAMBDA
    tmap = r.integers(0, case["types"], case["nx"] * case["ny"]).astype(np.int32)
    return sides, tmap


def _macromodels(n, sides):
    zl = B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T)
    Z = torch.empty((len(sides), 36 * n * n, 36 * n * n), dtype=torch.complex128, device=DEV)
    B.emsurf_macromodel_slab_patch(A, A, H, n, zl, sides, 4, W.RING_LAYERS, W.EPS_SLAB, K0, Z)
    return Z


def _tables(nx, ny, n, k):
    E = 18 * n * n
    L = torch.empty((2 * ny - 1, 2 * nx - 1, E, E), dtype=torch.complex128, device=DEV)
    K = torch.empty_like(L)
    B.emsurf_tabulate_offsets(A, A, H, n, nx, ny, k, L, K, zlevels=B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T))
    return L, K


def _operator(case, seed):
    """What a lattice's handle is made of."""
    nx, ny, n = case["nx"], case["ny"], case["n"]
    sides, tmap = _cells(case, seed)
    L, K = _tables(nx, ny, n, K0)
    idx, sgn, nu = B.emsurf_setup_overlap(n, nx, ny)
    return dict(L=L, K=K, Z=_macromodels(n, sides), tmap=tmap, idx=idx, sgn=sgn, nu=nu)


def _handle(case, op, precision, precond):
    nx, ny, n = case["nx"], case["ny"], case["n"]
    xy = B.emsurf_setup_unknown_xy(A, A, H, n, nx, ny, op["idx"], op["nu"]) if precond else None
    return B.emsurf_create(nx, ny, 18 * n * n, op["nu"], op["tmap"], op["Z"], op["L"], op["K"], COEF, op["idx"], op["sgn"],
                           precision=precision, max_rhs=case["rhs"], tables_on_device=True, unknown_xy=xy, cell=(A, A),
                           precond_overlap=A / n if precond else 0.0, tensor_cores=case.get("tc", False),
                           mirrors=B.emsurf_setup_box_mirrors(A, A, n) if case.get("mirrors") else None)


def _directions(step):
    th = np.radians(np.arange(0.0, 180.0 + 1e-9, step))
    ph = np.radians(np.arange(0.0, 360.0, step))
    T, P = np.meshgrid(th, ph, indexing="ij")
    return np.stack([np.sin(T) * np.cos(P), np.sin(T) * np.sin(P), np.cos(T)], -1).reshape(-1, 3)


def _frequency(seed):
    return K0 * _rng(seed).uniform(0.8, 1.2)


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "tabulate":
        E = 18 * n * n
        L = torch.empty((2 * case["ny"] - 1, 2 * case["nx"] - 1, E, E), dtype=torch.complex128, device=DEV)
        return dict(case=case, k=_frequency(seed), zl=B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T), L=L, K=torch.empty_like(L))
    if kind == "macromodel":
        sides = _rng(seed).uniform(0.15, 0.45, case["types"]) * W.LAMBDA
        Z = torch.empty((case["types"], 36 * n * n, 36 * n * n), dtype=torch.complex128, device=DEV)
        return dict(case=case, sides=sides, zl=B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T), Z=Z)
    if kind == "far_field":
        # a mixed-precision handle, as the solve leaves it; the far field reads its lattice and the currents
        idx, sgn, nu = B.emsurf_setup_overlap(n, case["nx"], case["ny"])
        L, K = _tables(case["nx"], case["ny"], n, K0)
        Z = torch.zeros((1, 36 * n * n, 36 * n * n), dtype=torch.complex128, device=DEV)
        h = _handle(case, dict(L=L, K=K, Z=Z, tmap=np.zeros(case["nx"] * case["ny"], np.int32), idx=idx, sgn=sgn, nu=nu), B.MIXED, False)
        r = _directions(case["step"])
        return dict(case=case, h=h, Y=_random((case["rhs"], nu), seed), r=r, zl=B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T),
                    F=torch.empty((case["rhs"], len(r), 3), dtype=torch.complex128, device=DEV),
                    rcs=torch.empty((case["rhs"], len(r)), dtype=torch.float64, device=DEV))
    op = _operator(case, seed)
    if kind == "product":
        # one right-hand side: the handle of a mixed solve; several: a single-precision or double-precision handle
        if case["operator"] == "fp64":
            precision = B.FP64
        else:
            precision = B.MIXED if case["rhs"] == 1 else B.FP32
        h = _handle(case, op, precision, False)
        x = _random((case["rhs"], op["nu"]), seed)
        return dict(case=case, h=h, x=x, y=torch.empty_like(x), precision=PRECISION[case["operator"]])
    h = _handle(case, op, B.MIXED, True)
    if kind == "precond":
        x = _random((case["rhs"], op["nu"]), seed)
        return dict(case=case, h=h, x=x, y=torch.empty_like(x))
    V = torch.empty((case["rhs"], op["nu"]), dtype=torch.complex128, device=DEV)
    khat, ehat = _waves(case["rhs"], seed)
    B.emsurf_excitation(h, A, A, H, n, K0, khat, ehat, V, zlevels=B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T))
    return dict(case=case, h=h, x=V, y=torch.empty_like(V))


def _waves(rhs, seed):
    r = _rng(seed + 7)
    khat, ehat = [], []
    for q in range(rhs):
        t, p = r.uniform(0.0, np.pi / 3), (0.0, np.pi / 2)[q % 2]
        khat.append([-np.sin(t) * np.cos(p), -np.sin(t) * np.sin(p), -np.cos(t)])
        ehat.append([np.cos(t) * np.cos(p), np.cos(t) * np.sin(p), -np.sin(t)])
    return np.array(khat), np.array(ehat)


# ---------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    kind, n = case["kind"], case["n"]
    if kind == "product":
        B.emsurf_matvec(state["h"], state["x"], state["y"], state["precision"])
        return state["y"] if case["operator"] == "fp64" else state["y"].to(torch.complex64)
    if kind == "precond":
        B.emsurf_precond_apply(state["h"], state["x"], state["y"])
        return state["y"].to(torch.complex64)
    if kind == "solve":
        # to 1e-6: six digits
        B.emsurf_solve(state["h"], state["x"], state["y"], rtol=1e-6, restart=30, max_iters=20000, max_refine=20)
        return state["y"].to(torch.complex64)
    if kind == "tabulate":
        B.emsurf_tabulate_offsets(A, A, H, n, case["nx"], case["ny"], state["k"], state["L"], state["K"], zlevels=state["zl"])
        return {"L": state["L"], "K": state["K"]}
    if kind == "macromodel":
        B.emsurf_macromodel_slab_patch(A, A, H, n, state["zl"], state["sides"], 4, W.RING_LAYERS, W.EPS_SLAB, K0, state["Z"])
        return state["Z"]
    B.emsurf_far_field(state["h"], A, A, H, n, K0, state["Y"], state["r"], state["F"], state["rcs"], zlevels=state["zl"])
    return {"F": state["F"].to(torch.complex64), "rcs": state["rcs"].to(torch.float32)}


# ---------------------------------------------------------------- what a pass cannot do without
def _smooth(m):
    while True:
        t = m
        for p in (2, 3, 5):
            while t % p == 0:
                t //= p
        if t == 1:
            return m
        m += 1


def _product_work(case, R, real_bytes):
    """Spectrum blocks of one bin per (k, -k) pair (per mirror orbit), macromodels, vectors."""
    K = 36 * case["n"] ** 2
    E, M = K // 2, case["nx"] * case["ny"]
    px, py = _smooth(2 * case["nx"] - 1), _smooth(2 * case["ny"] - 1)
    if case.get("mirrors"):
        hx, hy = px // 2 + 1, py // 2 + 1
        bins = hx * (hx + 1) // 2 if case["nx"] == case["ny"] else hx * hy
    else:
        bins = (px * py + 1) // 2
    nu = M * K * 0.65          # unique unknowns per local one, about
    types = min(case["types"], M)
    return (bins * 2 * E * E * 2 * real_bytes + types * K * K * 2 * real_bytes + 2 * nu * R * 16,
            R * (px * py * 4.0 * E * E * 8 + M * 8.0 * K * K))


def _precond_rows(case):
    """Entries of the owned rows of the subdomain inverses."""
    S, own, _, _ = _subdomains(case)
    return sum(len(s) * o for s, o in zip(S, own)), sum(own)


def work(case):
    kind = case["kind"]
    if kind == "product":
        b, f = _product_work(case, case["rhs"], 4 if case["operator"] == "fp32" else 8)
    elif kind == "precond":
        rows, nu = _precond_rows(case)
        b, f = rows * (8 if case["tc"] else 4) + 2 * 16 * nu * case["rhs"], 8.0 * rows * case["rhs"]
    elif kind == "solve":
        # 100 iterations, the headline solve's count: one product and one preconditioner apply each
        b, f = _product_work(case, case["rhs"], 4)
        rows, nu = _precond_rows(case)
        b, f = 100 * (b + rows * 4 + 2 * 16 * nu * case["rhs"]), 100 * (f + 8.0 * rows * case["rhs"])
    elif kind == "tabulate":
        E, T = 18 * case["n"] ** 2, 12 * case["n"] ** 2
        nof = (2 * case["nx"] - 1) * (2 * case["ny"] - 1)
        # both tables written; 49 point pairs of about 60 operations for each triangle pair of half of the offsets
        b, f = 2 * 16.0 * nof * E * E, (nof // 2 + 1) * T * T * 49 * 60.0
    elif kind == "macromodel":
        n, T = case["n"], case["types"]
        K = 36 * n * n
        Ni, Tr = 350, 12 * n * n // 2 + 130        # interior unknowns, triangles of one region
        b = 16.0 * T * K * K
        f = T * (8.0 * Ni * (K * K + K * Ni + Ni * Ni / 3) + 2.0 * Tr * Tr * (49 * 60 + 7 * 300))
    else:
        K, M, D, R = 36 * case["n"] ** 2, case["nx"] * case["ny"], len(_directions(case["step"])), case["rhs"]
        b, f = 16.0 * M * K * 0.65 * R + D * R * (3 * 16 + 8) + D * 24, 8.0 * D * R * (M * K + 3 * K)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- 64-bit values
def exact(case, seed):
    kind = case["kind"]
    if kind == "product":
        return _exact_product(case, seed)
    if kind == "precond":
        return _exact_precond(case, seed)
    if kind == "tabulate":
        return _exact_tables(case, seed)
    if kind == "far_field":
        return _exact_far_field(case, seed)
    # solve: hundreds of 64-bit products or a dense LU of up to 1e5 unknowns; macromodels: a composite
    # method-of-moments system of about 1500 unknowns for each of up to 32 types.  Minutes, both.
    return None


def _t(a, dtype=None):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV, dtype=dtype)


def _exact_product(case, seed):
    nx, ny, R = case["nx"], case["ny"], case["rhs"]
    K = 36 * case["n"] ** 2
    E, M = K // 2, nx * ny
    op = _operator(case, seed)
    x = _random((R, op["nu"]), seed)
    idx, sgn = _t(op["idx"], torch.int64), _t(op["sgn"], torch.float64)
    x1 = (x[:, idx] * sgn).reshape(R, M, K)
    py, px = 2 * ny, 2 * nx
    g = torch.zeros((py, px, K, R), dtype=torch.complex128, device=DEV)
    g[:ny, :nx] = x1.reshape(R, ny, nx, K).permute(1, 2, 3, 0)
    g = torch.fft.fft2(g, dim=(0, 1)).reshape(py * px, K, R)
    dy = torch.arange(-(ny - 1), ny, device=DEV) % py
    dx = torch.arange(-(nx - 1), nx, device=DEV) % px
    out = torch.zeros_like(g)
    for name, pairs in (("L", ((0, 0, COEF[0]), (1, 1, COEF[3]))), ("K", ((0, 1, COEF[1]), (1, 0, COEF[2])))):
        S = torch.zeros((py, px, E, E), dtype=torch.complex128, device=DEV)
        S[dy[:, None], dx[None, :]] = op.pop(name)
        S = torch.fft.fftn(S, dim=(0, 1)).reshape(py * px, E, E)
        for o, i, c in pairs:
            out[:, o * E:(o + 1) * E] += c * (S @ g[:, i * E:(i + 1) * E])
        del S
    y1 = torch.fft.ifft2(out.reshape(py, px, K, R), dim=(0, 1))[:ny, :nx].permute(3, 0, 1, 2).reshape(R, M, K).clone()
    tmap = _t(op["tmap"], torch.int64)
    for t in range(case["types"]):
        m = torch.nonzero(tmap == t).flatten()
        if len(m):
            y1[:, m] += x1[:, m] @ op["Z"][t].T
    y = torch.zeros_like(x)
    return y.index_add_(1, idx, y1.reshape(R, M * K) * sgn)


def _subdomains(case):
    """Unknowns of each cell's subdomain (the owned ones first), the counts owned, and the setup they come from."""
    nx, ny, n = case["nx"], case["ny"], case["n"]
    K, delta = 36 * n * n, A / n
    idx, sgn, nu = B.emsurf_setup_overlap(n, nx, ny)
    xy = B.emsurf_setup_unknown_xy(A, A, H, n, nx, ny, idx, nu)
    owner = np.full(nu, nx * ny)
    np.minimum.at(owner, idx, np.arange(len(idx)) // K)
    cells = idx.reshape(ny, nx, K)
    S, own = [], []
    for m in range(nx * ny):
        iy, ix = divmod(m, nx)
        u = np.unique(cells[max(0, iy - 1):iy + 2, max(0, ix - 1):ix + 2])
        near = (np.abs(xy[u, 0] - ix * A) <= 0.5 * A + delta + 1e-12) & (np.abs(xy[u, 1] - iy * A) <= 0.5 * A + delta + 1e-12)
        u = u[near]
        u = np.concatenate([u[owner[u] == m], u[owner[u] != m]])
        S.append(u)
        own.append(int((owner[u] == m).sum()))
    return S, own, idx, sgn


def _exact_precond(case, seed):
    nx, ny = case["nx"], case["ny"]
    K = 36 * case["n"] ** 2
    op = _operator(case, seed)
    S, own, idx, sgn = _subdomains(case)
    # copies of each unique unknown (at most 4), sign 0 where there are fewer
    order = np.argsort(idx, kind="stable")
    rank = np.arange(len(idx)) - np.searchsorted(idx[order], idx[order])
    copy, sign = np.zeros((op["nu"], 4), np.int64), np.zeros((op["nu"], 4))
    copy[idx[order], rank], sign[idx[order], rank] = order, sgn[order]
    copy, sign = _t(copy), _t(sign)
    # blocks B(d) for |dx|, |dy| <= 2 (subdomains reach the 3 x 3 neighbours)
    blocks = torch.zeros((5, 5, K, K), dtype=torch.complex128, device=DEV)
    for dy in range(-min(2, ny - 1), min(2, ny - 1) + 1):
        for dx in range(-min(2, nx - 1), min(2, nx - 1) + 1):
            L, Kk = op["L"][dy + ny - 1, dx + nx - 1], op["K"][dy + ny - 1, dx + nx - 1]
            blocks[dy + 2, dx + 2] = torch.cat([torch.cat([COEF[0] * L, COEF[1] * Kk], 1), torch.cat([COEF[2] * Kk, COEF[3] * L], 1)], 0)
    tmap = _t(op["tmap"], torch.int64)
    r = _random((case["rhs"], op["nu"]), seed)
    y = torch.zeros_like(r)
    for s, o in zip(S, own):
        u = _t(s, torch.int64)
        c, k, sg = copy[u] // K, copy[u] % K, sign[u]
        Am = torch.zeros((len(s), len(s)), dtype=torch.complex128, device=DEV)
        for p in range(4):
            for q in range(4):
                cp, cq, kp, kq = c[:, p, None], c[None, :, q], k[:, p, None], k[None, :, q]
                w = sg[:, p, None] * sg[None, :, q]
                dx, dy = (cp % nx - cq % nx).clamp(-2, 2) + 2, (cp // nx - cq // nx).clamp(-2, 2) + 2
                v = blocks[dy, dx, kp, kq] + torch.where(cp == cq, op["Z"][tmap[cp], kp, kq], torch.zeros((), dtype=torch.complex128, device=DEV))
                Am += w * v
        y[:, u[:o]] = torch.linalg.solve(Am, r[:, u].T)[:o].T
    return y


def _radon7():
    s = math.sqrt(15.0)
    a1, b1, a2, b2 = (6 - s) / 21, (9 + 2 * s) / 21, (6 + s) / 21, (9 - 2 * s) / 21
    bary = np.array([[1 / 3] * 3, [b1, a1, a1], [a1, b1, a1], [a1, a1, b1], [b2, a2, a2], [a2, b2, a2], [a2, a2, b2]])
    return bary, np.array([9 / 40] + [(155 - s) / 1200] * 3 + [(155 + s) / 1200] * 3)


def _box(n, zl):
    """Triangles [T, 3, 3], their areas, quadrature points [T, 7, 3] and weights [T, 7], and the
    matrix [E, 3 T] from slot integrals to RWG ones."""
    m = B.emsurf_setup_box_mesh(A, A, H, n, zlevels=zl)
    tri = m["verts"][m["tris"]]
    area = 0.5 * np.linalg.norm(np.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]), axis=1)
    bary, w = _radon7()
    P = np.zeros((len(m["tplus"]), 3 * len(tri)))
    for t in range(len(tri)):
        for i in range(3):
            e = m["slot_rwg"][t, i]
            if e >= 0:
                P[e, 3 * t + i] += m["slot_sgn"][t, i] * np.linalg.norm(tri[t, (i + 1) % 3] - tri[t, (i + 2) % 3]) / (2 * area[t])
    return _t(tri), _t(area), _t(np.einsum("qv,tvx->tqx", bary, tri)), _t(w[None] * area[:, None]), _t(P, torch.complex128)


def _potentials(r, tri):
    """Integrals of 1/R, (rho' - rho)/R and grad(1/R) over flat triangles in closed form (Wilton et
    al. 1984, Graglia 1993), and the projection rho of r; r [..., 3] against tri [S, 3, 3]."""
    v = [tri[:, i] for i in range(3)]
    n = torch.linalg.cross(v[1] - v[0], v[2] - v[0])
    n = n / n.norm(dim=-1, keepdim=True)
    scale = torch.maximum((v[1] - v[0]).norm(dim=-1), (v[2] - v[0]).norm(dim=-1))
    d = ((r - v[0]) * n).sum(-1)
    d = torch.where(d.abs() <= 1e-9 * scale, torch.zeros_like(d), d)
    rho = r - d[..., None] * n
    I0, I1, f_u, angle = 0.0, 0.0, 0.0, 0.0
    for i in range(3):
        a, b = v[i], v[(i + 1) % 3]
        lh = (b - a) / (b - a).norm(dim=-1, keepdim=True)
        u = torch.linalg.cross(lh, n)
        lp, lm, t = ((b - rho) * lh).sum(-1), ((a - rho) * lh).sum(-1), ((a - rho) * u).sum(-1)
        R0 = t * t + d * d
        Rp, Rm = (R0 + lp * lp).sqrt(), (R0 + lm * lm).sqrt()
        f = torch.where(lm >= 0, ((Rp + lp) / (Rm + lm)).log(), torch.where(lp <= 0, ((Rm - lm) / (Rp - lp)).log(), ((Rp + lp) * (Rm - lm) / R0).log()))
        beta = torch.atan2(t * lp, R0 + d.abs() * Rp) - torch.atan2(t * lm, R0 + d.abs() * Rm)
        I0 = I0 + t * f - d.abs() * beta
        I1 = I1 + 0.5 * u * (R0 * f + lp * Rp - lm * Rm)[..., None]
        f_u = f_u + u * f[..., None]
        angle = angle + beta
    return I0, I1, -n * (torch.sign(d) * angle)[..., None] - f_u, rho


def _exact_tables(case, seed):
    """The reciprocal part of the Galerkin tables by plain quadrature (closed-form 1/R parts for touching boxes)."""
    nx, ny, n = case["nx"], case["ny"], case["n"]
    k = _frequency(seed)
    tri, area, pts, wts, P = _box(n, B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T))
    T, E = len(tri), P.shape[0]
    b = pts[:, :, None, :] - tri[:, None, :, :]                       # [T, 7, 3 slots, 3]
    one = torch.ones_like(b[..., :1])
    x_of = lambda a, r: torch.linalg.cross(a, r[:, :, None, :].expand_as(a))  # noqa: E731
    offs = [(dy, dx) for dy in range(-(ny - 1), ny) for dx in range(-(nx - 1), nx)]
    out = [torch.empty((len(offs), E, E), dtype=torch.complex128, device=DEV) for _ in range(2)]
    chunk = max(1, int(2e7 // (49 * T * T)))
    for touching in (True, False):
        todo = [i for i, (dy, dx) in enumerate(offs) if (abs(dy) <= 1 and abs(dx) <= 1) == touching]
        for c0 in range(0, len(todo), 1 if touching else chunk):
            at = todo[c0:c0 + (1 if touching else chunk)]
            sh = _t(np.array([[offs[i][1] * A, offs[i][0] * A, 0.0] for i in at]))
            diff = (pts[None] + sh[:, None, None])[:, :, :, None, None, :] - pts[None, None, None]
            R = diff.norm(dim=-1)                                      # [C, t, q, s, p]
            del diff
            if touching:
                size = torch.maximum((tri[:, 1] - tri[:, 0]).norm(dim=-1), (tri[:, 2] - tri[:, 0]).norm(dim=-1))
                zero = R <= 1e-9 * size[None, None, None, :, None]
                Rs = torch.where(zero, 1.0, R)
                # e^{-jkR} - 1 = -2 sin^2(kR/2) - j sin kR; 1 - (1 + jkR) e^{-jkR} by its series for small kR
                e1 = torch.complex(-2 * torch.sin(0.5 * k * Rs) ** 2, -torch.sin(k * Rs))
                G = torch.where(zero, torch.full_like(e1, -1j * k / (4 * np.pi)), e1 / (4 * np.pi * Rs))
                h = -e1 - 1j * k * Rs * (1 + e1)
                z, term, ser = -1j * k * Rs, torch.ones_like(e1), torch.zeros_like(e1)
                for m in range(1, 18):
                    term = term * z / m
                    ser = ser + (m - 1) * term
                h = torch.where(k * Rs < 0.5, ser, h)
                g = torch.where(zero, torch.zeros_like(h), h / (4 * np.pi * Rs ** 3))
            else:
                e = torch.exp(-1j * k * R)
                G, g = e / (4 * np.pi * R), -(1 + 1j * k * R) * e / (4 * np.pi * R ** 3)
            ww = wts[:, :, None, None] * wts[None, None]
            G, g = (G * ww).reshape(len(at), T * 7, T, 7), (g * ww).reshape(len(at), T * 7, T, 7)
            # L: a . b - 4/k^2;  K: a . ((r - r') x b), r in the test box's frame shifted to the source's
            bL = torch.cat([b, one * (-4 / k ** 2)], -1).reshape(T, 7, 12).to(torch.complex128)
            aL = torch.cat([b, one], -1).to(torch.complex128)
            bK = torch.cat([b, x_of(b, pts)], -1).reshape(T, 7, 18).to(torch.complex128)   # b, b x r'
            sL = torch.einsum("cusp,spx->cusx", G, bL).reshape(len(at), T, 7, T, 3, 4)
            SL = torch.einsum("ctqsjx,tqix->ctisj", sL, aL)
            sK = torch.einsum("cusp,spx->cusx", g, bK).reshape(len(at), T, 7, T, 3, 6)
            SK = torch.empty_like(SL)
            for c in range(len(at)):
                rt = pts + sh[c]
                aK = torch.cat([x_of(b, rt), b], -1).to(torch.complex128)                    # a x r, a
                SK[c] = torch.einsum("tqsjx,tqix->tisj", sK[c], aK)
                if touching:
                    I0, I1, Ig, rho = _potentials(rt[:, :, None, :], tri)                    # [t, q, s]
                    wq = wts / (4 * np.pi)
                    vec = I1[:, :, :, None] + (rho[:, :, :, None] - tri[None, None]) * I0[..., None, None]
                    SL[c] += torch.einsum("tqix,tqsjx,tq->tisj", b, vec, wq) - (4 / k ** 2) * torch.einsum("tqs,tq->ts", I0, wq)[:, None, :, None]
                    cr = torch.linalg.cross(Ig[:, :, :, None].expand(-1, -1, -1, 3, -1), rt[:, :, None, None] - tri[None, None])
                    SK[c] += torch.einsum("tqix,tqsjx,tq->tisj", b, cr, wq)
            for o, S in zip(out, (SL, SK)):
                o[at] = P @ S.reshape(len(at), 3 * T, 3 * T) @ P.T
    L, K = (0.5 * (o + o.flip(0).transpose(1, 2)) for o in out)
    shape = (2 * ny - 1, 2 * nx - 1, E, E)
    return {"L": L.reshape(shape), "K": K.reshape(shape)}


def _exact_far_field(case, seed):
    nx, ny, n, R = case["nx"], case["ny"], case["n"], case["rhs"]
    K = 36 * n * n
    E, M = K // 2, nx * ny
    idx, sgn, nu = B.emsurf_setup_overlap(n, nx, ny)
    Y = _random((R, nu), seed)
    X = (Y[:, _t(idx, torch.int64)] * _t(sgn, torch.float64)).reshape(R, M, K).permute(1, 0, 2).reshape(M, R * K)
    r = _t(_directions(case["step"]))
    tri, area, pts, wts, P = _box(n, B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T))
    T = len(tri)
    a = (pts[:, :, None, :] - tri[:, None, :, :]) * wts[:, :, None, None]
    c = _t(np.stack([np.tile(np.arange(nx), ny) * A, np.repeat(np.arange(ny), nx) * A], -1))
    F = torch.empty((R, len(r), 3), dtype=torch.complex128, device=DEV)
    for d0 in range(0, len(r), 2048):
        rd = r[d0:d0 + 2048]
        D = len(rd)
        S = (torch.exp(1j * K0 * (rd[:, :2] @ c.T)) @ X).reshape(D, R, K)
        ph = torch.exp(1j * K0 * torch.einsum("dx,tqx->dtq", rd, pts))
        rad = torch.einsum("dtq,tqix->dxti", ph, a.to(torch.complex128)).reshape(D, 3, 3 * T) @ P.T       # [D, 3, E]
        N, Lm = (torch.einsum("dre,dxe->rdx", S[:, :, s], rad) for s in (slice(0, E), slice(E, K)))
        rc = rd.to(torch.complex128)[None].expand(R, -1, -1)
        Np = N - (N * rc).sum(-1, keepdim=True) * rc
        F[:, d0:d0 + D] = -(1j * K0 / (4 * np.pi)) * (Np - torch.linalg.cross(rc, Lm))
    return {"F": F, "rcs": 4 * np.pi * (F.abs() ** 2).sum(-1)}
