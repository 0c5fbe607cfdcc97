"""emsurf_launch_count against the kernels that a product issues: the product is
captured and the kernel nodes of the graph are counted.  Every variant: fused
transforms and passes, one and several rhs, FP64 digits in one and several
groups, tensor cores.
"""
import ctypes as C

import numpy as np
import pytest

from oracle import lattice
from oracle.mesh import box_mesh
from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H = W.PERIOD, W.BOX_H
COEF = (1j * W.K0, 1.0, -1.0, 1j * W.K0)


def kernels_of(call):
    """Kernel nodes of what call(stream) issues."""
    import torch
    rt = C.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, n, kind = C.c_void_p(), C.c_size_t(), C.c_int()
    assert rt.cudaStreamBeginCapture(C.c_void_p(st.cuda_stream), C.c_int(2)) == 0        # relaxed
    try:
        call(st.cuda_stream)
    finally:
        assert rt.cudaStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, C.byref(n)) == 0
    count = 0
    for q in nodes:
        assert rt.cudaGraphNodeGetType(C.c_void_p(q), C.byref(kind)) == 0
        count += kind.value == 0                                                         # a kernel node
    assert rt.cudaGraphDestroy(graph) == 0
    return count


@pytest.mark.parametrize("n,nx,ny,R,mx,tc,prec", [
    (2, 3, 2, 1, 1, False, "FP64"), (2, 3, 2, 7, 7, False, "FP64"), (1, 3, 2, 2, 2, False, "FP64"),
    (2, 3, 2, 1, 1, False, "FP32"), (2, 3, 2, 1, 3, False, "FP32"), (2, 3, 2, 9, 9, False, "FP32"),
    (2, 3, 2, 9, 9, True, "FP32"), (1, 3, 2, 5, 5, False, "FP32"), (1, 130, 2, 1, 1, False, "FP32"),
    (1, 130, 2, 2, 2, False, "FP64"),
])
def test_launches_are_counted(emsurf_lib, n, nx, ny, R, mx, tc, prec):
    import torch
    from paper_1911_04576_gb300 import binding as B
    box = box_mesh(A, A, H, n)
    E = box.n_rwg
    idx, sgn, nu = lattice.overlap_map(box, nx, ny, A, A)
    Lt, Kt = W.random_tables(nx, ny, E, 1)
    h = B.emsurf_create(nx, ny, E, nu, np.zeros(nx * ny, np.int32), W.random_macromodels(1, 2 * E, 2), Lt, Kt, COEF, idx,
                        sgn, precision=B.MIXED, max_rhs=mx, tensor_cores=tc)
    x = torch.from_numpy(W.random_vectors(R, nu, 3)).cuda()
    y = torch.empty_like(x)
    p = getattr(B, prec)
    B.emsurf_matvec(h, x, y, p)
    before = B.emsurf_launch_count(h)
    issued = kernels_of(lambda s: B.emsurf_matvec(h, x, y, p, stream=s))
    assert B.emsurf_launch_count(h) - before == issued
    h.close()
