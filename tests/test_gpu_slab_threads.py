"""Cell libraries built by several host threads at once, as the server's
workers do: libraries whose panels take different amounts of shared memory
(30 to 336 interior unknowns) must not change each other's launch limits.  Each
thread's macromodels are bit for bit those of the same library built alone.
"""
import threading

import numpy as np
import pytest

from paper_1911_04576_gb300 import workloads as W

pytestmark = pytest.mark.gpu

A, H, K0 = W.PERIOD, W.BOX_H, W.K0


def test_threads_with_panels_of_different_size(emsurf_lib):
    import torch
    from paper_1911_04576_gb300 import binding as B
    n = 2
    z = B.emsurf_setup_slab_zlevels(H, n, W.SLAB_T)

    def build(patch_n, layers, stream):
        Z = torch.empty((1, 144, 144), dtype=torch.complex128, device="cuda")
        B.emsurf_macromodel_slab_patch(A, A, H, n, z, np.array([0.3 * W.LAMBDA]), patch_n, layers, W.EPS_SLAB, K0, Z,
                                       stream=stream.cuda_stream)
        return Z

    kinds = [(4, 3), (1, 1), (4, 2), (2, 1)]
    streams = [torch.cuda.Stream() for _ in kinds]
    alone = [build(*k, s) for k, s in zip(kinds, streams)]
    errors = []

    def work(i):
        try:
            for _ in range(60):
                Z = build(*kinds[i], streams[i])
                if not torch.equal(Z, alone[i]):
                    raise AssertionError("library %d differs" % i)
        except Exception as e:        # noqa: BLE001 (reported below)
            errors.append((i, e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(kinds))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
