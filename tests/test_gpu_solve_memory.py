"""Device memory of a solve: with device buffers a context holds one FP64 field per
right-hand side less than with host buffers, whose copies are staged."""

import ctypes

import numpy as np
import pytest

import fieldgen as fg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _used():
    """Bytes in use in the device's default memory pool, from which the library allocates."""
    cu, pool, n = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    assert cu.cuMemPoolGetAttribute(pool, 7, ctypes.byref(n)) == 0  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT
    return n.value


@pytest.mark.parametrize("block", [(4, 4, 4, 4), (8, 4, 4, 4)])  # the second runs the stand-alone sweep
def test_device_buffers_need_no_staging_copy(block):
    import paper_1204_5463_gb300 as dw

    dims, nrhs = (16, 8, 8, 8), 2
    V = int(np.prod(dims))
    U = torch.from_numpy(fg.gauge_field(dims, 0.4, seed=3).view(np.float64).reshape(-1).copy())
    b = torch.from_numpy(np.ascontiguousarray(fg.gaussian_source(dims, 4, nrhs=nrhs)).view(np.float64).reshape(-1).copy())
    held = {}
    for host in (True, False):
        bd, x = (b, torch.zeros_like(b)) if host else (b.cuda(), torch.zeros_like(b).cuda())
        Ud = U.cuda()
        torch.cuda.synchronize()
        before = _used()
        ctx = dw.dw_create(dims, block, 0.25, torch.cuda.current_stream().cuda_stream)
        try:
            dw.dw_set_gauge(ctx, Ud, True)
            P = dw.dw_default_params(nrhs=nrhs, tol=1e-8, host_buffers=int(host))
            dw.fgmresdr_solve(ctx, bd, x, P)
            held[host] = _used() - before
        finally:
            dw.dw_destroy(ctx)
    assert held[False] + 192 * V * nrhs <= held[True]
