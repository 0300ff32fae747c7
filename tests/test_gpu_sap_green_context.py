"""SAP and a solve on a stream of a green context that has some of the SMs only:
the domains that the whole device holds at a time need not fit there, so the
application takes one launch per sweep. Same results to the bit."""

import ctypes

import numpy as np
import pytest

import fieldgen as fg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _green_stream(sms):
    """A stream of a green context with about `sms` SMs, and what destroys both."""
    cu = ctypes.CDLL("libcuda.so.1")
    whole, part = ctypes.create_string_buffer(256), ctypes.create_string_buffer(256)  # CUdevResource: 144 bytes
    n, desc, green, stream = ctypes.c_uint(1), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    dev = torch.cuda.current_device()
    try:
        rc = [cu.cuDeviceGetDevResource(dev, whole, 1),
              cu.cuDevSmResourceSplitByCount(part, ctypes.byref(n), whole, None, 0, sms),
              cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1),
              cu.cuGreenCtxCreate(ctypes.byref(green), desc, dev, 1),
              cu.cuGreenCtxStreamCreate(ctypes.byref(stream), green, 1, 0)]
    except AttributeError:
        pytest.skip("no green contexts in this driver")
    if any(rc):
        pytest.skip(f"no green context: {rc}")

    def close():
        cu.cuStreamDestroy_v2(stream)
        cu.cuGreenCtxDestroy(green)

    return stream.value, close


def test_fewer_sms_than_the_domains_need():
    import paper_1204_5463_gb300 as dw

    dims, block = (16, 16, 16, 16), (4, 4, 4, 4)  # 128 domains a colour: 64 SMs of two
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.float64).reshape(-1).copy()).cuda()  # noqa: E731
    U, v = dev(fg.gauge_field(dims, 0.4, seed=3)), dev(fg.gaussian_source(dims, 4))
    torch.cuda.synchronize()
    stream, close = _green_stream(16)
    got, launches = [], []
    try:
        for st in (torch.cuda.current_stream().cuda_stream, stream):
            ctx = dw.dw_create(dims, block, 0.25, st)
            z, x = torch.empty_like(v), torch.empty_like(v)
            try:
                dw.dw_set_gauge(ctx, U, True)
                for _ in range(2):
                    before = dw.dw_kernel_launches()
                    dw.sap_precondition(ctx, v, z, 3, 4, dw.DW_F32, 1)
                launches.append(dw.dw_kernel_launches() - before)
                S = dw.fgmresdr_solve(ctx, v, x, dw.dw_default_params(tol=1e-10))
                assert S.converged
            finally:
                dw.dw_destroy(ctx)
            got.append(z)
    finally:
        close()
    assert launches == [1 + 2, 6 + 2]
    assert torch.equal(got[0], got[1])
