"""Which form of the SAP preconditioner runs, by the launches of one call, and its
result against the oracle: the application split over two cooperative launches
(260 sweeps) in FP32 and FP64, FP64 over several cycles with several right-hand
sides and the clover term, one launch per sweep when the domains exceed what the
device holds at a time, the domains that run the stand-alone sweep, and domains one
site thick in the application kernel.

A call launches one conversion in, the application and one conversion out.
Tolerances in the 2-norm as in the parity tests (FP64 1e-11, FP32 4 u). The 260
sweeps in FP32 have converged to FP32's floor, so there the relative residual is
what is checked: 2.5 u, as derived in test_gpu_sap_iterate.py."""

import numpy as np
import pytest

import fieldgen as fg
import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [
    # dims, block, cycles, MR steps, nrhs, c_sw, precision, launches of the application
    ((4, 4, 4, 4), (2, 2, 2, 2), 130, 2, 1, 0.0, "f32", 2),
    ((8, 8, 8, 8), (4, 4, 4, 4), 130, 1, 1, 0.0, "f64", 2),
    ((8, 8, 8, 8), (4, 4, 4, 4), 4, 3, 3, 1.0, "f64", 1),
    ((8, 8, 8, 8), (4, 4, 4, 4), 4, 3, 3, 1.0, "f32", 1),
    ((16, 16, 16, 16), (4, 4, 4, 4), 3, 2, 2, 0.0, "f64", 6),    # 256 CTAs of one an SM
    ((8, 8, 8, 8), (4, 4, 4, 2), 3, 2, 1, 1.0, "f64", 6),        # the stand-alone sweep
    # one site in a direction: both its faces there are the same site
    ((4, 8, 8, 8), (1, 4, 4, 4), 3, 2, 2, 0.0, "f32", 1),
    ((8, 4, 8, 8), (4, 1, 4, 4), 3, 2, 1, 1.0, "f32", 1),
    ((8, 8, 4, 8), (4, 4, 1, 4), 3, 2, 1, 0.0, "f32", 1),
    ((8, 8, 8, 2), (4, 4, 4, 1), 3, 2, 1, 1.0, "f32", 1),
]


@pytest.mark.parametrize("dims,block,cycles,mr,nrhs,csw,prec,launches", CASES)
def test_form_and_result(dims, block, cycles, mr, nrhs, csw, prec, launches):
    import paper_1204_5463_gb300 as dw

    m0 = 0.25
    U = fg.gauge_field(dims, 0.4, seed=3)
    v = np.ascontiguousarray(fg.gaussian_source(dims, 4, nrhs=nrhs)).reshape(nrhs, -1, 4, 3)
    if prec == "f32":
        U, v = (a.astype(np.complex64).astype(np.complex128) for a in (U, v))
    kw = dict(A=oracle.clover(U, dims, csw)) if csw else {}
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.float64).reshape(-1).copy()).cuda()  # noqa: E731
    ctx = dw.dw_create(dims, block, m0, torch.cuda.current_stream().cuda_stream)
    try:
        dw.dw_set_gauge(ctx, dev(U), True)
        if csw:
            dw.dw_set_clover(ctx, csw)
        z, vd = torch.empty(v.size * 2, dtype=torch.float64, device="cuda"), dev(v)
        for _ in range(2):  # the first call also packs the links
            before = dw.dw_kernel_launches()
            dw.sap_precondition(ctx, vd, z, cycles, mr, dw.PREC[prec], nrhs)
        assert dw.dw_kernel_launches() - before == launches + 2
        got = z.cpu().numpy().view(np.complex128).reshape(v.shape)
    finally:
        dw.dw_destroy(ctx)
    for r in range(nrhs):
        if prec == "f32" and cycles > 100:
            assert np.linalg.norm(v[r] - oracle.dw(U, got[r], dims, m0)) <= 2.5 * 2.0 ** -24 * np.linalg.norm(v[r])
        else:
            ref = oracle.sap(U, v[r], dims, block, m0, cycles, mr, **kw)
            tol = 1e-11 if prec == "f64" else 4 * 2.0 ** -24
            assert np.linalg.norm(got[r] - ref) <= tol * np.linalg.norm(ref)
