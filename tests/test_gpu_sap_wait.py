"""A wait of the SAP preconditioner that runs out: with a limit of zero the domains
that have an SM to themselves, two thousand MR steps ahead of those that share one,
find the previous sweep unfinished and give up. The call returns DW_ETIMEOUT with
the stream idle, and the next application or solve on the same context is not
touched by the counters and scratch that the one before it left."""

import numpy as np
import pytest

import fieldgen as fg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_give_up_and_recover():
    import paper_1204_5463_gb300 as dw

    dims, block = (16, 16, 16, 32), (4, 4, 4, 4)  # 256 domains a colour
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.float64).reshape(-1).copy()).cuda()  # noqa: E731
    U, v = dev(fg.gauge_field(dims, 0.4, seed=3)), dev(fg.gaussian_source(dims, 4))
    st = torch.cuda.current_stream()
    ctx = dw.dw_create(dims, block, 0.25, st.cuda_stream)
    try:
        dw.dw_set_gauge(ctx, U, True)
        z, ref, x, xref = (torch.empty_like(v) for _ in range(4))
        P = dw.dw_default_params(tol=1e-10)
        dw.sap_precondition(ctx, v, ref, 3, 4, dw.DW_F32, 1)
        dw.fgmresdr_solve(ctx, v, xref, P)
        for _ in range(2):
            dw.dw_debug_sap_wait(ctx, 0)
            with pytest.raises(dw.DwError) as e:
                dw.sap_precondition(ctx, v, z, 3, 2000, dw.DW_F32, 1)
            assert e.value.code == dw.DW_ETIMEOUT and st.query()
            with pytest.raises(dw.DwError) as e:
                dw.fgmresdr_solve(ctx, v, x, dw.dw_default_params(tol=1e-10, mr_steps=2000))
            assert e.value.code == dw.DW_ETIMEOUT and st.query()
            dw.dw_debug_sap_wait(ctx, -1)
            dw.sap_precondition(ctx, v, z, 3, 4, dw.DW_F32, 1)
            assert torch.equal(z, ref)
            dw.fgmresdr_solve(ctx, v, x, P)
            assert torch.equal(x, xref)
    finally:
        dw.dw_destroy(ctx)
