"""SAP after the gauge field of a context was replaced, and in a further
precision: the first sweep reads the domains' packed links ahead of the kernel in
front of it, so the links have to be packed before that kernel is launched.
Against the oracle, on a lattice whose domains run sweep by sweep and with
domains of more than 256 sites. Tolerances as in the parity tests (2-norm; 4 u of
FP32, 2 u of FP16, 1e-11 in FP64); with the former field's links the results
differ by tens of per cent."""

import numpy as np
import pytest

import fieldgen as fg
import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"f64": 1e-11, "f32": 4 * 2.0 ** -24, "f16": 2 * 2.0 ** -11}


@pytest.mark.parametrize("dims,block,precs", [
    ((16, 16, 16, 32), (2, 2, 2, 2), ("f32", "f16")),  # 4096 domains a colour
    ((16, 8, 16, 8), (8, 4, 8, 2), ("f32", "f16")),    # 512 sites a domain
    ((8, 8, 8, 8), (4, 4, 4, 2), ("f64",)),
])
def test_replaced_gauge_field(dims, block, precs):
    import paper_1204_5463_gb300 as dw

    fields = [fg.gauge_field(dims, 0.4, seed=s) for s in (3, 4)]
    v = fg.gaussian_source(dims, 4)
    refs = [oracle.sap(U, v, dims, block, -0.2, 2, 3) for U in fields]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.float64).reshape(-1).copy()).cuda()  # noqa: E731
    vd, z = dev(v), torch.empty(v.size * 2, dtype=torch.float64, device="cuda")
    links = [dev(U) for U in fields]
    ctx = dw.dw_create(dims, block, -0.2, torch.cuda.current_stream().cuda_stream)
    try:
        for n in (0, 1, 0):
            dw.dw_set_gauge(ctx, links[n], True)
            for p in precs:
                dw.sap_precondition(ctx, vd, z, 2, 3, dw.PREC[p], 1)
                got = z.cpu().numpy().view(np.complex128).reshape(v.shape)
                assert np.linalg.norm(got - refs[n]) <= TOL[p] * np.linalg.norm(refs[n])
    finally:
        dw.dw_destroy(ctx)
