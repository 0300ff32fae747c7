"""GPU parity of the SAP preconditioner that carries the domains' residuals
(one cooperative launch, or one launch per sweep when the domains exceed what
the device holds at a time) with the oracle's Algorithm 2, at the shapes where
its index arithmetic can go wrong: one domain pair per direction, odd extents,
partly filled warps, one cycle, one MR step, and more domains than fit.

Tolerances as in the parity tests (2-norm; 4 u of FP32, 2 u of FP16 and BF16,
1e-11 in FP64): the carried residual rounds like the recomputed one, once per
hop and update."""

import numpy as np
import pytest

import fieldgen as fg
import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"f64": 1e-11, "f32": 4 * 2.0 ** -24, "f16": 2 * 2.0 ** -11, "bf16": 2 * 2.0 ** -8}
CASES = [
    # dims, block, cycles, MR steps, nrhs, c_sw
    ((6, 10, 14, 4), (3, 5, 7, 2), 3, 2, 1, 0.0),    # 210 sites: the last warp partly idle
    ((6, 6, 6, 6), (3, 3, 3, 3), 2, 1, 2, 1.0),      # 81 sites, one MR step, the clover term
    ((8, 8, 8, 16), (4, 4, 4, 4), 1, 4, 3, 0.0),     # a single cycle: nothing is kept between visits
    ((16, 8, 8, 4), (8, 4, 4, 2), 2, 3, 1, 1.0),
    ((4, 8, 8, 12), (2, 4, 4, 6), 3, 3, 2, 0.0),
    ((16, 16, 16, 32), (2, 2, 2, 2), 2, 3, 1, 0.0),  # 4096 domains a colour: sweep by sweep
]


# 260 sweeps: more than one cooperative launch takes
LONG = ((4, 4, 4, 4), (2, 2, 2, 2), 130, 1, 1, 0.0)


@pytest.mark.parametrize("dims,block,cycles,mr,nrhs,csw,prec",
                         [c + (p,) for c in CASES for p in TOL] + [LONG + ("f64",)])
def test_sap_matches_oracle(dims, block, cycles, mr, nrhs, csw, prec):
    import paper_1204_5463_gb300 as dw

    U = fg.gauge_field(dims, 0.4, seed=3)
    v = np.ascontiguousarray(fg.gaussian_source(dims, 4, nrhs=nrhs))
    kw = dict(A=oracle.clover(U, dims, csw)) if csw else {}
    dev = lambda a: torch.from_numpy(a.view(np.float64).reshape(-1).copy()).cuda()  # noqa: E731
    ctx = dw.dw_create(dims, block, -0.2, torch.cuda.current_stream().cuda_stream)
    try:
        dw.dw_set_gauge(ctx, dev(U), True)
        if csw:
            dw.dw_set_clover(ctx, csw)
        z = torch.empty(v.size * 2, dtype=torch.float64, device="cuda")
        vd = dev(v)
        for _ in range(2):  # the second application starts from counters and scratch the first one left
            dw.sap_precondition(ctx, vd, z, cycles, mr, dw.PREC[prec], nrhs)
        got = z.cpu().numpy().view(np.complex128).reshape(v.shape)
    finally:
        dw.dw_destroy(ctx)
    for r in range(nrhs):
        ref = oracle.sap(U, v[r], dims, block, -0.2, cycles, mr, **kw)
        assert np.linalg.norm(got[r] - ref) <= TOL[prec] * np.linalg.norm(ref)
