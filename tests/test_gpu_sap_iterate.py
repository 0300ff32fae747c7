"""What a SAP application keeps between its sweeps: the iterate x in the storage
precision, and nothing else, the residual v - D x being formed anew from it.

FP32 as a solver (40 cycles): its relative residual reaches the floor that the
rounding of x and of one residual set. With u = 2^-24, a rounding of x (0.4 u |x|)
enters through D (norm sqrt((4 + m0)^2 + 4) on a random vector) and |x| is about a
quarter of |v|: 0.5 u, and the eight hops' rounding about as much; 2.5 u leaves
room for both. A residual that is carried along never sees the rounding of x and
collects it from all cycles.

16-bit: one more cycle continues from what the cycle before it returned. On the
domains swept first the oracle's cycle from there, rounded to the format, is the
kernel's up to values whose FP32 error (2e-7) crosses a rounding boundary: one in
a thousand, by one unit in the last place, so 0.03 u in the 2-norm; 0.1 u is
allowed. An iterate kept in FP32 is off by the format's rounding, about 0.5 u."""

import numpy as np
import pytest

import fieldgen as fg
import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DIMS, BLOCK = (8, 8, 8, 16), (4, 4, 4, 4)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.complex128).view(np.float64).reshape(-1).copy()).cuda()


def _sap(m0, U, v, prec, cycles, mr):
    import paper_1204_5463_gb300 as dw

    ctx = dw.dw_create(DIMS, BLOCK, m0, torch.cuda.current_stream().cuda_stream)
    try:
        dw.dw_set_gauge(ctx, _dev(U), True)
        z = torch.empty(v.size * 2, dtype=torch.float64, device="cuda")
        out = []
        for n in cycles:
            dw.sap_precondition(ctx, _dev(v), z, n, mr, dw.PREC[prec], 1)
            out.append(z.cpu().numpy().view(np.complex128).reshape(v.shape).copy())
        return out
    finally:
        dw.dw_destroy(ctx)


def test_f32_solver_floor():
    m0 = 0.3 - 0.6135  # 0.3 right of the left edge of the spectrum at this disorder
    U = fg.gauge_field(DIMS, 0.5, seed=3).astype(np.complex64).astype(np.complex128)
    v = fg.gaussian_source(DIMS, 4).astype(np.complex64).astype(np.complex128)
    (z,) = _sap(m0, U, v, "f32", [40], 4)
    assert np.linalg.norm(v - oracle.dw(U, z, DIMS, m0)) <= 2.5 * 2.0 ** -24 * np.linalg.norm(v)


def _parts(a, to):
    """Real and imaginary parts through the 16-bit type."""
    t = torch.from_numpy(np.ascontiguousarray(a).view(a.real.dtype)).float().to(to).float()
    return t.numpy().view(np.complex64).reshape(a.shape)


def _rounded(x, to):
    """A spinor field through the storage format: 16-bit parts relative to each site's largest."""
    x = np.ascontiguousarray(x, np.complex64)
    flat = x.reshape(-1, 12)
    sc = np.maximum(np.abs(flat.real), np.abs(flat.imag)).max(1, keepdims=True).astype(np.float32)
    sc = np.where(sc > 0, sc, np.float32(1))
    inv = np.float32(1) / sc
    h = _parts((flat.real * inv + 1j * (flat.imag * inv)).astype(np.complex64), to)
    return (sc * h.real + 1j * (sc * h.imag)).astype(np.complex128).reshape(x.shape)


@pytest.mark.parametrize("prec,to,u", [("f16", torch.float16, 2.0 ** -11), ("bf16", torch.bfloat16, 2.0 ** -8)])
def test_16_bit_cycles_continue_from_the_stored_iterate(prec, to, u):
    m0, mr = -0.25, 4
    U = _parts(fg.gauge_field(DIMS, 0.4, seed=3), to).astype(np.complex128)
    v = _rounded(fg.gaussian_source(DIMS, 4), to)
    z1, z2, z3 = _sap(m0, U, v, prec, [1, 2, 3], mr)
    first = oracle.site_colours(DIMS, BLOCK).reshape(-1) == 0
    for before, after in ((z1, z2), (z2, z3)):
        ref = _rounded(oracle.sap(U, v, DIMS, BLOCK, m0, 1, mr, x0=before), to)
        d = (after - ref).reshape(first.size, -1)[first]
        assert np.linalg.norm(d) <= 0.1 * u * np.linalg.norm(ref.reshape(first.size, -1)[first])
