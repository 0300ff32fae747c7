"""Rounding of the FP64 operator against extended precision (numpy's long double):
no larger than that of the plain form, hop after hop into one accumulator.

Random SU(3) links, Gaussian spinors, m0 = -0.6: in a simulation of the roundings
over 20000 sites the plain form is off by 8.74e-17 (2-norm, relative), separate FMA
chains whose results are joined by 8.41e-17, chains that run on from one hop into the
other by 9.14e-17. 40320 numbers give the norm to 0.5%; 8.8e-17 is allowed."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DIMS, M0 = (6, 10, 14, 2), -0.6


def _inputs():
    rng, V = np.random.default_rng(5), int(np.prod(DIMS))
    q, _ = np.linalg.qr(rng.standard_normal((V, 4, 3, 3)) + 1j * rng.standard_normal((V, 4, 3, 3)))
    U = q / np.linalg.det(q)[..., None, None] ** (1 / 3)
    return U, rng.standard_normal((V, 4, 3)) + 1j * rng.standard_normal((V, 4, 3))


def dw_long(U, psi):
    """D psi in long double."""
    C = np.clongdouble
    grid = DIMS[::-1]
    U, psi = U.astype(C).reshape(*grid, 4, 3, 3), psi.astype(C).reshape(*grid, 4, 3)
    mul = lambda m, h: (m[..., None, :, :] * h[..., None, :]).sum(-1)  # noqa: E731  (colour)
    spin = lambda g, h: (g[:, :, None] * h[..., None, :, :]).sum(-2)  # noqa: E731
    out = np.longdouble(4.0 + M0) * psi
    for mu in range(4):
        ax, g, eye = 3 - mu, oracle.gamma(mu).astype(C), np.eye(4, dtype=C)
        u = U[..., mu, :, :]
        fwd = mul(u, spin(eye + g, np.roll(psi, -1, ax)))
        bwd = np.roll(mul(np.conj(np.swapaxes(u, -1, -2)), spin(eye - g, psi)), 1, ax)
        out = out - (fwd + bwd) / 2
    return out.reshape(-1, 4, 3)


def test_no_less_exact_than_hop_by_hop():
    import paper_1204_5463_gb300 as dw

    U, psi = _inputs()
    ref = dw_long(U, psi)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.float64).reshape(-1).copy()).cuda()  # noqa: E731
    ctx = dw.dw_create(DIMS, tuple(d // 2 for d in DIMS), M0, torch.cuda.current_stream().cuda_stream)
    try:
        dw.dw_set_gauge(ctx, dev(U), True)
        out = torch.empty(psi.size * 2, dtype=torch.float64, device="cuda")
        dw.dw_apply(ctx, dev(psi), out, dw.DW_F64, 1)
        got = out.cpu().numpy().view(np.complex128).reshape(psi.shape)
    finally:
        dw.dw_destroy(ctx)
    d = np.abs(got.astype(np.clongdouble) - ref).astype(np.float64)
    assert np.linalg.norm(d) <= 8.8e-17 * np.linalg.norm(np.abs(ref).astype(np.float64))
