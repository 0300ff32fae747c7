"""The conversions between the caller's FP64 layout and the storage formats,
exactly: with all links zero and 4 + m0 = 1 the operator is the identity, so
dw_apply returns its input rounded to the storage format and widened again.
Sizes: less than a warp of sites, ragged warps and thread blocks, several fields;
values: ordinary ones, ties of the rounding, zeros, FP32 denormals, the largest
FP32 numbers, overflow, infinities and NaN. The result has to be the same number
(tolerance 0), as numpy's correctly rounded conversions give it."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _values(rng, nrhs, V, special):
    x = rng.standard_normal((nrhs, V, 24)) * 10.0 ** rng.integers(-3, 4, (nrhs, V, 1))
    x[:, ::3] = 0.0
    if special:
        odd = [1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, 1 + 2.0 ** -24 + 2.0 ** -52, -0.0, 2.0 ** -126, 2.0 ** -127, 3e-41,
               1e-50, 3.4028234e38, 3.4028235677973366e38, 1e39, -1e300, np.inf, -np.inf, np.nan, 5e-324]
        x[0, 1, : len(odd)] = odd
        x[-1, V - 2, 24 - len(odd):] = odd
    return x


def _identity(dw, dims, x, prec):
    V = int(np.prod(dims))
    ctx = dw.dw_create(dims, [d // 2 for d in dims], -3.0, torch.cuda.current_stream().cuda_stream)
    try:
        dw.dw_set_gauge(ctx, torch.zeros(V * 72, dtype=torch.float64, device="cuda"), True)
        out = torch.empty(x.size, dtype=torch.float64, device="cuda")
        dw.dw_apply(ctx, torch.from_numpy(x.reshape(-1).copy()).cuda(), out, dw.PREC[prec], x.shape[0])
        return out.cpu().numpy().reshape(x.shape)
    finally:
        dw.dw_destroy(ctx)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 6), (6, 10, 14, 2)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_f32_and_f16_round_trip(dims, nrhs):
    import paper_1204_5463_gb300 as dw

    x = _values(np.random.default_rng(1), nrhs, int(np.prod(dims)), False)
    f = x.astype(np.float32)
    assert np.array_equal(_identity(dw, dims, x, "f32"), f.astype(np.float64))
    s = np.abs(f).max(-1, keepdims=True)
    s = np.where(s > 0, s, np.float32(1))
    h = (f * (np.float32(1) / s)).astype(np.float16)
    assert np.array_equal(_identity(dw, dims, x, "f16"), (s * h.astype(np.float32)).astype(np.float64))


def test_f32_special_values():
    """Two sites far apart hold them; zero links times infinity make their
    neighbours NaN, so only those two sites and the untouched rest are compared."""
    import paper_1204_5463_gb300 as dw

    dims, V = (6, 10, 14, 2), 6 * 10 * 14 * 2
    x = _values(np.random.default_rng(2), 2, V, True)
    with np.errstate(over="ignore"):
        ref = x.astype(np.float32).astype(np.float64)
    got = _identity(dw, dims, x, "f32")
    # the site's own value: diag * psi - 1/2 * (hops of finite neighbours through zero links)
    assert np.array_equal(got[0, 1], ref[0, 1], equal_nan=True)
    assert np.array_equal(got[1, V - 2], ref[1, V - 2], equal_nan=True)
    same = np.isclose(got, ref, rtol=0, atol=0, equal_nan=True).all(-1)
    assert (~same).sum() <= 2 * 8
