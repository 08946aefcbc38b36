"""Plain PNOP_MIXED keeps the banded products in FP64: the transposed curl adds
its products to an FP64 field, so only the caller's PNOP_DF may shorten them.

With u = e_z (a constant, whose curl vanishes) and a cotangent in u_r of mode
(0, 0) on one radial row, wbar = nb x u has one row of one component, and each
u_z value of the result is one product of a D1 entry with that FP32 number.
The entries themselves come from an FP64 context's curl of unit vectors.  A
quotient then carries at most four roundings of 2^-53; double-FP32 products
carry 2^-49 each."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_transposed_curl_products_are_fp64():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_10103_gb300 import build
    build.build()
    from paper_2509_10103_gb300 import _lib as L
    nr, M, K = 24, 3, 5
    grid = (nr, 2 * (M + 1), 2 * (K + 1), 8.0, 1800.0, 0.005, 8.0, 0.0, 0.0)
    ref, ctx = L.Context(*grid, L.PNOP_FP64, 1), L.Context(*grid, L.PNOP_MIXED, 1)
    zero = lambda: torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda")  # noqa: E731
    out = zero()
    D1 = np.zeros((nr, nr))
    for j in range(nr):
        e = zero()
        e[2, j, M, 0] = 1.0
        ref.pnop_apply(L.OP_CURL, e, None, out)
        D1[:, j] = -out[1, :, M, 0].real.cpu().numpy()
    u = zero()
    u[2, :, M, 0] = 1.0
    worst = 0.0
    for j0 in range(nr):
        nb = zero()
        nb[0, j0, M, 0] = 0.7
        ctx.pnop_apply(L.OP_NONLINEAR_T, u, nb, out, 0.0)
        got = out[2, :, M, 0].real.cpu().numpy()
        js = [j for j in np.flatnonzero(D1[j0]) if j != j0]
        q = got[js] / D1[j0, js]
        worst = max(worst, float(np.ptp(q) / abs(q).max()))
    ctx.close()
    ref.close()
    assert worst < 2.0 ** -50
