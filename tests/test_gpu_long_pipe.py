"""Pressure solves of nearly singular matrices: m = 0 and small k_z in a long pipe.

The forcing is the gradient of a smooth pressure p of order one (zero slope at
the wall), so that the divergence it leaves in the pressure equation is of order
one too, although the matrix's inverse has norm (Lz / 2 pi)^2: a backward stable
solve returns p to rounding, and the stage almost nothing.

Measured by <S F, v> = <F, S^H v>, which needs no second set of matrices (at
these lengths a rounding in a matrix entry moves the solution by more than the
solver does).  Bound, over dt |F|: the solve's error, a few 2^-53 of p off the
null vector (the constant), times the largest row sum of D1, which takes the
gradient; 2^6 of these for both solves, and 2^3 for the sums of 3 nr terms."""
import numpy as np
import pytest

from oracle import pipe_oracle as po

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lz", [1000.0, 3000.0])
@pytest.mark.parametrize("nr", [24, 32, 48, 64])
def test_compatible_forcing(nr, Lz):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_10103_gb300 import build
    build.build()
    from paper_2509_10103_gb300 import _lib as L
    M, K, dt = 1, 3, 0.005
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), Lz, 2000.0, dt, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    o = po.Oracle(po.Params(nr=nr, M=M, K=K, Lz=Lz, Re=2000.0, dt=dt, Wo=8.0, A=1.0))
    r, kz = o.r, o.kz[1]
    F = np.zeros((3, nr, 2 * M + 1, K + 1), complex)
    F[0, :, M, 1] = -4.0 * r * (1 - r ** 2) * (1 + 0.3j)
    F[2, :, M, 1] = 1j * kz * (1 - r ** 2) ** 2 * (1 + 0.3j)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to("cuda")  # noqa: E731
    out = torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda")
    zero = np.zeros_like(F)
    ctx.pnop_apply(L.OP_STAGE, dev(zero), dev(F), out)
    got = out.cpu().numpy()
    bound = 2.0 ** -44 * np.abs(o.d1(0)).sum(axis=1).max() * dt * np.abs(F).max()
    v = np.zeros_like(F)
    v[:, :, M, 1] = np.random.default_rng(nr).standard_normal((3, nr)) / np.sqrt(3.0 * nr)
    ctx.pnop_apply(L.OP_STAGE_T_F, dev(v), None, out)
    ctx.close()
    assert abs(np.vdot(v, got).real - np.vdot(out.cpu().numpy(), F).real) < bound
