"""The FP64 transforms (fixed-point FFTs) at lengths where they can go wrong,
through the nonlinear term and its transpose against the oracle: the smallest
grids, odd and radix-3 lengths, partial blocks of k, fields far from 1, NaN.
Tolerance as in test_gpu_parity.py (1e-10 of the largest value; the transforms
round below 1e-15 of it)."""
import numpy as np
import pytest

from oracle import pipe_oracle as po

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_10103_gb300 import build
    build.build()
    from paper_2509_10103_gb300 import _lib
    return torch, _lib


def fields(nr, M, K, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((2, 3, nr, 2 * M + 1, K + 1)) + 1j * rng.standard_normal((2, 3, nr, 2 * M + 1, K + 1))
    x[..., 0] = 0.5 * (x[..., 0] + np.conj(x[..., ::-1, 0]))
    return x


@pytest.mark.parametrize("M,K", [(1, 1), (2, 7), (8, 26), (15, 17), (17, 53), (31, 3), (5, 127)])
def test_nonlinear_and_transpose(env, M, K):
    torch, L = env
    nr = 9
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), 6.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    o = po.Oracle(po.Params(nr=nr, M=M, K=K, Lz=6.0, Re=1800.0, dt=0.005, Wo=8.0, A=1.0))
    u, nb = fields(nr, M, K, M + K)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to("cuda")  # noqa: E731
    out = torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda")
    for op, args, want in ((L.OP_NONLINEAR, (u, None), o.nonlinear(u, 0.3)), (L.OP_NONLINEAR_T, (u, nb), o.nonlinearT(u, 0.3, nb))):
        ctx.pnop_apply(op, dev(args[0]), None if args[1] is None else dev(args[1]), out, 0.3)
        assert np.abs(out.cpu().numpy() - want).max() < TOL * np.abs(want).max()
    ctx.close()


@pytest.mark.parametrize("e", [-400, 300])
def test_fields_far_from_one(env, e):
    """Powers of two on both factors of the transpose's products (linear in nb and in u)."""
    torch, L = env
    nr, M, K = 9, 3, 8
    ctx = L.Context(nr, 8, 18, 6.0, 1800.0, 0.005, 8.0, 0.0, 0.0, L.PNOP_FP64, 1)
    u, nb = fields(nr, M, K, 3)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to("cuda")  # noqa: E731
    a, b = (torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda") for _ in range(2))
    ctx.pnop_apply(L.OP_NONLINEAR_T, dev(u), dev(nb), a, 0.0)
    ctx.pnop_apply(L.OP_NONLINEAR_T, dev(u), dev(np.ldexp(nb.real, e) + 1j * np.ldexp(nb.imag, e)), b, 0.0)
    assert torch.equal(torch.ldexp(torch.view_as_real(a), torch.tensor(float(e), dtype=torch.float64, device="cuda")),
                       torch.view_as_real(b))
    ctx.close()


def test_nan_reaches_its_rows_only(env):
    torch, L = env
    nr, M, K = 12, 3, 8
    ctx = L.Context(nr, 8, 18, 6.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    u, _ = fields(nr, M, K, 4)
    u[0, 11, 2, 3] = np.nan
    out = torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda")
    ctx.pnop_apply(L.OP_NONLINEAR, torch.from_numpy(u).to("cuda"), None, out, 0.0)
    bad = torch.isnan(torch.view_as_real(out)).any(-1).any(0)
    assert bad[11].any() and not bad[:11].any()
    ctx.close()
