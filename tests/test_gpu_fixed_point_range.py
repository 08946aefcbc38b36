"""The fixed-point solver and transforms at the ends of the FP64 range, and with
infinities: an infinity (like a NaN) makes the whole column of its mode NaN in a
solve, and the rows it reaches in a transform; nothing else changes.

Far from 1 a mode is the same mode times a power of two (results of all rows far
above the subnormals), per mode to 1e-10 of its largest value against the oracle
as in test_gpu_band_solver.py."""
import numpy as np
import pytest

from oracle import pipe_oracle as po

pytestmark = pytest.mark.gpu


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
    shape = (2, 3, nr, 2 * M + 1, K + 1)
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    x[..., 0] = 0.5 * (x[..., 0] + np.conj(x[..., ::-1, 0]))
    return x


@pytest.mark.parametrize("e", [-960, 940])
@pytest.mark.parametrize("nr", [24, 41])
def test_solves_at_the_ends_of_the_range(env, nr, e):
    torch, L = env
    M, K = 1, 17
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), 8.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    o = po.Oracle(po.Params(nr=nr, M=M, K=K, Lz=8.0, Re=1800.0, dt=0.005, Wo=8.0, A=1.0))
    u, F = fields(nr, M, K, nr)
    put = lambda x: torch.from_numpy(np.ldexp(x.real, e) + 1j * np.ldexp(x.imag, e)).to("cuda")  # noqa: E731
    out = torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda")
    for op, args, want in ((L.OP_STAGE, (u, F), o.stage(u, F)), (L.OP_STAGE_T_F, (F,), o.stageT(F)[1])):
        a = [put(x) for x in args]
        ctx.pnop_apply(op, a[0], a[1] if len(a) > 1 else None, out)
        got = out.cpu().numpy()
        got = np.ldexp(got.real, -e) + 1j * np.ldexp(got.imag, -e)
        d = np.abs(got - want).max(axis=(0, 1)) / np.abs(want).max(axis=(0, 1))
        assert d.max() < 1e-10
    ctx.close()


@pytest.mark.parametrize("nr", [24, 41, 66])
@pytest.mark.parametrize("K", [3, 17])
def test_stage_to_its_roundings(env, nr, K):
    """Smooth columns: per mode to 2^-42 of its largest value, some hundred roundings of 2^-53 on
    either side times 2^3 for the influence and flux sums; sixteen bits lost anywhere show."""
    torch, L = env
    M = 2
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), 8.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    o = po.Oracle(po.Params(nr=nr, M=M, K=K, Lz=8.0, Re=1800.0, dt=0.005, Wo=8.0, A=1.0))
    z = fields(nr, M, K, nr + K)[0, :2, :1]
    shape = (1 - o.r ** 2)[None, :] * np.cos(np.arange(3)[:, None] + 3.0 * o.r[None, :])
    u, F = z[:, None] * shape[None, :, :, None, None]
    out = torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda")
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to("cuda")  # noqa: E731
    ctx.pnop_apply(L.OP_STAGE, dev(u), dev(F), out)
    got, want = out.cpu().numpy(), o.stage(u, F)
    ctx.close()
    d = np.abs(got - want).max(axis=(0, 1)) / np.abs(want).max(axis=(0, 1))
    assert d.max() < 2.0 ** -42


@pytest.mark.parametrize("value", [np.inf, -np.inf])
def test_infinity_in_a_solve(env, value):
    torch, L = env
    nr, M, K = 37, 2, 17
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), 8.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    u, F = (torch.from_numpy(x).to("cuda") for x in fields(nr, M, K, 5))
    a, b = torch.zeros_like(u), torch.zeros_like(u)
    ctx.pnop_apply(L.OP_STAGE, u, F, a)
    F[2, 30, 3, 4] = complex(value, 0.0)
    ctx.pnop_apply(L.OP_STAGE, u, F, b)
    ctx.close()
    hit = ~torch.isfinite(torch.view_as_real(b)).all(-1)
    assert torch.isnan(torch.view_as_real(b)[2, 1:, 3, 4]).any(-1).all()
    hit[:, :, 3, 4] = False
    assert not hit.any()
    a[:, :, 3, 4] = 0
    b[:, :, 3, 4] = 0
    assert torch.equal(a, b)


def test_infinity_in_a_transform(env):
    torch, L = env
    nr, M, K = 24, 3, 8
    ctx = L.Context(nr, 8, 18, 6.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    u = torch.from_numpy(fields(nr, M, K, 4)[0].copy()).to("cuda")
    a, b = torch.zeros_like(u), torch.zeros_like(u)
    ctx.pnop_apply(L.OP_NONLINEAR, u, None, a, 0.0)
    u[0, 23, 2, 3] = complex(0.0, np.inf)
    ctx.pnop_apply(L.OP_NONLINEAR, u, None, b, 0.0)
    ctx.close()
    rows = ~torch.isfinite(torch.view_as_real(b)).all(-1).all(0).all(-1).all(-1)
    assert bool(rows[23]) and not rows[:19].any()  # u_r enters the curl of its own row only; u_theta and u_z do not see it
    keep = ~rows
    assert torch.equal(a[:, keep], b[:, keep])
