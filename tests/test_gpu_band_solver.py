"""The integer band solver (two-sided, 16 systems and four rows at a time) at
the sizes where it can go wrong, through the stage operators against the
oracle: radial sizes around whole chunks and around the smallest grid it takes
(21; smaller ones and tables that do not fit the fixed point keep the FP64
solver), ragged tiles of k, columns of very different magnitude, NaN.

Tolerance as in test_gpu_parity.py: 1e-10 of the largest value, here per mode
(the operators reach 1e-12; the solver rounds below 2^-53 of its window)."""
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
    shape = (2, 3, nr, 2 * M + 1, K + 1)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def per_mode(got, want):
    d = np.abs(got - want).max(axis=(0, 1))
    return float((d / np.abs(want).max(axis=(0, 1))).max())


def run(env, nr, M, K, scale=None, stretch=0.0, dt=0.005, Re=1800.0):
    torch, L = env
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), 8.0, Re, dt, 8.0, 1.0, 0.0, L.PNOP_FP64, 1, stretch=stretch)
    o = po.Oracle(po.Params(nr=nr, M=M, K=K, Lz=8.0, Re=Re, dt=dt, Wo=8.0, A=1.0, stretch=stretch))
    u, F = fields(nr, M, K, nr + K)
    s = np.ones((2 * M + 1, K + 1)) if scale is None else scale
    put = lambda x: torch.from_numpy(np.ascontiguousarray(x * s)).to("cuda")  # noqa: E731
    out = torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda")
    worst = 0.0
    for op, args, want in ((L.OP_STAGE, (u, F), lambda: o.stage(u, F)),
                           (L.OP_STAGE_T_U, (F,), lambda: o.stageT(F)[0]),
                           (L.OP_STAGE_T_F, (F,), lambda: o.stageT(F)[1])):
        a = [put(x) for x in args]
        ctx.pnop_apply(op, a[0], a[1] if len(a) > 1 else None, out)
        worst = max(worst, per_mode(out.cpu().numpy() / s, want()))
    ctx.close()
    return worst


@pytest.mark.parametrize("nr", [20, 21, 22, 23, 24, 25, 33, 41, 66])
@pytest.mark.parametrize("K", [3, 17])
def test_stage_and_transposes(env, nr, K):
    assert run(env, nr, 1, K) < TOL


def test_stiff_matrices(env):
    assert run(env, 48, 2, 5, Re=30.0, dt=0.05) < TOL


def test_modes_of_very_different_magnitude(env):
    rng = np.random.default_rng(1)
    s = np.ldexp(1.0, rng.integers(-600, 600, size=(5, 18)))
    assert run(env, 32, 2, 17, scale=s) < TOL


def test_stretched_grid_keeps_the_fp64_pressure_solver(env):
    assert run(env, 32, 2, 5, stretch=0.1) < TOL


def test_nan_stays_in_its_mode(env):
    torch, L = env
    nr, M, K = 37, 2, 17
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), 8.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    u, F = (torch.from_numpy(x).to("cuda") for x in fields(nr, M, K, 5))
    a, b = torch.zeros_like(u), torch.zeros_like(u)
    ctx.pnop_apply(L.OP_STAGE, u, F, a)
    F[2, 30, 3, 4] = complex(float("nan"), 0.0)
    ctx.pnop_apply(L.OP_STAGE, u, F, b)
    hit = torch.isnan(torch.view_as_real(b)).any(-1)
    assert hit[2, 1:, 3, 4].all()
    hit[:, :, 3, 4] = False
    assert not hit.any()
    a[:, :, 3, 4] = 0
    b[:, :, 3, 4] = 0
    assert torch.equal(a, b)
    ctx.close()
