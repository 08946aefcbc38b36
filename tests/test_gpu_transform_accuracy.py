"""Accuracy of the FP64 transforms per component and per row of the field.

Forward term: u x omega is (N(u) + N(-u)) / 2 (the base-flow terms are odd), and
omega is the library's own curl, so that the reference (FP64 library FFTs, every
component transformed on its own) sees the same inputs.  Bound: an output value
passes four roundings to FP64 (two factors after the theta synthesis, after the
z pass, after the analysis) and fixed-point errors below each of them, so the
error of a component is about 2^-53 times its root mean square, and its largest
of some 10^4 values, on either side, stays below 2^-49 of the largest value.
The transpose adds the FP64 transposed curl of g x u, whose sums of nine
products cancel to about a tenth: 2^-47, row by row."""
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


LZ = 1.0e6  # wavenumbers near zero: the base-flow terms stay below the products


def setup(env, M, K, scale, seed, nr=9):
    torch, L = env
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), LZ, 1800.0, 0.005, 8.0, 0.0, 0.0, L.PNOP_FP64, 1)
    o = po.Oracle(po.Params(nr=nr, M=M, K=K, Lz=LZ, Re=1800.0, dt=0.005, Wo=8.0, A=0.0))
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((2, 3, nr, 2 * M + 1, K + 1)) + 1j * rng.standard_normal((2, 3, nr, 2 * M + 1, K + 1))
    x *= np.asarray(scale)[None, :, None, None, None]
    x[..., 0] = 0.5 * (x[..., 0] + np.conj(x[..., ::-1, 0]))

    def apply(op, a, b=None):
        out = torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda")
        dev = lambda v: None if v is None else torch.from_numpy(np.ascontiguousarray(v)).to("cuda")  # noqa: E731
        ctx.pnop_apply(op, dev(a), dev(b), out, 0.0)
        return out.cpu().numpy()
    return ctx, o, x, apply


def forward_error(env, M, K, u_of, scale, seed):
    _, L = env
    ctx, o, x, apply = setup(env, M, K, scale, seed)
    u = u_of(x[0])
    got = 0.5 * (apply(L.OP_NONLINEAR, u) + apply(L.OP_NONLINEAR, -u))
    w = apply(L.OP_CURL, u)
    ctx.close()
    up, wp = (np.stack([o.synth(c) for c in f]) for f in (u, w))
    want = np.stack([o.analysis(c) for c in np.cross(up, wp, axis=0)])
    return [float(np.abs(got[c] - want[c]).max() / np.abs(want[c]).max()) for c in range(3)]


STREAKS = [(1, 1, 1), (1e-4, 1e-4, 1), (1e-4, 1, 1e-4), (1, 1e-4, 1e-4), (1e-3, 1, 1e-6)]


@pytest.mark.parametrize("scale", STREAKS)
@pytest.mark.parametrize("M,K", [(1, 127), (2, 26), (8, 17)])
def test_forward_term_per_component(env, M, K, scale):
    assert max(forward_error(env, M, K, lambda x: x, scale, M + K)) < 2.0 ** -49


@pytest.mark.parametrize("scale", STREAKS)
@pytest.mark.parametrize("M,K", [(1, 127), (2, 26)])
def test_transpose_per_component_and_row(env, M, K, scale):
    _, L = env
    ctx, o, (u, nb), apply = setup(env, M, K, scale, M + K + 1)
    got, want = apply(L.OP_NONLINEAR_T, u, nb), o.nonlinearT(u, 0.0, nb)
    ctx.close()
    assert float((np.abs(got - want).max(axis=(2, 3)) / np.abs(want).max(axis=(2, 3))).max()) < 2.0 ** -47


@pytest.mark.parametrize("e", [-440, -40, -10, 0, 300])
@pytest.mark.parametrize("M,K", [(1, 127), (2, 26), (8, 17)])
def test_powers_of_two_and_vanishing_components(env, M, K, e):
    """u = (0, u_theta, 0) of m = 0: the theta component of u x omega vanishes, exactly, and
    a factor 2^e on u (a row at the wall being 0) is a factor 2^(2e) on the others."""
    _, L = env
    ctx, o, x, apply = setup(env, M, K, (0, 1, 0), M + K)
    u = x[0]
    u[:, :, :M] = 0
    u[:, :, M + 1:] = 0
    u[:, 0] = 0
    term = lambda v: 0.5 * apply(L.OP_NONLINEAR, v) + 0.5 * apply(L.OP_NONLINEAR, -v)  # noqa: E731
    a, b = term(u), term(np.ldexp(u.real, e) + 1j * np.ldexp(u.imag, e))
    ctx.close()
    assert np.abs(a[0]).max() > 0.1 and not a[1].any() and not b[1].any()
    for part in (np.real, np.imag):
        assert np.array_equal(np.ldexp(part(a), 2 * e), part(b))


@pytest.mark.parametrize("e", [-400, -30, 30, 300])
def test_transpose_in_powers_of_two(env, e):
    """A factor 2^e on the cotangent, bit for bit, with a row of u that vanishes (g x u is 0
    there) and a component of the cotangent that does."""
    _, L = env
    ctx, o, (u, nb), apply = setup(env, 3, 8, (1, 1, 1), 3)
    u[:, 0] = 0
    nb[0, 4] = 0
    a, b = apply(L.OP_NONLINEAR_T, u, nb), apply(L.OP_NONLINEAR_T, u, np.ldexp(nb.real, e) + 1j * np.ldexp(nb.imag, e))
    ctx.close()
    for part in (np.real, np.imag):
        assert np.array_equal(np.ldexp(part(a), e), part(b))
