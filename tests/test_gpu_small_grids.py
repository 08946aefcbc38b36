"""FP64 Helmholtz solves of grids below 21 radial points: the register form, taken
where the systems of a grid need a second wave, against the shared-memory form.
Both do the same operations in the same order, so the stages of the modes that a
large and a small grid share are equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr,ntheta", [(9, 128), (16, 96), (17, 96), (18, 96), (20, 64)])
def test_large_and_small_grid_agree(nr, ntheta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_10103_gb300 import build
    build.build()
    from paper_2509_10103_gb300 import _lib as L
    phys = (8.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    big, small = L.Context(nr, ntheta, 256, *phys), L.Context(nr, 8, 32, *phys)
    rng = np.random.default_rng(nr)
    x = [torch.from_numpy(rng.standard_normal(small.shape) + 1j * rng.standard_normal(small.shape)).to("cuda") for _ in range(2)]
    M, m0 = ntheta // 2 - 1, ntheta // 2 - 4

    def wide(a):
        y = torch.zeros(big.shape, dtype=torch.complex128, device="cuda")
        y[:, :, m0:m0 + 7, :16] = a
        return y
    for op, n in ((L.OP_STAGE, 2), (L.OP_STAGE_T_U, 1), (L.OP_STAGE_T_F, 1)):
        a, b = torch.zeros_like(x[0]), wide(x[0])
        small.pnop_apply(op, x[0], x[1] if n == 2 else None, a)
        out = torch.zeros_like(b)
        big.pnop_apply(op, b, wide(x[1]) if n == 2 else None, out)
        assert torch.equal(out[:, :, m0:m0 + 7, :16], a) and bool(a.abs().max() > 0)
    big.close()
    small.close()
