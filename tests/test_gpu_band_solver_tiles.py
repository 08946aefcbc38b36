"""A mode's solve does not depend on the other modes of its tile: the stage of a
mode alone is, bit for bit, the stage of the same mode in company (the sixteen
systems of a block share their multipliers' stream, not their units)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr", [24, 41, 64, 81])
@pytest.mark.parametrize("local", [False, True])
def test_mode_alone_equals_mode_in_company(nr, local):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_10103_gb300 import build
    build.build()
    from paper_2509_10103_gb300 import _lib as L
    M, K = 3, 31
    ctx = L.Context(nr, 2 * (M + 1), 2 * (K + 1), 8.0, 1800.0, 0.005, 8.0, 1.0, 0.0, L.PNOP_FP64, 1)
    rng = np.random.default_rng(nr)
    F = rng.standard_normal((3, nr, 2 * M + 1, K + 1)) + 1j * rng.standard_normal((3, nr, 2 * M + 1, K + 1))
    if local:  # every mode on a few rows of its own
        at = rng.integers(0, nr, size=(1, 1, 2 * M + 1, K + 1))
        F *= np.exp2(-3.0 * np.abs(np.arange(nr)[None, :, None, None] - at))
    F[..., 0] = 0.5 * (F[..., 0] + np.conj(F[..., ::-1, 0]))
    zero, out, alone = (torch.zeros(ctx.shape, dtype=torch.complex128, device="cuda") for _ in range(3))
    for op, args in ((L.OP_STAGE, lambda x: (zero, x)), (L.OP_STAGE_T_F, lambda x: (x, None))):
        ctx.pnop_apply(op, *args(torch.from_numpy(F).to("cuda")), out)
        for k in (1, 7, 18, 31):
            G = np.zeros_like(F)
            G[..., k] = F[..., k]
            ctx.pnop_apply(op, *args(torch.from_numpy(G).to("cuda")), alone)
            assert torch.equal(torch.view_as_real(out[..., k]), torch.view_as_real(alone[..., k]))
    ctx.close()
