"""T r of a BF16 handle is a bfloat16 vector wherever it is handed out: smg_apply and smg_apply_batched return the
values krylov_solve's iterations use, the FP32 cycle's result rounded once (the cycle itself computes in FP32)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1212_6680_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def smg():
    from paper_1212_6680_gb300 import build

    build.build()
    from paper_1212_6680_gb300 import smg as m

    assert torch.cuda.is_available()
    return m


# narrow and wide transform tiles, odd and even lines, lines folded on the way in and by a pass of their own
@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 17, 20), (128, 64, 70), (301, 9, 12)])
@pytest.mark.parametrize("npost", [0, 1])
@pytest.mark.parametrize("nb", [1, 3])
def test_bf16_apply_returns_bfloat16_values(smg, shape, npost, nb):
    n = int(np.prod(shape))
    R = torch.from_numpy(np.stack([inputs.rhs(*shape, seed=40 + b).ravel() for b in range(nb)])).cuda()
    out = {}
    for prec in ("fp32", "bf16"):
        with smg.Handle(*shape, 1, npost, precision=prec) as h:
            S = torch.full((nb, n), float("nan"), dtype=torch.float64, device="cuda")
            smg.smg_apply_batched(h.h, nb, R, S)
            out[prec] = S
    # the same FP32 cycle, rounded to nearest even: every element equal
    assert torch.equal(out["bf16"], out["fp32"].float().bfloat16().double())
