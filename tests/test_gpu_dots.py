"""T = I: (s, r) and (s, q) formed by the x/r update against the kernel that reads r and q again (the fused-tail
option keeps it), and the preconditioned steps beside them, for all three variants, ragged and 16-byte lines.

Tolerance.  The two ways add the same products in another order: n <= 110,592 products, each chain of FMAs
below 1e-14 of the sum of magnitudes, and the first ten steps of the recurrences multiply a relative change
of a scalar by less than 1e3; 1e-9 of each residual norm covers it."""
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


def history(smg, shape, prec, precond, variant, fused, graph=1):
    h = smg.Handle(*shape, 1, 0)
    smg.smg_set_precision(h.h, prec)
    smg.smg_set_option(h.h, smg.SMG_OPT_PRECOND, precond)
    smg.smg_set_option(h.h, smg.SMG_OPT_FUSED_TAIL, fused)
    smg.smg_set_option(h.h, smg.SMG_OPT_GRAPH, graph)
    b = torch.from_numpy(inputs.rhs(*shape, seed=31).ravel()).cuda()
    x = torch.zeros_like(b)
    smg.krylov_solve(h.h, variant, b, x, 1e-12, 10)
    return np.array(smg.smg_krylov_history(h.h)), x


@pytest.mark.parametrize("variant", ["pcg", "fpcg", "psd"])
@pytest.mark.parametrize("shape,prec,precond", [((1, 1, 1), "fp32", 1), ((24, 20, 16), "fp32", 1), ((33, 65, 7), "fp32", 1),
                                                ((129, 30, 20), "bf16", 1), ((48, 48, 48), "bf16", 1),
                                                ((300, 60, 20), "fp32", 1), ((31, 13, 9), "fp32", 0), ((64, 20, 12), "fp64", 0)])
def test_dots_where_s_is_written(smg, shape, prec, precond, variant):
    ref, xr = history(smg, shape, prec, precond, variant, 1)
    for graph in (0, 1):
        got, x = history(smg, shape, prec, precond, variant, 0, graph)
        assert len(got) == len(ref)
        np.testing.assert_allclose(got, ref, rtol=1e-9, atol=1e-13)
        assert float((x - xr).norm()) <= 1e-9 * float(xr.norm())
