"""FP64 cycles on both sides of the line between mode space and the plane kernels (nx times the points, 1.5e9): the
largest lines in mode space, and every plane kernel (6, 8 and 16 rows a lane, two to four warps a line) just above
the line, against the oracle and with the plane kernels' bit-identical switches flipped.

Tolerance: 1e-12 of the result's norm, as test_gpu_parity.py's for FP64; the transforms' sums of up to 1024 products add
below 1e-14 each to it."""
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


def apply(smg, shape, npost, options=()):
    h = smg.Handle(*shape, 1, npost)
    smg.smg_set_precision(h.h, "fp64")
    for o, v in options:
        smg.smg_set_option(h.h, o, v)
    r = inputs.rhs(*shape, seed=3)
    d = torch.from_numpy(np.ascontiguousarray(r).ravel()).cuda()
    s = torch.empty_like(d)
    smg.smg_apply(h.h, d, s)
    return r, s.cpu().numpy()


@pytest.mark.parametrize("npost", [0, 1])
@pytest.mark.parametrize("shape", [(161, 12, 9), (256, 20, 17), (257, 9, 30), (513, 33, 7), (1280, 10, 12), (2047, 5, 6), (2048, 3, 1)])
def test_long_lines_in_mode_space(smg, orc, shape, npost):
    r, s = apply(smg, shape, npost)
    ref = orc.SMG(*shape, 1, npost).apply(r).ravel()
    assert np.linalg.norm(s - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("shape", [(180, 220, 220), (256, 160, 150), (300, 140, 120), (512, 96, 62), (1280, 40, 24), (2048, 24, 16)])
def test_plane_kernels_above_the_line(smg, orc, shape):
    assert shape[0] * np.prod(shape) > 1.5e9
    r, s = apply(smg, shape, 0)
    ref = orc.SMG(*shape, 1, 0).apply(r).ravel()
    assert np.linalg.norm(s - ref) <= 1e-12 * np.linalg.norm(ref)
    for options in ([(smg.SMG_OPT_LEAN, 0)], [(smg.SMG_OPT_CLUSTER_MAX, 1)], [(smg.SMG_OPT_SOLO, 0)],
                    [(smg.SMG_OPT_RESTRICT_COLUMN, 0), (smg.SMG_OPT_WIDE_FACTORS, 0)]):
        _, t = apply(smg, shape, 0, options)
        assert np.array_equal(s, t)
