"""smg_apply under stream capture: once a handle's vectors exist a call launches kernels and allocates nothing, also
after an option that changes only what is launched.  A captured graph repeats the call it was captured from."""
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


def captured(smg, h, R, S):
    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=side):
        smg.smg_apply(h, R, S)
    return g


# planes in one CTA's shared memory and planes that need slabs; FP64 and FP32: 1e-12 and 1e-6 of the norm, as in
# test_gpu_modal.py
@pytest.mark.parametrize("shape", [(20, 37, 6), (6, 300, 120)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-6)])
def test_capture_after_the_number_of_coarsest_steps_changed(smg, orc, shape, prec, tol):
    r = inputs.rhs(*shape, seed=25)
    R = torch.from_numpy(r.ravel().copy()).cuda()
    S = torch.empty_like(R)
    with smg.Handle(*shape, 1, 1, precision=prec) as h:
        smg.smg_apply(h.h, R, S)
        graphs = []
        for iters in (2, 1):
            smg.smg_set_option(h.h, smg.SMG_OPT_COARSE_ITERS, iters)
            graphs.append((iters, captured(smg, h.h, R, S)))
        for iters, g in graphs:
            S.fill_(float("nan"))
            g.replay()
            torch.cuda.synchronize()
            ref = orc.SMG(*shape, 1, 1, iters).apply(r).ravel()
            assert np.linalg.norm(S.cpu().numpy() - ref) <= tol * np.linalg.norm(ref), iters
