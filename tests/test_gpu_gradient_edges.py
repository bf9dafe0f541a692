"""The training gradient at the edges of the weight-gradient kernels' tiles (32 x 4 x 4 points, rows dealt to
4 or 16 groups of threads), from more tiles than CTAs and from a single one, and called in turn from two
threads on streams of their own (the work buffers come from one pool), against the oracle.

Tolerances: those of test_gpu_learned.py -- FP32 activations 1e-5 of the layer's norm; the sums over n points
run in FP32 chains of n / (152 * 4) products at the largest grid here (a few hundred), below 1e-5."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1212_6680_gb300 import inputs  # noqa: E402
from tests.parity import assert_close  # noqa: E402


@pytest.fixture(scope="module")
def smg():
    from paper_1212_6680_gb300 import build

    build.build()
    from paper_1212_6680_gb300 import smg as m

    assert torch.cuda.is_available()
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64).ravel()).cuda()


@pytest.mark.parametrize("shape", [(1, 2, 1), (31, 3, 5), (32, 4, 4), (33, 5, 4), (65, 4, 3), (34, 41, 37)])
def test_gradient_at_tile_edges(smg, orc, shape):
    w = inputs.net_init_weights(seed=5, last_scale=1.0)
    rho, e = inputs.rhs(*shape, seed=6), inputs.rhs(*shape, seed=7)
    loss, g = smg.smg_net_loss_grad(shape, "fp32", w, dev(rho), dev(e))
    loss_ref, g_ref = orc.net_loss_grad(w, rho, e, act_bf16=False)
    assert abs(loss - loss_ref) <= 1e-5 * abs(loss_ref)
    for lo, hi in ((0, 432), (432, 7344), (7344, 7776)):
        assert_close(g[lo:hi], g_ref[lo:hi], 1e-5, None, f"gradient [{lo}:{hi}]", elem_tol=1e-5)


def test_gradients_from_two_threads(smg):
    shapes = [(40, 17, 9), (33, 12, 20)]
    w = inputs.net_init_weights(seed=8, last_scale=1.0)
    data = [(dev(inputs.rhs(*s, seed=9)), dev(inputs.rhs(*s, seed=10))) for s in shapes]
    torch.cuda.synchronize()
    alone = [smg.smg_net_loss_grad(s, "bf16", w, r, e) for s, (r, e) in zip(shapes, data)]
    got = [[], []]

    def work(i):
        st = torch.cuda.Stream()
        for _ in range(8):
            got[i].append(smg.smg_net_loss_grad(shapes[i], "bf16", w, *data[i], stream=st))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for i in range(2):
        assert len(got[i]) == 8
        for loss, g in got[i]:
            assert loss == alone[i][0] and np.array_equal(g, alone[i][1])
