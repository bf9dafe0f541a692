"""The training calls' work memory: at most 1 GB of it stays with the library between calls, however large a call
was, and smg_net_release gives that back without a handle."""
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


def free_bytes():
    return torch.cuda.mem_get_info()[0]


SLACK = 64 << 20  # code and allocator blocks that a first launch brings with it


@pytest.mark.parametrize("call", ["forward", "loss_grad", "train"])
@pytest.mark.parametrize("dims,most", [((64, 64, 64), 1 << 30), ((256, 256, 160), 1 << 30)])
def test_idle_memory_is_bounded_and_given_back(smg, call, dims, most):
    n = dims[0] * dims[1] * dims[2]
    w = inputs.net_init_weights(seed=3)
    g = torch.Generator(device="cuda").manual_seed(1)
    kind = torch.float32 if call == "train" else torch.float64
    rho = torch.rand(n, generator=g, dtype=kind, device="cuda") - 0.5
    e = torch.rand(n, generator=g, dtype=kind, device="cuda") - 0.5
    out = torch.empty_like(rho)

    def run():
        if call == "forward":
            smg.smg_net_forward(dims, "bf16", w, rho, out)
        elif call == "loss_grad":
            smg.smg_net_loss_grad(dims, "bf16", w, rho, e)
        else:
            smg.smg_net_train([dims], [rho], [e], w, epochs=1)

    smg.smg_net_loss_grad((8, 8, 8), "bf16", w, torch.ones(512, dtype=torch.float64, device="cuda"),
                          torch.ones(512, dtype=torch.float64, device="cuda"))
    smg.smg_net_release()
    before = free_bytes()
    run()
    assert before - free_bytes() <= most + SLACK
    smg.smg_net_release()
    assert before - free_bytes() <= SLACK
    run()  # and the pool serves the next call
    smg.smg_net_release()
    assert before - free_bytes() <= SLACK
