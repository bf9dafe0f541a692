"""The bytes smg_batched_profile_read reports are those the cycles that ran have to move: 6 words of 4 bytes a point and
application for systems whose modes fit in one CTA's shared memory, more for one that does not."""
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


def profiled_bytes(smg, dims, npost):
    dims = np.array(dims)
    b = [torch.from_numpy(inputs.rhs(*map(int, d), seed=60 + i).ravel().copy()).cuda() for i, d in enumerate(dims)]
    x = [torch.zeros_like(v) for v in b]
    h = smg.smg_batched_setup(dims, npre=1, npost=npost)
    try:
        smg.smg_batched_set_profile(h, 1)
        _, it, _ = smg.smg_batched_solve(h, "fpcg", b, x)
        launches, ms, by = smg.smg_batched_profile_read(h, 0)
    finally:
        smg.smg_batched_destroy(h)
    assert launches == it.max() and ms > 0
    return by, int(np.sum(np.prod(dims.astype(np.int64), axis=1) * it))


@pytest.mark.parametrize("npost", [0, 1])
def test_bytes_of_cycles_in_shared_memory(smg, npost):
    by, points = profiled_bytes(smg, [(33, 20, 17), (64, 64, 40), (8, 96, 90)], npost)
    assert by == 24 * points


def test_bytes_of_a_cycle_with_levels_above(smg):
    by, points = profiled_bytes(smg, [(5, 300, 120)], 0)
    # levels 0 and 1 (120 and 60 planes) in global memory, level 2 (30) in shared memory; in words a point of level 0:
    # transforms 4, level 0 4 + 2 / 2, level 1 4 / 2 + 2 / 4, level 2 2 / 4
    assert by == 4 * points * 12
