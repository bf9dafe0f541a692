"""FP64 cycles on the plane kernels (smg_cycle_form says which calls take them; the rest run in mode space): every number
of rows a lane (1, 2, 3, 4, 6, 8, and 16 in lines of one warp), two to four warps a line, one line, one plane, lines
that are no multiple of a vector, correction sweeps (mode 2, in (1,1) and (2,1) cycles), several right-hand sides,
against the oracle; the options that promise bit-identical results, flipped; and that a call's form does not
depend on the calls before it.

Tolerance: 1e-12 of the norm and of each plane's largest value, as test_gpu_parity.py's for FP64."""
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


def rhs(shape, nb):
    return np.stack([inputs.rhs(*shape, seed=70 + b).ravel() for b in range(nb)])


def apply(smg, shape, cycle, r, options=()):
    nb = len(r)
    assert smg.smg_cycle_form(*shape, *cycle, "fp64", nb) == smg.SMG_FORM_PLANES
    R = torch.from_numpy(r.copy()).cuda()
    S = torch.full_like(R, float("nan"))
    with smg.Handle(*shape, *cycle) as h:
        for o, v in options:
            smg.smg_set_option(h.h, o, v)
        smg.smg_apply_batched(h.h, nb, R, S)
        return S.cpu().numpy()


def check(orc, shape, cycle, r, s, what=""):
    nx, ny, nz = shape
    for b in {0, len(r) - 1}:
        ref = orc.SMG(*shape, *cycle).apply(r[b].reshape(nz, ny, nx)).ravel()
        assert_close(s[b], ref, 1e-12, shape, f"{shape} {cycle} vector {b} {what}")


CASES = [
    # rows a lane 1, 2, 3, 4: a line, a plane, and planes of several lines and levels
    ((8, 1, 1), (1, 0), 1), ((32, 1, 4), (1, 1), 1), ((30, 3, 1), (2, 1), 1), ((32, 5, 4), (1, 1), 64), ((40, 5, 4), (1, 0), 64),
    ((64, 5, 4), (2, 1), 48), ((75, 5, 4), (1, 0), 48), ((96, 5, 4), (2, 1), 32), ((96, 100, 1), (1, 0), 1),
    ((100, 1, 100), (1, 0), 1), ((101, 5, 4), (1, 1), 32), ((128, 5, 4), (2, 1), 24), ((128, 60, 12), (1, 0), 64),
    # 6 and 8
    ((161, 5, 4), (2, 1), 32), ((192, 5, 4), (1, 1), 24), ((192, 60, 12), (1, 0), 32),
    ((200, 5, 4), (1, 1), 32), ((256, 5, 4), (2, 1), 24), ((256, 128, 3), (1, 0), 24), ((256, 60, 12), (1, 0), 32),
    # two warps of 8; two, three and four warps of 16
    ((300, 1, 64), (2, 0), 1), ((300, 5, 4), (1, 1), 32), ((512, 5, 4), (2, 1), 12), ((512, 32, 32), (1, 0), 8), ((500, 300, 1), (1, 0), 1),
    ((777, 1, 6), (1, 1), 1), ((777, 5, 4), (1, 1), 12), ((777, 60, 50), (1, 0), 2), ((1024, 5, 4), (2, 1), 12),
    ((1290, 5, 4), (2, 1), 8), ((1536, 5, 4), (1, 1), 1), ((2047, 5, 4), (2, 1), 2), ((2048, 512, 1), (1, 0), 1),
]


@pytest.mark.parametrize("shape,cycle,nb", CASES)
def test_plane_kernels_match_oracle(smg, orc, shape, cycle, nb):
    r = rhs(shape, nb)
    check(orc, shape, cycle, r, apply(smg, shape, cycle, r))


@pytest.mark.parametrize("shape,cycle,nb", [c for c in CASES if c[0][1] > 1 and c[0] != (128, 60, 12)])
def test_bit_identical_options(smg, shape, cycle, nb):
    r = rhs(shape, nb)
    s = apply(smg, shape, cycle, r)
    wide = shape[0] > 256
    for options in ([(smg.SMG_OPT_LEAN, 0)], [(smg.SMG_OPT_CLUSTER_MAX, 1)], [(smg.SMG_OPT_CLUSTER_MAX, 4)],
                    [(smg.SMG_OPT_WIDE_FACTORS, 0) if wide else (smg.SMG_OPT_SOLO, 0)], [(smg.SMG_OPT_RESTRICT_COLUMN, 0)]):
        assert np.array_equal(s, apply(smg, shape, cycle, r, options)), options


@pytest.mark.parametrize("shape,cycle,nb", [((96, 100, 1), (1, 0), 1), ((101, 5, 4), (1, 1), 32), ((256, 60, 12), (1, 0), 32),
                                            ((500, 300, 1), (1, 0), 1), ((1290, 5, 4), (2, 1), 8)])
def test_cta_size(smg, orc, shape, cycle, nb):
    r = rhs(shape, nb)
    check(orc, shape, cycle, r, apply(smg, shape, cycle, r, [(smg.SMG_OPT_THREADS, 256)]), "256 threads")


@pytest.mark.parametrize("shape,cycle,nb", [((300, 1, 64), (2, 0), 1), ((300, 5, 4), (1, 1), 32), ((512, 5, 4), (2, 1), 12),
                                            ((512, 32, 32), (1, 0), 8), ((511, 300, 1), (1, 0), 1)])
def test_sixteen_rows_a_lane_in_one_warp(smg, orc, shape, cycle, nb):
    """Lines of 257 to 512 rows on one warp (SMG_OPT_WIDE_MIN_ROWS = 513): the general plane cycle."""
    r = rhs(shape, nb)
    check(orc, shape, cycle, r, apply(smg, shape, cycle, r, [(smg.SMG_OPT_WIDE_MIN_ROWS, 513)]), "one warp a line")


@pytest.mark.parametrize("iters", [2, 5])
def test_coarsest_steps_on_planes(smg, orc, iters):
    shape, cycle, nb = (101, 5, 4), (1, 1), 32
    r = rhs(shape, nb)
    s = apply(smg, shape, cycle, r, [(smg.SMG_OPT_COARSE_ITERS, iters)])
    ref = orc.SMG(*shape, *cycle, iters).apply(r[nb - 1].reshape(shape[::-1])).ravel()
    assert_close(s[nb - 1], ref, 1e-12, shape, f"{iters} coarsest steps")


@pytest.mark.parametrize("shape", [(100, 1, 100), (777, 1, 60), (1024, 30, 2)])
def test_solves_on_planes_follow_the_oracle(smg, orc, shape):
    """krylov_solve with the plane kernels' cycle: iterations and history of the oracle's solve."""
    assert smg.smg_cycle_form(*shape, 1, 0, "fp64", 1) == smg.SMG_FORM_PLANES
    b = inputs.rhs(*shape, seed=3)
    ref = orc.krylov(b, "fpcg", orc.SMG(*shape, 1, 0), tol=1e-8, maxit=100)
    with smg.Handle(*shape, 1, 0) as h:
        x = torch.zeros(b.size, dtype=torch.float64, device="cuda")
        rc, it, rel = smg.krylov_solve(h.h, "fpcg", torch.from_numpy(b.ravel().copy()).cuda(), x, tol=1e-8, maxit=100)
        hist = smg.smg_krylov_history(h.h)
    assert rc == smg.SMG_OK and rel <= 1e-8 and it == ref["iters"]
    assert np.all(np.abs(hist - ref["hist"]) <= 1e-6 * ref["hist"])


@pytest.mark.parametrize("shape,block", [((96, 5, 4), 32), ((512, 32, 12), 12)])
def test_form_follows_from_the_call_alone(smg, shape, block):
    """One vector runs in mode space and a block on the planes: neither call changes the other's result, in either
    order, and the single one can be captured after the block (its vectors are there)."""
    assert smg.smg_cycle_form(*shape, 1, 0, "fp64", 1) == smg.SMG_FORM_MODES
    assert smg.smg_cycle_form(*shape, 1, 0, "fp64", block) == smg.SMG_FORM_PLANES
    R = torch.from_numpy(rhs(shape, block)).cuda()
    one, many = torch.empty_like(R[0]), torch.empty_like(R)

    def single(h):
        smg.smg_apply(h, R[0], one)
        return one.cpu().numpy()

    def batch(h):
        smg.smg_apply_batched(h, block, R, many)
        return many.cpu().numpy()

    with smg.Handle(*shape, 1, 0) as h:
        s0 = single(h.h)
        b0 = batch(h.h)
        assert np.array_equal(single(h.h), s0)
        x = torch.zeros_like(R[0])
        _, it0, _ = smg.krylov_solve(h.h, "fpcg", R[0], x, 1e-8, 50)
    with smg.Handle(*shape, 1, 0) as h:
        assert np.array_equal(batch(h.h), b0)
        g = torch.cuda.CUDAGraph()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(g, stream=side):
            smg.smg_apply(h.h, R[0], one)
        one.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(one.cpu().numpy(), s0)
        y = torch.zeros_like(R[0])
        _, it1, _ = smg.krylov_solve(h.h, "fpcg", R[0], y, 1e-8, 50)
    assert it0 == it1 and torch.equal(x, y)


def test_eigenpairs_across_the_line(smg):
    """A block whose applications start on the planes and go to mode space as columns converge: eigenvalues
    within 1e-10 of the closed form, as test_gpu_parity.py's."""
    shape, m = (128, 5, 4), 12
    assert smg.smg_cycle_form(*shape, 1, 0, "fp64", m) == smg.SMG_FORM_PLANES
    assert smg.smg_cycle_form(*shape, 1, 0, "fp64", 2) == smg.SMG_FORM_MODES
    w = [4 * np.sin(np.pi * np.arange(1, n + 1) / (2 * (n + 1))) ** 2 for n in shape]
    ref = np.sort((w[2][:, None, None] + w[1][None, :, None] + w[0][None, None, :]).ravel())[:m]
    with smg.Handle(*shape, 1, 0) as h:
        X = torch.from_numpy(np.ascontiguousarray(inputs.initial_block(*shape, m, seed=7))).cuda()
        rc, it, lam = smg.lobpcg_solve(h.h, m, X, tol=1e-8, maxit=200)
    assert rc == smg.SMG_OK and np.all(np.abs(lam - ref) <= 1e-10 * ref)
