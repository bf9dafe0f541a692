"""The V-cycle in the x-lines' sine eigenvectors (modal.cuh) against the oracle's cycle, at the sizes
where its layout changes: the lanes and lines a plane is spread over (32, 64, 128, 256, 512 lines and
one more), odd and even x-lines (the transform's fold), rows that are no multiple of a vector, one
line, one plane, one point, planes too many for one CTA's shared memory (slabs, and step by step with
two sweeps), several right-hand sides.

Tolerances.  FP64: 1e-12 as for the plane kernels (test_gpu_parity.py).  FP32: every value passes two
transforms (each a rounding of the input, the fold, the matrix and sums of 16: below 2e-7 of the norm
up to 2048 points) and a cycle of relaxations that round at 6e-8 a step without amplification; 1e-6 of the
norm covers both.  BF16 storage computes in FP32 and rounds the result once (2^-9 = 2e-3 an element)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1212_6680_gb300 import inputs  # noqa: E402

SHAPES = [(1, 1, 1), (2, 1, 3), (7, 2, 2), (31, 32, 5), (32, 33, 4), (33, 64, 7), (12, 65, 6), (9, 127, 4), (8, 128, 9),
          (5, 129, 3), (6, 256, 3), (4, 257, 2), (3, 512, 3), (65, 3, 40), (16, 13, 257), (130, 6, 5), (257, 4, 6),
          (11, 200, 150), (6, 300, 120), (3, 400, 160)]


@pytest.fixture(scope="module")
def smg():
    from paper_1212_6680_gb300 import build

    build.build()
    from paper_1212_6680_gb300 import smg as m

    assert torch.cuda.is_available()
    return m


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("cycle", [(1, 0), (1, 1), (2, 1)])
def test_modal_cycle_matches_oracle(smg, orc, shape, cycle):
    nx, ny, nz = shape
    r = np.stack([inputs.rhs(nx, ny, nz, seed=s) for s in (21, 22)])
    T = orc.SMG(nx, ny, nz, *cycle)
    ref = np.stack([T.apply(v) for v in r])
    R = torch.from_numpy(r.reshape(2, -1).copy()).cuda()
    for prec, tol in (("fp64", 1e-12), ("fp32", 1e-6), ("bf16", 4e-3)):
        with smg.Handle(nx, ny, nz, *cycle, precision=prec) as h:
            if prec == "bf16":  # the stored result of one right-hand side, through a solve of one step
                S = torch.zeros(R.shape[1], dtype=torch.float64, device="cuda")
                smg.krylov_solve(h.h, "psd", R[0].clone(), S, 1e-30, 1, check=False)
                p = S.cpu().numpy()
                alpha = np.dot(p, ref[0].ravel()) / np.dot(ref[0].ravel(), ref[0].ravel())
                err = np.linalg.norm(p - alpha * ref[0].ravel()) / np.linalg.norm(p)
            else:
                S = torch.full_like(R, float("nan"))
                smg.smg_apply_batched(h.h, 2, R, S)
                s = S.cpu().numpy().reshape(ref.shape)
                err = max(np.linalg.norm(s[b] - ref[b]) / np.linalg.norm(ref[b]) for b in range(2))
        assert err <= tol, (shape, cycle, prec, err)


@pytest.mark.parametrize("iters", [2, 3])
def test_modal_coarsest_steps_match_oracle(smg, orc, iters):
    nx, ny, nz = 20, 37, 6
    r = inputs.rhs(nx, ny, nz, seed=23)
    ref = orc.SMG(nx, ny, nz, 1, 1, iters).apply(r).ravel()
    R = torch.from_numpy(r.ravel().copy()).cuda()
    S = torch.empty_like(R)
    for prec, tol in (("fp64", 1e-12), ("fp32", 1e-6)):
        with smg.Handle(nx, ny, nz, 1, 1, precision=prec) as h:
            smg.smg_set_option(h.h, smg.SMG_OPT_COARSE_ITERS, iters)
            smg.smg_apply(h.h, R, S)
            err = np.linalg.norm(S.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= tol, (prec, err)


def test_modal_nan_reaches_the_solver(smg):
    """A NaN in the right-hand side is reported, not lost, and the handle stays usable."""
    b = torch.from_numpy(inputs.rhs(20, 9, 8, seed=24).ravel().copy()).cuda()
    with smg.Handle(20, 9, 8, 1, 0, precision="fp32") as h:
        bad = b.clone()
        bad[100] = float("nan")
        x = torch.zeros_like(b)
        rc, _, _ = smg.krylov_solve(h.h, "fpcg", bad, x, 1e-8, 20, check=False)
        assert rc == smg.SMG_ERR_NAN
        x.zero_()
        rc, it, rel = smg.krylov_solve(h.h, "fpcg", b, x, 1e-8, 50)
        assert rc == 0 and rel <= 1e-8


@pytest.mark.parametrize("npost", [0, 1])
def test_modal_batch_of_mixed_sizes_matches_oracle(smg, orc, npost):
    """One batch of a point, a line, planes that share an SM, planes that fill one and planes that need
    slabs, at one lane configuration."""
    dims = np.array([(1, 1, 1), (5, 1, 1), (3, 2, 9), (17, 40, 33), (6, 128, 127), (5, 300, 120), (128, 5, 3)])
    rh = [inputs.rhs(int(a), int(b), int(c), seed=30 + i) for i, (a, b, c) in enumerate(dims)]
    r = [torch.from_numpy(v.ravel().copy()).cuda() for v in rh]
    h = smg.smg_batched_setup(dims, npre=1, npost=npost)
    try:
        out = [torch.full_like(v, float("nan")) for v in r]
        smg.smg_batched_apply(h, r, out)
        x = [torch.zeros_like(v) for v in r]
        rc, iters, rel = smg.smg_batched_solve(h, "fpcg", r, x)
        assert rc == 0 and (rel <= 1e-8).all()
    finally:
        smg.smg_batched_destroy(h)
    for i, (a, b, c) in enumerate(dims):
        ref = orc.SMG(int(a), int(b), int(c), 1, npost).apply(rh[i])
        err = np.linalg.norm(out[i].cpu().numpy() - ref.ravel()) / np.linalg.norm(ref)
        assert err <= 1e-6, (tuple(dims[i]), err)
