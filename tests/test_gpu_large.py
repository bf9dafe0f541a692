"""Solves on grids of about 2^31 points, where 32-bit counts of elements end: just below (an index plus one stride
overflows) on odd lines, and above on lines of four-element chunks.  The residual is checked with torch, slab by slab."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def smg():
    from paper_1212_6680_gb300 import build

    build.build()
    from paper_1212_6680_gb300 import smg as m

    assert torch.cuda.is_available()
    return m


def residual_norms(x, b):
    """||b - A x|| and ||b|| of x, b [nz, ny, nx]."""
    nz, rr, bb = x.shape[0], 0.0, 0.0
    for z in range(0, nz, 32):
        e = min(z + 32, nz)
        u = x[z:e]
        r = b[z:e] - 6.0 * u
        r[:, :, 1:] += u[:, :, :-1]
        r[:, :, :-1] += u[:, :, 1:]
        r[:, 1:] += u[:, :-1]
        r[:, :-1] += u[:, 1:]
        if z > 0:
            r[0] += x[z - 1]
        if e < nz:
            r[-1] += x[e]
        r[1:] += u[:-1]
        r[:-1] += u[1:]
        rr += float(r.square().sum())
        bb += float(b[z:e].square().sum())
    return rr ** 0.5, bb ** 0.5


@pytest.mark.parametrize("shape", [(2047, 512, 2049), (2048, 512, 2050)])
def test_solve_near_2_to_the_31_points(smg, shape):
    nx, ny, nz = shape
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 200e9:
        pytest.skip("needs 150 GB of free device memory")
    g = torch.Generator(device="cuda").manual_seed(5)
    b = torch.rand((nz, ny, nx), generator=g, dtype=torch.float64, device="cuda") - 0.5
    x = torch.zeros_like(b)
    with smg.Handle(nx, ny, nz, 1, 0, precision="fp32") as h:
        rc, it, rel = smg.krylov_solve(h.h, "fpcg", b, x, 1e-6, 40)
    assert rc == smg.SMG_OK and 4 <= it <= 20
    rr, bb = residual_norms(x, b)
    # FP64 sums of 2^31 squares on both sides: 1e-6 of the value is far above their rounding
    assert rr <= 1e-6 * bb and abs(rr / bb - rel) <= 1e-6 * rel
    del b, x
    torch.cuda.empty_cache()
