"""Right sides of any size: multiplied by a power of two, a solve takes the same path
and its solution is multiplied by it, bit for bit, as long as the numbers themselves stay
in range -- the solvers' sums of squares must not leave it first."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2301_04698_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def les_mod():
    from paper_2301_04698_gb300 import les
    les.load_library()
    return les


def check(les_mod, shape, precision, exponents, spacing, tol, maxit, tuning=None, **kw):
    nx, ny, nz = shape
    case = inputs.Case(name="scale", nx=nx, ny=ny, nz=nz, dx=spacing, dy=spacing, dz=spacing, walls=True,
                       precision=precision, init="zero", physics=(), **kw)
    dt = torch.float64 if precision == 64 else torch.float32
    b = torch.from_numpy(inputs.uniform(91, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", dt)
    sim = les_mod.Simulation(case)
    if tuning:
        sim.set_tuning(**tuning)
    ref = torch.zeros_like(b)
    rc0, it0, rel0 = sim.poisson_solve(b, ref, tol, maxit, allow_not_converged=True)
    assert it0 > 1
    for e in exponents:
        x = torch.zeros_like(b)
        rc, it, rel = sim.poisson_solve(b * 2.0 ** e, x, tol, maxit, allow_not_converged=True)
        assert (rc, it) == (rc0, it0), e
        assert abs(rel - rel0) <= 1e-12 * rel0, e
        assert torch.equal(x, ref * 2.0 ** e), e
    sim.close()


# each in the registers of bricks, with x in registers and in shared memory, and in FP32
# with p in shared memory
@pytest.mark.parametrize("precision,shape", [(64, (24, 24, 24)), (64, (50, 47, 33)), (64, (77, 60, 50)),
                                             (32, (50, 47, 33)), (32, (100, 76, 61)), (32, (150, 130, 110))])
def test_on_chip_cg(les_mod, precision, shape):
    """FP64: r.r p.q would leave the range from 2^256 on.  FP32 at a spacing of 1 / 64: q.q
    would, whose terms are those of r.r times (12 x 64^2)^2 at most, from 2^43 on."""
    if precision == 64:
        check(les_mod, shape, 64, (-300, 300), 1.0, 1e-8, 2000)
    else:
        check(les_mod, shape, 32, (-30, 43), 1 / 64, 1e-5, 2000)


@pytest.mark.parametrize("shape", [(128, 24, 40), (70, 33, 40)])
def test_streaming_cg(les_mod, shape):
    """Whole tiles, and ragged ones.  Squares of 2^57 fit FP32, their sum over the grid
    does not."""
    check(les_mod, shape, 32, (-20, 57), 35.0, 1e-3, 2000, tuning=dict(cg_resident=1, cg_variant=0))


@pytest.mark.parametrize("precision,shape", [(32, (65, 33, 20)), (32, (128, 40, 20)), (64, (33, 31, 9))])
def test_jacobi(les_mod, precision, shape):
    e = 80 if precision == 32 else 250
    check(les_mod, shape, precision, (-e, e), 1.0, 1e-30, 20, solver="jacobi")
