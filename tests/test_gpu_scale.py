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
    """FP64: r.r p.q would leave the range from 2^256 on.  FP32: r.r would from 2^64 on,
    its terms from 2^-63 down; at a spacing of 1 / 64 q.q would from 2^43 on, whose terms
    are those of r.r times (12 x 64^2)^2 at most."""
    if precision == 64:
        check(les_mod, shape, 64, (-300, 300), 1.0, 1e-8, 2000)
    else:
        check(les_mod, shape, 32, (-30, 43), 1 / 64, 1e-5, 2000)
        check(les_mod, shape, 32, (-75, 80), 1.0, 1e-5, 2000)


def test_first_guess_far_larger_than_the_right_side(les_mod):
    """A first guess of 1e3 for a right side of 1e-17, its residual 1e21 times that: the
    FP32 squares of neither may leave their range."""
    case = inputs.Case(name="guess", nx=50, ny=47, nz=33, dx=1.0, dy=1.0, dz=1.0, walls=True, precision=32,
                       init="zero", physics=())
    sim = les_mod.Simulation(case)
    b = torch.from_numpy(inputs.uniform(92, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", torch.float32)
    x0 = torch.from_numpy(inputs.uniform(93, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", torch.float32) * 1e3
    got = []
    for e in (0, -57):
        x = x0.clone()
        rc, it, res = sim.poisson_solve(b * 2.0 ** e * 1e-17 ** (e == 0), x, 1e-30, 30, allow_not_converged=True)
        got.append((rc, it, torch.isfinite(x).all().item()))
    assert got == [(les_mod.LES_ERR_NOT_CONVERGED, 30, True)] * 2
    sim.close()


@pytest.mark.parametrize("shape", [(128, 24, 40), (70, 33, 40)])
def test_streaming_cg(les_mod, shape):
    """Whole tiles, and ragged ones.  Squares of 2^57 fit FP32, their sum over the grid
    does not."""
    check(les_mod, shape, 32, (-20, 57), 35.0, 1e-3, 2000, tuning=dict(cg_resident=1, cg_variant=0))


@pytest.mark.parametrize("precision,shape", [(32, (65, 33, 20)), (32, (128, 40, 20)), (64, (33, 31, 9))])
def test_jacobi(les_mod, precision, shape):
    e = 80 if precision == 32 else 250
    check(les_mod, shape, precision, (-e, e), 1.0, 1e-30, 20, solver="jacobi")


@pytest.mark.parametrize("shape", [(50, 47, 33), (150, 130, 110)])
def test_solution_beyond_fp32_is_reported(les_mod, shape):
    """A right side of 1e34 at a spacing of 100 has a solution past 1e38: non-finite, not
    a solve that went well."""
    nx, ny, nz = shape
    case = inputs.Case(name="over", nx=nx, ny=ny, nz=nz, dx=100.0, dy=100.0, dz=100.0, walls=True, precision=32,
                       init="zero", physics=())
    sim = les_mod.Simulation(case)
    b = torch.from_numpy(inputs.uniform(94, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", torch.float32) * 1e34
    with pytest.raises(les_mod.LesError) as e:
        sim.poisson_solve(b, torch.zeros_like(b), 1e-4, 2000)
    assert e.value.status == les_mod.LES_ERR_NONFINITE
    sim.close()


@pytest.mark.parametrize("shape,tuning", [((24, 24, 24), {}), ((50, 47, 33), {}), ((77, 60, 50), {}),
                                          ((64, 32, 32), dict(cg_resident=2))])
def test_norm_beyond_fp64_is_a_breakdown(les_mod, shape, tuning):
    """|b|^2 of a right side of 1e200 is infinite, and so is the bound of r.r: no solve
    that went well."""
    nx, ny, nz = shape
    case = inputs.Case(name="inf", nx=nx, ny=ny, nz=nz, dx=1.0, dy=1.0, dz=1.0, walls=True, precision=64,
                       init="zero", physics=())
    sim = les_mod.Simulation(case)
    sim.set_tuning(**tuning)
    b = torch.from_numpy(inputs.uniform(95, 0, case.n, -1, 1).reshape(case.shape)).cuda() * 1e200
    with pytest.raises(les_mod.LesError) as e:
        sim.poisson_solve(b, torch.zeros_like(b), 1e-8, 100)
    assert e.value.status == les_mod.LES_ERR_NONFINITE
    sim.close()
