"""The bytes that the profile books for a launch holding a whole solve."""
import pytest

torch = pytest.importorskip("torch")

from paper_2301_04698_gb300 import inputs

pytestmark = pytest.mark.gpu


def booked(shape, tuning, sweeps, precision=32, **kw):
    from paper_2301_04698_gb300 import les
    les.load_library()
    nx, ny, nz = shape
    case = inputs.Case(name="bytes", nx=nx, ny=ny, nz=nz, dx=1.0, dy=1.0, dz=1.0, walls=False, precision=precision,
                       init="zero", physics=(), **kw)
    sim = les.Simulation(case)
    sim.set_tuning(**tuning)
    sim.profile_reset()
    b = torch.rand(case.shape, device="cuda", dtype=torch.float64 if precision == 64 else torch.float32)
    rc, it, res = sim.poisson_solve(b, torch.zeros_like(b), 1e-30, sweeps, allow_not_converged=True)
    assert it == sweeps
    (k,) = [k for k in sim.profile_read() if k["launches"]]
    sim.close()
    return k["name"], k["bytes_per_launch"] / (case.n * precision // 8)


@pytest.mark.parametrize("sweeps", [1, 20])
def test_jacobi_books_its_sweeps(sweeps):
    """Set-up and gauge 5 fields, each pass over the grid 3."""
    assert booked((40, 33, 9), {}, sweeps, solver="jacobi") == ("jacobi", 5 + 3 * (sweeps + 1))


@pytest.mark.parametrize("variant,name,shape,setup,per", [(4, "cg_wave", (128, 64, 32), 8, 5), (3, "cg_roll", (40, 33, 9), 8, 6),
                                                          (0, "cg_fused", (40, 33, 9), 7, 8), (2, "cg_fused", (128, 64, 32), 7, 8)])
def test_streaming_cg_books_what_its_algorithm_needs(variant, name, shape, setup, per):
    """8 fields per iteration, fewer where one pass forms all of it: a rate above that of
    memory would not be one."""
    assert booked(shape, dict(cg_resident=1, cg_variant=variant), 10) == (name, setup + per * 10)
