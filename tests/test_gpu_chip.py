"""The register-brick CG (cg_resident 0 on grids the 128-wide register kernel
does not take) at the edges of its plans: bricks of unequal extents in every
direction, sides that wrap onto themselves, walls, one block, few and many
planes per thread, ghosts in registers and in shared memory."""
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


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def setup(les_mod, shape, precision, walls, max_blocks):
    nx, ny, nz = shape
    case = inputs.Case(name="chip", nx=nx, ny=ny, nz=nz, dx=35.0, dy=30.0, dz=10.0, walls=walls,
                       precision=precision, init="zero", physics=())
    sim = les_mod.Simulation(case)
    sim.set_tuning(cg_resident=0, cg_variant=0, cg_max_blocks=max_blocks if max_blocks else 1 << 20)
    return case, sim


def launches(sim):
    return {k["name"]: k["launches"] for k in sim.profile_read()}


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("precision,shape,max_blocks", [
    (64, (3, 3, 2), 0),         # the smallest grid: bricks of one node along a side
    (32, (5, 3, 7), 1),         # one block: every side wraps onto itself or mirrors
    (64, (37, 11, 13), 0),      # no extent divides into equal bricks
    (32, (50, 47, 33), 0),
    (32, (33, 31, 29), 3),      # three bricks would need 29 planes per thread: not on chip
    (32, (33, 31, 24), 3),      # 24 planes per thread, three bricks along x
    (32, (20, 24, 24), 1),      # 24 planes per thread, x and no ghosts in shared memory
    (32, (40, 25, 23), 2),      # 23 of 24 planes, z or y faces between two bricks
    (64, (22, 23, 12), 1),      # 12 planes per thread in FP64
    (64, (30, 30, 11), 2),      # runs of unequal length
    (32, (500, 3, 3), 0),       # long rows, several bricks along x
    (64, (17, 130, 5), 20),     # more ghosts than registers take
    # p in shared memory, r in registers, q formed twice:
    (32, (64, 32, 64), 4),      # whole bricks of 64 planes, walls or their own z neighbour
    (32, (60, 31, 57), 5),      # partial rows and columns, 57 of 64 planes
    (32, (64, 32, 90), 8),      # two bricks along z
    (32, (96, 48, 28), 9),      # 28 of 32 planes
    (32, (50, 30, 80), 6),      # 80 planes of a brick: not on chip
    (32, (50, 31, 80), 8)])     # 40 of 40 planes
def test_chip_cg_matches_oracle(les_mod, precision, shape, max_blocks, walls):
    """Against the FP64 oracle (its CG to 1e-12) and the one-pass streaming CG,
    which follows the same iterates; tolerances as for the other CG kernels:
    the solve's own 1e-11 (FP64) or 1e-6 (FP32) times the condition of these
    grids, a few hundred at most."""
    from oracle import Oracle
    case, sim = setup(les_mod, shape, precision, walls, max_blocks)
    ref = Oracle(case.replace(precision=64))
    b = inputs.uniform(41, 0, case.n, -1, 1).reshape(case.shape) + 0.25
    xr, st, itr, _ = ref.poisson(b, tol=1e-12, maxit=20000)
    dt = torch.float64 if precision == 64 else torch.float32
    tol = 1e-11 if precision == 64 else 1e-6
    bt = torch.from_numpy(b).to("cuda", dt)
    x0 = torch.from_numpy(0.1 * inputs.uniform(42, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", dt)
    its = []
    for stream in (0, 1):
        sim.set_tuning(cg_resident=stream, cg_variant=0 if stream == 0 else 3,
                       cg_max_blocks=max_blocks if stream == 0 and max_blocks else 1 << 20)
        sim.profile_reset()
        x = x0.clone()
        rc, it, res = sim.poisson_solve(bt, x, tol, 20000)
        assert rc == 0 and res <= tol
        chip = "cg_fused" if shape in ((33, 31, 29), (50, 30, 80)) else "cg_resident"
        assert launches(sim) == {"cg_roll" if stream else chip: 1}
        xn = x.cpu().double().numpy()
        assert abs(xn.mean()) < (1e-14 if precision == 64 else 1e-6) * np.abs(xn).max()
        assert rel(xn, xr) < (1e-8 if precision == 64 else 5e-4), stream
        its.append(it)
    assert abs(its[0] - its[1]) <= 3
    sim.set_tuning(cg_resident=0, cg_variant=0, cg_max_blocks=max_blocks if max_blocks else 1 << 20)
    rc, it, res = sim.poisson_solve(bt, torch.zeros_like(bt), 1e-30, 5, allow_not_converged=True)
    if rc == les_mod.LES_ERR_NOT_CONVERGED:  # the smallest grids end before the fifth iteration
        assert it == 5
    x = torch.ones_like(bt)
    rc, it, res = sim.poisson_solve(torch.zeros_like(bt), x, tol, 100)
    assert rc == 0 and it == 0 and float(x.abs().max()) == 0.0
    sim.close()


@pytest.mark.parametrize("precision,shape,max_blocks", [(32, (40, 25, 23), 0), (64, (37, 11, 13), 0),
                                                        (32, (40, 25, 23), 2)])
def test_chip_cg_barrier_timeout_is_reported(les_mod, precision, shape, max_blocks):
    """A wait for an arrival that never comes ends after its limit with a
    status, and the handle solves normally afterwards."""
    case, sim = setup(les_mod, shape, precision, False, max_blocks)
    dt = torch.float64 if precision == 64 else torch.float32
    b = torch.from_numpy(inputs.uniform(43, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", dt)
    sim.set_tuning(barrier_timeout_ms=20.0, fault_missing_arrivals=1)
    with pytest.raises(les_mod.LesError) as e:
        sim.poisson_solve(b, torch.zeros_like(b), 1e-6, 100)
    assert e.value.status == les_mod.LES_ERR_TIMEOUT
    sim.set_tuning(barrier_timeout_ms=2000.0, fault_missing_arrivals=0)
    rc, it, res = sim.poisson_solve(b, torch.zeros_like(b), 1e-6, 2000)
    assert rc == 0 and res <= 1e-6
    sim.close()


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_chip_cg_nonfinite_right_side_is_a_breakdown(les_mod, value):
    case, sim = setup(les_mod, (50, 47, 33), 32, True, 0)
    b = torch.rand(case.shape, device="cuda")
    b[3, 4, 5] = value
    with pytest.raises(les_mod.LesError) as e:
        sim.poisson_solve(b, torch.zeros_like(b), 1e-6, 100)
    assert e.value.status == les_mod.LES_ERR_NONFINITE
    sim.close()


@pytest.mark.parametrize("precision,shape", [(32, (40, 40, 40)), (64, (24, 24, 24)), (32, (100, 76, 61))])
def test_chip_cg_repeats_bit_for_bit(les_mod, precision, shape):
    """The sums and the neighbours' faces carry the number of their iteration: a
    solve must not take what an earlier one of the same handle left, and the sums
    are folded in a fixed order, so solves in turn repeat those of a new handle."""
    nx, ny, nz = shape
    case = inputs.Case(name="chiprep", nx=nx, ny=ny, nz=nz, dx=35.0, dy=30.0, dz=10.0, walls=True,
                       precision=precision, init="zero", physics=())
    dt = torch.float64 if precision == 64 else torch.float32
    bs = [torch.from_numpy(inputs.uniform(70 + s, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", dt) for s in range(2)]

    def solve(sim, b, n):
        x = torch.zeros_like(b)
        sim.poisson_solve(b, x, 1e-30, n, allow_not_converged=True)
        return x.cpu()

    fresh = {(s, n): solve(les_mod.Simulation(case), bs[s], n) for s in range(2) for n in (7, 30)}
    sim = les_mod.Simulation(case)
    for s, n in [(0, 30), (1, 30), (1, 7), (0, 30), (0, 7), (1, 30)]:
        assert torch.equal(solve(sim, bs[s], n), fresh[s, n]), (s, n)
