"""The two-phase streaming CG on grids of any extents (what variant 0 runs when a
grid is not on chip and not whole FP32 columns): the edges of its tiles and runs
of planes against the FP64 oracle and the one-pass streaming CG."""
import numpy as np
import pytest
import torch

from paper_2301_04698_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def les_mod():
    from paper_2301_04698_gb300 import les
    les.load_library()
    return les


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def setup(les_mod, shape, precision, walls, max_blocks=0):
    nx, ny, nz = shape
    case = inputs.Case(name="stream", nx=nx, ny=ny, nz=nz, dx=35.0, dy=30.0, dz=10.0, walls=walls,
                       precision=precision, init="zero", physics=())
    sim = les_mod.Simulation(case)
    sim.set_tuning(cg_resident=1, cg_variant=0, cg_max_blocks=max_blocks if max_blocks else 1 << 20)
    return case, sim


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("precision,shape,max_blocks", [
    (64, (3, 3, 2), 0),        # the smallest grid, its ring on every node
    (64, (64, 16, 7), 0),      # one whole tile, its own neighbour on every side
    (64, (65, 17, 13), 0),     # one node more in either extent
    (64, (37, 45, 6), 3),      # several runs per block
    (32, (33, 31, 9), 0),      # partial tiles of the square shape
    (32, (100, 7, 40), 0),     # runs of unequal length
    (32, (70, 50, 3), 1),      # one block walks every tile
    (64, (130, 33, 24), 0),    # three tiles along x, of unequal width
    (64, (130, 50, 24), 3),    # equal shares of 80 planes: four tiles of 32 x 32 or five
    (64, (64, 50, 37), 13)])   # shares of 23 planes: one tile or two, of 32 x 16
def test_streaming_cg_matches_oracle(les_mod, precision, shape, max_blocks, walls):
    """Tolerances as for the other CG kernels: the solve's own 1e-11 (FP64) or
    1e-6 (FP32) times the condition of these grids, a few hundred at most."""
    from oracle import Oracle
    case, sim = setup(les_mod, shape, precision, walls, max_blocks)
    ref = Oracle(case.replace(precision=64))
    b = inputs.uniform(51, 0, case.n, -1, 1).reshape(case.shape) + 0.25
    xr, st, itr, _ = ref.poisson(b, tol=1e-12, maxit=20000)
    dt = torch.float64 if precision == 64 else torch.float32
    tol = 1e-11 if precision == 64 else 1e-6
    bt = torch.from_numpy(b).to("cuda", dt)
    x0 = torch.from_numpy(0.1 * inputs.uniform(52, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", dt)
    its = []
    for variant, kern in ((0, "cg_fused"), (3, "cg_roll")):
        sim.set_tuning(cg_resident=1, cg_variant=variant, cg_max_blocks=max_blocks if max_blocks else 1 << 20)
        sim.profile_reset()
        x = x0.clone()
        rc, it, res = sim.poisson_solve(bt, x, tol, 20000)
        assert rc == 0 and res <= tol
        assert {k["name"]: k["launches"] for k in sim.profile_read()} == {kern: 1}
        xn = x.cpu().double().numpy()
        assert abs(xn.mean()) < (1e-14 if precision == 64 else 1e-6) * np.abs(xn).max()
        assert rel(xn, xr) < (1e-8 if precision == 64 else 5e-4), variant
        its.append(it)
    assert abs(its[0] - its[1]) <= 3
    # stopped by maxit x holds every update so far: as the one-pass kernel leaves it
    left = []
    for variant in (0, 3):
        sim.set_tuning(cg_resident=1, cg_variant=variant)
        x = x0.clone()
        rc, it, res = sim.poisson_solve(bt, x, 1e-30, 4, allow_not_converged=True)
        left.append((it, x.cpu().double().numpy()))
    assert left[0][0] == left[1][0]
    assert rel(left[0][1], left[1][1]) < (1e-10 if precision == 64 else 1e-4)
    sim.set_tuning(cg_resident=1, cg_variant=0)
    x = torch.ones_like(bt)
    rc, it, res = sim.poisson_solve(torch.zeros_like(bt), x, tol, 100)
    assert rc == 0 and it == 0 and float(x.abs().max()) == 0.0
    # a caller's arrays at an odd offset (8- or 4-byte aligned)
    buf, out = torch.zeros(case.n + 1, device="cuda", dtype=dt), torch.zeros(case.n + 1, device="cuda", dtype=dt)
    buf[1:] = bt.reshape(-1)
    rc, it, res = sim.poisson_solve(buf[1:], out[1:], tol, 20000)
    assert rc == 0 and rel(out[1:].cpu().double().numpy().reshape(case.shape), xr) < (1e-8 if precision == 64 else 5e-4)
    sim.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_streaming_cg_failures_are_reported(les_mod, precision):
    case, sim = setup(les_mod, (70, 33, 12), precision, True)
    dt = torch.float64 if precision == 64 else torch.float32
    b = torch.from_numpy(inputs.uniform(53, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", dt)
    sim.set_tuning(barrier_timeout_ms=20.0, fault_missing_arrivals=1)
    with pytest.raises(les_mod.LesError) as e:
        sim.poisson_solve(b, torch.zeros_like(b), 1e-6, 100)
    assert e.value.status == les_mod.LES_ERR_TIMEOUT
    sim.set_tuning(barrier_timeout_ms=2000.0, fault_missing_arrivals=0)
    rc, it, res = sim.poisson_solve(b, torch.zeros_like(b), 1e-6, 2000)
    assert rc == 0 and res <= 1e-6
    bad = b.clone()
    bad[1, 2, 3] = float("inf")
    with pytest.raises(les_mod.LesError) as e:
        sim.poisson_solve(bad, torch.zeros_like(b), 1e-6, 100)
    assert e.value.status == les_mod.LES_ERR_NONFINITE
    sim.close()
