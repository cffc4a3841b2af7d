"""Weighted Jacobi in one persistent launch on tiles of any extents, against the
launch per sweep (solver_path 1, the same sweeps) and the FP64 oracle."""
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


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("precision,shape,max_blocks", [(64, (3, 3, 2), 0), (64, (65, 17, 5), 0), (32, (33, 31, 9), 0),
                                                        (32, (128, 40, 20), 0), (64, (70, 50, 3), 1)])
@pytest.mark.parametrize("sweeps", [0, 1, 20])
def test_jacobi_sweeps(les_mod, precision, shape, max_blocks, walls, sweeps):
    """After the same number of sweeps both paths hold the same x but for the
    rounding of a sweep's few operations (an unfused division here, a factor
    there): 1e-12 in FP64 and 1e-5 in FP32 of the solution's norm, and the same
    residual of it."""
    from oracle import Oracle
    nx, ny, nz = shape
    case = inputs.Case(name="jac", nx=nx, ny=ny, nz=nz, dx=35.0, dy=30.0, dz=10.0, walls=walls,
                       precision=precision, init="zero", physics=(), solver="jacobi")
    dt = torch.float64 if precision == 64 else torch.float32
    b = inputs.uniform(61, 0, case.n, -1, 1).reshape(case.shape) + 0.25
    x0 = 30.0 * inputs.uniform(62, 0, case.n, -1, 1).reshape(case.shape)
    bt = torch.from_numpy(b).to("cuda", dt)
    got = []
    for path in (0, 1):
        sim = les_mod.Simulation(case.replace(solver_path=path))
        if max_blocks:
            sim.set_tuning(cg_max_blocks=max_blocks)
        x = torch.from_numpy(x0).to("cuda", dt)
        rc, it, res = sim.poisson_solve(bt, x, 1e-30, sweeps, allow_not_converged=True)
        assert rc == les_mod.LES_ERR_NOT_CONVERGED and it == sweeps
        got.append((res, x.cpu().double().numpy()))
        sim.close()
    tol = 1e-12 if precision == 64 else 1e-5
    assert rel(got[0][1], got[1][1]) < tol
    assert abs(got[0][0] - got[1][0]) <= 10 * tol * got[1][0]
    xr, st, itr, resr = Oracle(case.replace(precision=64)).poisson(b, x0=x0, solver="jacobi", tol=1e-30,
                                                                  maxit=sweeps)
    assert rel(got[0][1], xr) < tol


def test_jacobi_stops_and_fails_as_documented(les_mod):
    case = inputs.Case(name="jac", nx=40, ny=33, nz=6, dx=1.0, dy=1.0, dz=1.0, precision=64, init="zero", physics=(),
                       solver="jacobi")
    sim = les_mod.Simulation(case)
    b = torch.from_numpy(inputs.uniform(63, 0, case.n, -1, 1).reshape(case.shape)).cuda()
    x = torch.zeros_like(b)
    rc, it, res = sim.poisson_solve(b, x, 1e-2, 20000)
    assert rc == 0 and 0 < it < 20000 and res <= 1e-2
    x = torch.ones_like(b)
    rc, it, res = sim.poisson_solve(torch.zeros_like(b), x, 1e-2, 100)
    assert rc == 0 and it == 0 and float(x.abs().max()) == 0.0
    bad = b.clone()
    bad[1, 2, 3] = float("nan")
    with pytest.raises(les_mod.LesError) as e:
        sim.poisson_solve(bad, torch.zeros_like(b), 1e-2, 100)
    assert e.value.status == les_mod.LES_ERR_NONFINITE
    sim.set_tuning(barrier_timeout_ms=20.0, fault_missing_arrivals=1)
    with pytest.raises(les_mod.LesError) as e:
        sim.poisson_solve(b, torch.zeros_like(b), 1e-2, 100)
    assert e.value.status == les_mod.LES_ERR_TIMEOUT
    sim.close()
