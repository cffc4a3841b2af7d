"""The one-pass streaming CG over whole columns: its column shapes, the columns at
every edge of the grid (which wrap by their own copies), and the ways the planes
are dealt to the blocks, against the FP64 oracle and the two-phase streaming CG."""
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


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("precision,shape,max_blocks", [
    (32, (128, 16, 2), 0),      # one column, its own neighbour on every side; two planes
    (32, (384, 48, 7), 0),      # 128 x 16 columns, one of them inside the grid
    (32, (256, 32, 9), 1),      # one block walks every column
    (32, (384, 48, 60), 11),    # nine columns in equal shares of 50 planes
    (32, (384, 48, 20), 4),     # two turns, the planes of the ninth column shared
    (32, (192, 48, 60), 11),    # the same with 64 x 16 columns,
    (32, (96, 96, 60), 11),     # 32 x 32,
    (64, (192, 48, 60), 11),    # and in FP64
    (64, (64, 16, 3), 0),
    (64, (96, 96, 5), 2)])
def test_wave_cg_columns(les_mod, precision, shape, max_blocks, walls):
    """Tolerances as for the other CG kernels: the solve's own 1e-11 (FP64) or
    1e-6 (FP32) times the condition of these grids, a few hundred at most."""
    from oracle import Oracle
    nx, ny, nz = shape
    case = inputs.Case(name="wavecol", nx=nx, ny=ny, nz=nz, dx=35.0, dy=30.0, dz=10.0, walls=walls,
                       precision=precision, init="zero", physics=())
    b = inputs.uniform(51, 0, case.n, -1, 1).reshape(case.shape) + 0.25
    xr = Oracle(case.replace(precision=64)).poisson(b, tol=1e-12, maxit=20000)[0]
    dt = torch.float64 if precision == 64 else torch.float32
    tol = 1e-11 if precision == 64 else 1e-6
    bt = torch.from_numpy(b).to("cuda", dt)
    x0 = torch.from_numpy(0.1 * inputs.uniform(52, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", dt)
    out = []
    for variant, kern in ((4, "cg_wave"), (3, "cg_roll")):
        sim = les_mod.Simulation(case)
        sim.set_tuning(cg_resident=1, cg_variant=variant, cg_max_blocks=max_blocks if max_blocks else 1 << 20)
        sim.profile_reset()
        x = x0.clone()
        rc, it, res = sim.poisson_solve(bt, x, tol, 20000)
        assert rc == 0 and res <= tol
        assert {k["name"] for k in sim.profile_read() if k["launches"] and k["name"].startswith("cg_")} == {kern}
        xn = x.cpu().double().numpy()
        assert abs(xn.mean()) < (1e-14 if precision == 64 else 1e-6) * np.abs(xn).max()
        assert rel(xn, xr) < (1e-8 if precision == 64 else 5e-4), kern
        # stopped after an odd and an even count: x has every update
        part = []
        for n in (3, 4):
            x = x0.clone()
            rc, it, res = sim.poisson_solve(bt, x, 1e-30, n, allow_not_converged=True)
            assert rc == les_mod.LES_ERR_NOT_CONVERGED and it == n
            part.append(x.cpu().double().numpy())
        out.append((xn, part))
    for a, b in zip([out[0][0], *out[0][1]], [out[1][0], *out[1][1]]):
        assert rel(a, b) < (1e-9 if precision == 64 else 5e-4)
