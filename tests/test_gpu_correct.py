"""The correction on grids that no column fits, from its own inputs on the device:
one plane per thread and four, partial tiles and runs, walls and periodic z."""
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


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("precision,shape", [
    (64, (3, 3, 2)),        # the smallest grid
    (32, (33, 9, 5)),       # a node past a tile in x and in y
    (64, (97, 75, 66)),     # four planes per thread, two of the last four
    (32, (100, 76, 61))])   # ... and one of them
def test_correct_from_its_inputs(les_mod, precision, shape, walls):
    """Each value is hat - dt (a - b) h, four roundings at most: eight half units in
    the last place of its terms' sizes bound the difference from the FP64 formula."""
    nx, ny, nz = shape
    case = inputs.Case(name="corr", nx=nx, ny=ny, nz=nz, dx=35.0, dy=30.0, dz=10.0, walls=walls,
                       precision=precision, init="zero", physics=(), dt=0.5, rho0_const=1.25,
                       tol=1e-10 if precision == 64 else 1e-5, maxit=20000)
    sim = les_mod.Simulation(case)
    dt = torch.float64 if precision == 64 else torch.float32
    st = {k: torch.from_numpy((s * inputs.uniform(90 + i, 0, case.n, -1, 1)).reshape(case.shape)).to("cuda", dt)
          for i, (k, s) in enumerate([("u", 3.0), ("v", 2.0), ("w", 1.0), ("p", 10.0)])}
    sim.set_state({k: v.cpu().double().numpy() for k, v in st.items()})
    for stage in ("begin", "scalar", "momentum", "solve"):
        sim.stage(stage)
    get = lambda f: np.asarray(sim.get(f), dtype=np.float64)
    psi, p = get("psi"), get("p")
    hats = [get(f) for f in ("u_hat", "v_hat", "w_hat")]
    sim.stage("correct")
    up = np.concatenate([psi[1:], psi[-1:] if walls else psi[:1]])
    down = np.concatenate([psi[:1] if walls else psi[-1:], psi[:-1]])
    pairs = [(np.roll(psi, -1, 2), np.roll(psi, 1, 2), case.dx), (np.roll(psi, -1, 1), np.roll(psi, 1, 1), case.dy),
             (up, down, case.dz)]
    eps = 8 * np.finfo(np.float64 if precision == 64 else np.float32).eps / 2
    assert np.abs(psi).max() > 0
    for f, hat, (a, b, d) in zip(("u", "v", "w"), hats, pairs):
        step = sim.dt * 0.5 / d
        assert np.all(np.abs(get(f) - (hat - step * (a - b))) <= eps * (np.abs(hat) + step * (np.abs(a) + np.abs(b)))), f
    assert np.all(np.abs(get("p") - (p + 1.25 * psi)) <= eps * (np.abs(p) + 1.25 * np.abs(psi)))
