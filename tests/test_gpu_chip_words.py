"""The on-chip CG's tagged words (the sums' partials and, on small bricks, the faces
of q) across the solves of one handle that end after few iterations: their words
carry the tags that the next solve's first iterations await."""
import pytest

torch = pytest.importorskip("torch")

from paper_2301_04698_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,shape", [(64, (24, 24, 24)), (64, (50, 47, 33)), (32, (40, 40, 40))])
def test_short_solves_in_turn_repeat_those_of_a_new_handle(precision, shape):
    from paper_2301_04698_gb300 import les
    les.load_library()
    nx, ny, nz = shape
    case = inputs.Case(name="chipwords", nx=nx, ny=ny, nz=nz, dx=35.0, dy=30.0, dz=10.0, walls=True,
                       precision=precision, init="zero", physics=())
    dt = torch.float64 if precision == 64 else torch.float32
    bs = [torch.from_numpy(inputs.uniform(80 + s, 0, case.n, -1, 1).reshape(case.shape)).to("cuda", dt) for s in range(2)]

    def solve(sim, s, n):
        x = torch.zeros_like(bs[s])
        sim.poisson_solve(bs[s], x, 1e-30, n, allow_not_converged=True)
        return x.cpu()

    fresh = {}
    for s in range(2):
        for n in (0, 1, 2):
            sim = les.Simulation(case)
            fresh[s, n] = solve(sim, s, n)
            sim.close()
    sim = les.Simulation(case)
    for turn in range(60):
        for n in (1, 2, 0):
            s = (turn + n) % 2
            assert torch.equal(solve(sim, s, n), fresh[s, n]), (turn, s, n)
    sim.close()
