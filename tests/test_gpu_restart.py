"""A learned first guess that is worse than none is dropped inside the persistent CG
kernels: the step is then, bit for bit, that of a zero first guess."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import unet_oracle as U
from paper_2301_04698_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,precision,tuning,kern", [
    (32, 64, {}, "cg_resident"),                                   # register bricks
    (36, 32, {}, "cg_resident"),
    (64, 32, {}, "cg_resident"),                                   # ... with more planes
    (128, 32, {}, "cg_resident"),                                  # bricks with p in shared memory
    (32, 64, dict(cg_resident=2), "cg_resident"),                  # vectors in shared memory
    (64, 32, dict(cg_resident=2), "cg_resident"),
    (32, 64, dict(cg_resident=1), "cg_fused"),                     # two phases, any grid
    (36, 32, dict(cg_resident=1), "cg_fused"),
    (64, 64, dict(cg_resident=1, cg_variant=2), "cg_fused"),       # two phases, whole tiles
    (36, 32, dict(cg_resident=1, cg_variant=3), "cg_roll"),
    (64, 32, dict(cg_resident=1, cg_variant=4), "cg_wave")])
def test_rejected_guess_is_a_zero_guess(n, precision, tuning, kern):
    from paper_2301_04698_gb300 import les
    les.load_library()
    case = inputs.tgv(n, precision=precision, warm="learned", steps_tol=1e-8 if precision == 64 else 1e-5)
    state = inputs.initial_state(case)
    model = les.UNet(n, max_batch=1)
    model.set_weights(U.init_weights(5) + 0.05 * np.random.default_rng(1).standard_normal(U.n_params()))
    model.out_scale = 1e6  # far from any solution
    got = []
    for c in (case, case.replace(warm="zero")):
        sim = les.Simulation(c)
        sim.set_tuning(**tuning)
        sim.set_state(state)
        if c.warm == "learned":
            les.attach_model(sim, model)
        sim.profile_reset()
        st = sim.step(1)
        launches = {k["name"]: k["launches"] for k in sim.profile_read() if k["name"].startswith("cg_")}
        assert launches == {kern: c.K}
        got.append((st["iters_total"], [sim.get(f) for f in ("u", "v", "w", "p")]))
        sim.close()
    assert got[0][0] == got[1][0]
    for a, b in zip(got[0][1], got[1][1]):
        assert np.array_equal(a, b)
