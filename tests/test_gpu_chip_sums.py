"""The precision of the FP32 on-chip solves' sums and of the scalars formed from them,
against FP64, on right sides whose sums lose most in plain FP32."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2301_04698_gb300 import inputs

pytestmark = pytest.mark.gpu


def laplacian(v):
    return sum(np.roll(v, 1, a) + np.roll(v, -1, a) for a in range(3)) - 6 * v


def first_step(shape, b):
    """One CG iteration from zero: alpha as the kernel took it, and the relative residual."""
    from paper_2301_04698_gb300 import les
    les.load_library()
    nx, ny, nz = shape
    case = inputs.Case(name="chipsum", nx=nx, ny=ny, nz=nz, dx=1.0, dy=1.0, dz=1.0, walls=False, precision=32,
                       init="zero", physics=())
    sim = les.Simulation(case)
    x = torch.zeros(case.shape, device="cuda")
    rc, it, res = sim.poisson_solve(torch.from_numpy(b).cuda(), x, 1e-30, 1, allow_not_converged=True)
    assert it == 1
    sim.close()
    x = x.cpu().double().numpy()
    r0 = b.astype(np.float64) - b.astype(np.float64).mean()
    # x = alpha r_0 rounded node by node: its projection is alpha to much less than an ulp
    return np.float32((x * r0).sum() / (r0 * r0).sum()), res, r0


@pytest.mark.parametrize("shape,planes", [((64, 64, 64), 8),       # vectors in registers
                                          ((100, 76, 61), 8),
                                          ((150, 140, 70), 16),    # x and the ghosts in shared memory
                                          ((150, 130, 110), 16)])  # p in shared memory
@pytest.mark.parametrize("seed", [1, 2])
def test_residual_norm_of_spikes_in_a_faint_field(shape, planes, seed):
    """Clusters [[1, -1], [-1, 1]] in a field of +-a, everything a multiple of 2^-23:
    alpha is -1/8, and the residual after a step is exact in FP32, 1/8 beside the clusters
    and a elsewhere, with a^2 over a thread's 16 planes 2^-29 of 1/64.  Added in plain FP32
    within a warp, half of the field is lost (3.6e-9 of the norm).  Compensated from the
    threads on, the 12 columns of a cluster may lose theirs: 12 x 2^-35 of 1/4, 0.7e-9 of
    the norm at most.  Bound: 1e-9."""
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    a = np.round(2.0 ** 5.5 / np.sqrt(planes)) * 2.0 ** -23
    b = np.zeros((nz, ny, nx))
    h = ny // 2  # the two halves are each other's negative but for the clusters: no mean
    b[:, :h], b[:, h:] = a, -a
    g = (nz // 4, h // 5, nx // 5)
    m = min(b.size // (256 * planes), g[0] * g[1] * g[2])
    for z, y, x in np.stack(np.unravel_index(rng.permutation(g[0] * g[1] * g[2])[:m], g), 1) * (4, 5, 5) + 1:
        for yy in (y, y + h):
            b[z - 1:z + 2, yy - 1:yy + 3, x - 1:x + 3] = 0
            b[z, yy:yy + 2, x:x + 2] = [[1, -1], [-1, 1]]
    assert b.sum() == 0
    alpha, res, r0 = first_step(shape, b.astype(np.float32))
    assert alpha == -0.125
    r1 = r0 + laplacian(r0) / 8
    assert np.array_equal(r1, r1.astype(np.float32))
    assert abs(res / np.sqrt((r1 * r1).sum() / (r0 * r0).sum()) - 1) < 1e-9


@pytest.mark.parametrize("shape", [(64, 64, 64), (100, 76, 61), (150, 140, 70), (150, 130, 110)])
def test_alpha_is_rounded_once(shape):
    """alpha = r.r / p.q from the totals' full precision: within half an ulp of its value
    in FP64, and what the sums themselves are off (random over the threads, 1e-9 of a
    total; allowed: a twentieth of an ulp).  From the high parts alone it is up to one and
    a half."""
    nx, ny, nz = shape
    for seed in range(8):
        b = inputs.uniform(300 + seed, 0, nx * ny * nz, -1, 1).reshape(nz, ny, nx).astype(np.float32)
        alpha, res, r0 = first_step(shape, b)
        exact = (r0 * r0).sum() / (r0 * laplacian(r0)).sum()
        assert abs(alpha - exact) <= 0.55 * np.spacing(np.abs(np.float32(exact))), seed
