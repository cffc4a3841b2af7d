"""The network's convolutions on grids that no tile divides -- every level's
remainder, a last tile of a few voxels, the smallest grid, samples whose last
tile ends mid-way -- against the FP64 oracle.  Tolerances as for the other
network tests: BF16 values (2^-9 relative rounding) through 11 layers, a few
1e-2 relative L2."""
import numpy as np
import pytest

from oracle import unet_oracle as U

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def les_mod():
    from paper_2301_04698_gb300 import les
    les.load_library()
    return les


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300))


def field(n, seed):
    rng = np.random.default_rng(seed)
    x = 2 * np.pi * (np.arange(n) + 0.5) / n
    z, y, x = np.meshgrid(x, x, x, indexing="ij")
    f = np.zeros((n, n, n))
    for _ in range(4):
        k, ph = rng.integers(1, 3, size=3), rng.uniform(0, 2 * np.pi, size=3)
        f += rng.standard_normal() * np.sin(k[0] * x + ph[0]) * np.sin(k[1] * y + ph[1]) * np.cos(k[2] * z + ph[2])
    return f + 0.1 * rng.standard_normal((n, n, n))


@pytest.mark.parametrize("n,batch", [(8, 1), (12, 1), (20, 2), (28, 3), (12, 70)])
def test_forward_on_ragged_grids(les_mod, n, batch):
    w = U.init_weights(7)
    b = np.stack([field(n, s) for s in range(batch)])
    model = les_mod.UNet(n, max_batch=batch)
    model.set_weights(w)
    psi = model.forward(torch.from_numpy(b).to("cuda", torch.float32)).cpu().double().numpy()
    for s in sorted({0, batch // 2, batch - 1}):
        ref = U.warm_start(w.astype(np.float32).astype(np.float64), b[s].astype(np.float32).astype(np.float64))
        assert rel(psi[s], ref) < 3e-2, s


@pytest.mark.parametrize("n,batch", [(8, 1), (12, 3), (20, 1)])
def test_gradients_on_ragged_grids(les_mod, n, batch):
    w = U.init_weights(11) + 0.02 * np.random.default_rng(0).standard_normal(U.n_params())
    w32 = w.astype(np.float32).astype(np.float64)
    b = np.stack([field(n, 10 + s) for s in range(batch)])
    t = np.stack([field(n, 20 + s) for s in range(batch)])
    model = les_mod.UNet(n, max_batch=batch)
    model.set_weights(w32)
    loss, grad = model.loss_grad(torch.from_numpy(b).cuda(), torch.from_numpy(t).cuda())
    grad = grad.cpu().double().numpy()
    P = U.unpack(w32)
    gsum, lsum = np.zeros_like(w32), 0.0
    for s in range(batch):
        sc = np.sqrt(np.mean(b[s] ** 2))
        y, cache = U.forward(P, (b[s] / sc)[None])
        d = y - (t[s] / sc)[None]
        lsum += float((d * d).sum())
        gsum += U.backward(P, cache, 2.0 * d / (batch * n ** 3))[0]
    assert abs(loss - lsum / (batch * n ** 3)) < 2e-2 * loss
    off = 0
    for name, ci, co, k in U.LAYERS:
        nw = co * ci * k ** 3
        assert rel(grad[off:off + nw], gsum[off:off + nw]) < 5e-2, name
        assert rel(grad[off + nw:off + nw + co], gsum[off + nw:off + nw + co]) < 5e-2, name
        off += nw + co
