"""The network on batches whose voxels end a few past a multiple of 64 on the coarsest
level, against the FP64 oracle; tolerances as in test_gpu_unet_tiles.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import unet_oracle as U

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300))


@pytest.mark.parametrize("n,batch", [(24, 3), (28, 6), (40, 5)])
def test_forward_and_gradient(n, batch):
    from paper_2301_04698_gb300 import les
    les.load_library()
    w32 = (U.init_weights(11) + 0.02 * np.random.default_rng(0).standard_normal(U.n_params())).astype(np.float32)
    w = w32.astype(np.float64)
    rng = np.random.default_rng(n)
    x = 2 * np.pi * (np.arange(n) + 0.5) / n
    z, y, x = np.meshgrid(x, x, x, indexing="ij")
    b = np.stack([np.sin(x + s) * np.cos(2 * y - s) * np.sin(z) + 0.1 * rng.standard_normal((n, n, n)) for s in range(batch)])
    t = np.stack([np.cos(x - s) * np.sin(y + s) * np.cos(2 * z) + 0.1 * rng.standard_normal((n, n, n)) for s in range(batch)])
    model = les.UNet(n, max_batch=batch)
    model.set_weights(w32)
    psi = model.forward(torch.from_numpy(b).cuda()).cpu().numpy()
    loss, grad = model.loss_grad(torch.from_numpy(b).cuda(), torch.from_numpy(t).cuda())
    grad = grad.cpu().double().numpy()
    P = U.unpack(w)
    gsum = np.zeros_like(w)
    for s in range(batch):
        sc = np.sqrt(np.mean(b[s] ** 2))
        yv, cache = U.forward(P, (b[s] / sc)[None])
        assert rel(psi[s], sc * (yv - yv.mean())[0]) < 3e-2, s
        gsum += U.backward(P, cache, 2.0 * (yv - (t[s] / sc)[None]) / (batch * n ** 3))[0]
    off = 0
    for name, ci, co, k in U.LAYERS:
        nw = co * ci * k ** 3
        assert rel(grad[off:off + nw], gsum[off:off + nw]) < 5e-2, name
        assert rel(grad[off + nw:off + nw + co], gsum[off + nw:off + nw + co]) < 5e-2, name
        off += nw + co
