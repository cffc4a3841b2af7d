"""The training gradient's sums over voxels: their error must not grow with the grid
and the batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import unet_oracle as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(64, 16), (64, 64), (96, 16)])
def test_gradient_of_equal_samples_is_that_of_one(n, batch):
    """A batch of one sample repeated a power of two times has that sample's gradient:
    the loss's mean scales every BF16 value exactly, so the two differ by the rounding
    of their FP32 sums alone.  An accumulator takes 4096 voxels, 256 additions that may
    each lose the last bit of the partial sum; the partials come on top, 2^-24 each and
    at most 100 in a row.  Twice (256 + 100) 2^-24 = 4.3e-5 of a layer's norm, and of
    its biases', for sums that do not cancel; layers whose terms cancel (here to about
    a third) may show three times that."""
    from paper_2301_04698_gb300 import les
    les.load_library()
    w = U.init_weights(11) + 0.02 * np.random.default_rng(0).standard_normal(U.n_params())
    rng = np.random.default_rng(5)
    b, t = (torch.from_numpy(rng.standard_normal((1, n, n, n))).to("cuda", torch.float32) for _ in range(2))
    grads = []
    for k in (1, batch):
        model = les.UNet(n, max_batch=k)
        model.set_weights(w)
        grads.append(model.loss_grad(b.expand(k, n, n, n).contiguous(), t.expand(k, n, n, n).contiguous())[1].cpu().double().numpy())
        del model
    one, many = grads
    off = 0
    for name, ci, co, k in U.LAYERS:
        nw = co * ci * k ** 3
        for part in (slice(off, off + nw), slice(off + nw, off + nw + co)):
            assert np.linalg.norm(many[part] - one[part]) <= 1.3e-4 * np.linalg.norm(one[part]), name
        off += nw + co
