"""The weight gradient's tiling: images of one to many 8 x 32 tiles, and more
tiles than CTAs.

The loss is a sum over images and the BF16 activations of an image do not
depend on its batch, so a batch's gradients are the sums of its images'
gradients up to the FP32 rounding of at most a few hundred accumulations per
CTA and element: 1e-5 of the gradient's norm."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    return F


def _params(seed):
    rng = np.random.default_rng(seed)
    out = []
    for l, (w, b) in enumerate(fs.cnn_init_weights(seed)):
        if l == 5:  # the zero-initialised last layer would hide every earlier layer
            w = (rng.standard_normal(w.shape) * 0.05).astype(np.float32)
        out.append((w, (rng.standard_normal(b.shape) * 0.05).astype(np.float32)))
    return out


@pytest.mark.parametrize("n,batch", [(32, 1), (32, 3), (96, 2), (160, 3), (256, 3)])
def test_batch_gradient_is_the_sum_of_its_images(F, n, batch):
    g = torch.Generator(device="cuda").manual_seed(n + batch)
    c = lambda: torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda"))  # noqa: E731
    atb, tgt = c(), c()
    mask = (torch.rand(batch, n, n, generator=g, device="cuda") < 0.3).to(torch.uint8)
    params = _params(n)

    def grads(sel):
        net = F.Cnn(n, len(sel))
        net.set_params(params)
        net.train_step(atb[sel].contiguous(), mask[sel].contiguous(), tgt[sel].contiguous(), lr=0.0)
        out = net.get_grads()
        net.close()
        return out

    whole = grads(list(range(batch)))
    single = [grads([i]) for i in range(batch)]
    again = grads(list(range(batch)))
    for l in range(6):
        for k in range(2):
            ref = sum(s[l][k].astype(np.float64) for s in single)
            assert np.linalg.norm(ref) > 0
            assert np.linalg.norm(whole[l][k] - ref) <= TOL * np.linalg.norm(ref), (l, k)
            assert np.array_equal(whole[l][k], again[l][k])
