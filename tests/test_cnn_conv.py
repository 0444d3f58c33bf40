"""The tensor-core convolution's persistent schedule: fewer tiles than CTAs, one
more than CTAs, and enough tiles per CTA to wrap its rings of stages and
accumulators.

A pixel's value depends on its own tile's products and their order only, so an
image gives the same bits alone and in a batch."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    return F


@pytest.mark.parametrize("n,batch", [(128, 2), (128, 5), (256, 3), (128, 48), (384, 9)])
def test_image_alone_and_in_a_batch(F, n, batch):
    rng = np.random.default_rng(n + batch)
    params = [(w if l < 5 else (rng.standard_normal(w.shape) * 0.05).astype(np.float32),
               (rng.standard_normal(b.shape) * 0.05).astype(np.float32))
              for l, (w, b) in enumerate(fs.cnn_init_weights(n))]
    g = torch.Generator(device="cuda").manual_seed(n)
    atb = torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda"))
    mask = (torch.rand(batch, n, n, generator=g, device="cuda") < 0.3).to(torch.uint8)

    def forward(sel):
        net = F.Cnn(n, len(sel))
        net.set_params(params)
        out = net.forward(atb[sel].contiguous(), mask[sel].contiguous()).clone()
        net.close()
        return out

    whole = forward(list(range(batch)))
    assert float(torch.linalg.norm(whole - atb)) > 0
    for i in sorted({0, 1, batch // 2, batch - 1}):
        assert torch.equal(torch.view_as_real(whole[i]), torch.view_as_real(forward([i])[0])), i
