"""The column FFT passes over every supported size, one and several slices:
A^H A, A^H b, data consistency and the data term against torch's FP64 FFT.

Two FP32 FFTs of at most 512 points per direction and dimension round at about
log2(512) x 6e-8 each: 2e-6 of the norm, as for the other FFT tests."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-6


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    return F


@pytest.mark.parametrize("n", [16, 32, 48, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512])
@pytest.mark.parametrize("batch", [1, 3])
def test_column_passes_of_every_size(F, n, batch):
    g = torch.Generator(device="cuda").manual_seed(n)
    crandn = lambda: torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda"))  # noqa: E731
    mask = (torch.rand(batch, n, n, generator=g, device="cuda") < 0.4).to(torch.uint8)
    mask[:, 0, 0] = 1
    ctx = F.Context(n, batch=batch)
    ctx.set_operator(mask, fs.PSI_TV, 0)
    x, b, m = crandn(), crandn() * mask, mask.double()
    fft = lambda v: torch.fft.fft2(v.to(torch.complex128), norm="ortho")  # noqa: E731
    ifft = lambda v: torch.fft.ifft2(v, norm="ortho")  # noqa: E731
    q = torch.empty_like(x)
    ctx.apply_AHA(x, q)
    pairs = [(q, ifft(m * fft(x))), (ctx.adjoint(b), ifft(m * b)),
             (ctx.data_consistency(b, x), ifft((1 - m) * fft(x) + m * b))]
    torch.cuda.synchronize()
    for got, want in pairs:
        assert float(torch.linalg.norm(got - want)) <= TOL * float(torch.linalg.norm(want))
    f = np.array(ctx.objective(b, F.make_params(1, 1), x))
    want = 0.5 * (m * fft(x) - b).abs().square().sum((1, 2)).cpu().numpy()
    assert np.all(np.abs(f - want) <= TOL * want)
    ctx.close()
