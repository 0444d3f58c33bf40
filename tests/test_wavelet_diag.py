"""diag(Phi^T W Phi) at the edges of the kernel's shapes: filters folded into the
image (16 and 48 rows, all levels), column counts that leave threads idle, levels
whose step is larger than a CTA's 16 rows, both kinds, several slices; against the
oracle's dense products on the GPU's own weights.

FP32 sums of at most 12 x 9 positive products: 2e-5 relative, as for the larger
shapes."""
import numpy as np
import pytest

import firls_synth as fs
from oracle import firls_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    return F


@pytest.mark.parametrize("n,levels", [(16, 1), (16, 4), (48, 4), (80, 3), (96, 5), (128, 7), (320, 6)])
@pytest.mark.parametrize("psi", [fs.PSI_HAAR, fs.PSI_DB4], ids=["haar", "db4"])
def test_diagonal_at_the_edges(F, n, levels, psi):
    B = 2
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.view_as_complex(torch.randn(B, n, n, 2, generator=g, device="cuda"))
    mask = torch.from_numpy(fs.vd_mask(n, 0.4, 3).astype(np.uint8)).cuda()[None].repeat(B, 1, 1).contiguous()
    ctx = F.Context(n, batch=B)
    ctx.set_operator(mask, psi | fs.PSI_TV, levels)
    q, z = torch.empty_like(x), torch.empty_like(x)
    ctx.apply_S_P(F.make_params(1, 1, lam=1e-3, lam_tv=1e-3), x, x, q, x, z)
    ww = torch.empty(B, n, n, device="cuda")
    wt, wd, ia = torch.empty_like(ww), torch.empty_like(ww), torch.empty_like(ww)
    ctx.get_weights(ww, wt)
    ctx.get_precond(wd, ia)
    torch.cuda.synchronize()
    kind = O.PSI_DB4 if psi == fs.PSI_DB4 else O.PSI_HAAR
    for s in range(B):
        ref = O.wavelet_diag(ww[s].cpu().numpy().astype(np.float64), n, kind, levels)
        assert np.allclose(wd[s].cpu().numpy().astype(np.float64), ref, rtol=2e-5, atol=0), s
    ctx.close()
