"""The sweeps' one-pass set-up against the diagonal's own kernel (the Jacobi scale): 1/a
bit for bit, with and without a wavelet term, for full and part bands; and P^-1 r from
the packed weights of a later preconditioner change."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tv", [fs.PSI_TV, 8], ids=["iso", "l1"])
@pytest.mark.parametrize("wavelet,levels", [(0, 0), (fs.PSI_HAAR, 1)], ids=["tv", "tv_haar"])
@pytest.mark.parametrize("n,batch", [(16, 5), (32, 1), (48, 3), (80, 2), (256, 3), (512, 1)])
def test_set_up_equals_the_diagonal(n, batch, wavelet, levels, tv):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n)
    x, d, r = (torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda")) for _ in range(3))
    mask = torch.from_numpy(fs.vd_mask(n, 0.3, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    q, z = torch.empty_like(d), torch.empty_like(d)
    out = []
    for precond in ("jacobi", "paper"):
        ctx = F.Context(n, batch=batch)
        ctx.set_operator(mask, tv | wavelet, levels)
        ctx.apply_S_P(F.make_params(1, 1, lam=1e-2, lam_tv=1e-2, precond=precond), x, d, q, r, z)
        ia = torch.empty(batch, n, n, device="cuda")
        ctx.get_precond(None, ia)
        torch.cuda.synchronize()
        out.append(ia)
        ctx.close()
    assert bool((out[0] > 0).all())
    assert torch.equal(*out)
