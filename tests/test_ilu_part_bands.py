"""Sizes whose last band of 32 rows is part empty: the sweeps' lanes past the image
repeat the last row's loads, so nothing that an earlier call left in the workspace
may reach the result, not even a NaN."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", ["paper", "ilu0"])
@pytest.mark.parametrize("psi", [fs.PSI_TV, 8], ids=["iso", "l1"])
@pytest.mark.parametrize("n", [16, 48, 80])
def test_nan_left_in_the_workspace(n, psi, precond):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    batch = 3
    g = torch.Generator(device="cuda").manual_seed(n)
    x, d, r = (torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda")) for _ in range(3))
    mask = torch.from_numpy(fs.vd_mask(n, 0.3, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    params = F.make_params(1, 1, lam_tv=1e-2, precond=precond)
    out = []
    for spoil in (False, True):
        ctx = F.Context(n, batch=batch)
        ctx.set_operator(mask, psi, 0)
        q, z = torch.empty_like(d), torch.empty_like(d)
        if spoil:
            ctx.apply_S_P(params, x, d * float("nan"), q, r * float("nan"), z)
            torch.cuda.synchronize()
            assert bool(torch.isnan(z.real).all())
        ctx.apply_S_P(params, x, d, q, r, z)
        torch.cuda.synchronize()
        out.append((q, z))
        ctx.close()
    for a, b in zip(*out):
        assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
