"""||r||^2 of the residual update inside the wavelet transform where a CTA's sum leaves
the FP32 range though every pixel's square is inside it.

With b -> s b, lambda -> s lambda and eps -> s^2 eps the iteration scales by s, exactly
for a power of two: the same PCG steps to a tolerance, the same relative residual
but for the last bits of the inner products (alpha and beta in FP32, 6e-8 each, over
at most 30 steps of a system of condition below 1e2: 1e-4 of the residual)."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,levels,batch,channels", [(64, 3, 1, 1), (64, 3, 4, 2), (160, 2, 2, 1), (256, 4, 2, 1)])
@pytest.mark.parametrize("psi", [fs.PSI_HAAR, fs.PSI_DB4], ids=["haar", "db4"])
def test_scaled_residual_norm(n, levels, batch, channels, psi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n)
    mask = torch.from_numpy(fs.vd_mask(n, 0.35, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    b = torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda")) * mask
    ctx = F.Context(n, batch=batch)
    ctx.set_operator(mask, psi, levels)
    if channels > 1:
        ctx.set_channels(channels)

    def solve(s, **kw):
        _, st = ctx.solve(b * s, F.make_params(1, 30, lam=s, eps=1e-2 * s * s, **kw), stats=True)
        return st

    # the first residual's squares are about s^2 each: 5e36, 1e39 and more in a CTA
    for kw in (dict(pcg_tol=1e-2, pcg_tol_rel=True), dict(pcg_tol=1e-3)):
        one, far = (solve(s, **kw) for s in (1.0, 2.0 ** 61))
        assert 0 < one["pcg_steps"] < 30 * batch
        assert far["pcg_steps"] == one["pcg_steps"]
        assert far["max_rel_residual"] == pytest.approx(one["max_rel_residual"], rel=1e-4)
    ctx.close()
