"""The residual update inside the one-launch wavelet transform against the separate
update that the tiled forms keep: fixed-schedule wavelet solves, slices at the
start of their outer step and in PCG, one contrast and joint ones, real images,
clusters of 4 to 16 CTAs.

The residuals are formed alike; the transforms round alike and ||r||^2 only decides
tolerance stops, so after 2 x 3 PCG steps the iterates differ by the transforms'
rounding through <r, z>: 1e-5 of the norm."""
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


@pytest.mark.parametrize("n,levels,batch,channels,real", [
    (16, 1, 2, 1, False), (32, 3, 3, 1, True), (48, 2, 2, 2, False), (160, 3, 1, 1, False), (256, 4, 3, 3, False),
    (256, 3, 2, 1, True), (320, 4, 2, 1, False), (512, 5, 9, 1, False)])
@pytest.mark.parametrize("psi", [fs.PSI_HAAR, fs.PSI_DB4], ids=["haar", "db4"])
def test_fused_update_equals_the_separate_one(F, n, levels, batch, channels, real, psi):
    g = torch.Generator(device="cuda").manual_seed(n)
    mask = torch.from_numpy(fs.vd_mask(n, 0.35, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    b = torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda")) * mask
    out, stats = [], []
    for rows in (0, 8):
        ctx = F.Context(n, batch=batch, real=real)
        ctx.set_operator(mask, psi, levels)
        if channels > 1:
            ctx.set_channels(channels)
        ctx.set_tuning(rows_per_cta=rows)
        x, st = ctx.solve(b, F.make_params(2, 3, lam=1e-2, eps=1e-4), stats=True)
        torch.cuda.synchronize()
        out.append(x.clone())
        stats.append(st)
        ctx.close()
    assert float(torch.linalg.norm(out[1])) > 0
    assert float(torch.linalg.norm(out[0] - out[1])) <= TOL * float(torch.linalg.norm(out[1]))
    assert stats[0]["pcg_steps"] == stats[1]["pcg_steps"]
    a, c = (s["max_rel_residual"] for s in stats)
    assert abs(a - c) <= 1e-4 * c
