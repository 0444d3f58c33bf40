"""Sizes above 256^2 in one launch on clusters of 10, 12 and 16 CTAs against the
tiled levels: S d and P^-1 r of both kinds, the fewest and the most levels, one
slice and more slices than clusters fit on the device.

Both forms lift the same values in FP32: at most a few roundings per level and
direction apart, 2 x 5 levels of 2D steps x 6e-8 each, below 5e-6 of the norm."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 5e-6


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    return F


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("psi", [fs.PSI_HAAR, fs.PSI_DB4], ids=["haar", "db4"])
@pytest.mark.parametrize("n,levels,batch", [(320, 1, 1), (320, 4, 17), (384, 2, 1), (384, 5, 13), (512, 1, 1),
                                            (512, 5, 9)])
def test_wide_cluster_equals_tiled_levels(F, n, levels, batch, psi, real):
    g = torch.Generator(device="cuda").manual_seed(n + levels)
    def crandn():
        v = torch.randn(batch, n, n, 2, generator=g, device="cuda")
        if real:
            v[..., 1] = 0
        return torch.view_as_complex(v)
    x, d, r = crandn(), crandn(), crandn()
    mask = torch.from_numpy(fs.vd_mask(n, 0.25, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    out = []
    for rows in (0, 8):
        ctx = F.Context(n, batch=batch, real=real)
        ctx.set_operator(mask, psi, levels)
        ctx.set_tuning(rows_per_cta=rows)
        q, z = torch.empty_like(d), torch.empty_like(d)
        ctx.apply_S_P(F.make_params(1, 1, lam=1e-2), x, d, q, r, z)
        out.append((q, z))
        ctx.close()
    for a, b in zip(*out):
        assert float(torch.linalg.norm(b)) > 0
        assert float(torch.linalg.norm(a - b)) <= TOL * float(torch.linalg.norm(b))
