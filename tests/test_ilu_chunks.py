"""The sweeps' chunk forms (long, short, with and without the fetches into L2, which start
above 100 MB of data) give the same iterate bit for bit, for both forms of TV and for
sizes with full and part bands."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("psi", [fs.PSI_TV, 8], ids=["iso", "l1"])
@pytest.mark.parametrize("n,batch", [(16, 10000), (48, 1300), (80, 450), (128, 170), (256, 42), (320, 27), (512, 11)])
def test_chunk_forms_agree(n, batch, psi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n)
    mask = torch.from_numpy(fs.vd_mask(n, 0.35, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    b = torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda")) * mask
    params = F.make_params(1, 4, lam_tv=1e-2, eps=1e-4)

    def solve(part, shape):
        ctx = F.Context(n, batch=part.shape[0])
        ctx.set_operator(mask[:part.shape[0]].contiguous(), psi, 0)
        if shape:
            ctx.set_tuning(ilu_depth=shape)
        x = torch.view_as_real(ctx.solve(part, params)).clone()
        torch.cuda.synchronize()
        ctx.close()
        return x

    whole = solve(b, 0)
    assert bool(torch.isfinite(whole).all())
    for shape in (22, 42) if n <= 256 else (22,):
        assert torch.equal(solve(b, shape), whole), shape
    for part in (b[:1], b[-3:].contiguous()):  # without the fetches
        x = solve(part, 0)
        assert torch.equal(x, whole[:1] if part.shape[0] == 1 else whole[-3:])
