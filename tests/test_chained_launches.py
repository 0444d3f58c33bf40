"""Solves on both sides of the line up to which a context chains its launches
(2^16 pixels): a slice's arithmetic does not depend on its batch, so it keeps its
bits, with and without TV, the diagonal preconditioners and several contrasts,
from a captured graph and from eager launches."""
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


@pytest.mark.parametrize("own_stream", [True, False], ids=["graph", "eager"])
@pytest.mark.parametrize("psi,levels,precond", [(fs.PSI_HAAR, 3, "paper"), (fs.PSI_TV | fs.PSI_DB4, 3, "paper"),
                                                (fs.PSI_TV, 0, "ilu0"), (fs.PSI_DB4, 2, "jacobi"),
                                                (fs.PSI_TV, 0, "none")])
@pytest.mark.parametrize("n,batch", [(64, 16), (128, 4), (256, 1)])
def test_same_bits_on_both_sides_of_the_line(F, n, batch, psi, levels, precond, own_stream):
    g = torch.Generator(device="cuda").manual_seed(n)
    mask = torch.from_numpy(fs.vd_mask(n, 0.3, 3).astype(np.uint8)).cuda()[None].repeat(batch + 1, 1, 1).contiguous()
    b = torch.view_as_complex(torch.randn(batch + 1, n, n, 2, generator=g, device="cuda")) * mask
    params = F.make_params(2, 4, lam=1e-2, lam_tv=1e-2 if psi & fs.PSI_TV else 0.0, eps=1e-4, precond=precond)
    torch.cuda.synchronize()
    out = []
    for count in (batch, batch + 1):
        stream = torch.cuda.Stream() if own_stream else None
        ctx = F.Context(n, batch=count, stream=stream)
        ctx.set_operator(mask[:count].contiguous(), psi, levels)
        torch.cuda.synchronize()
        x = ctx.solve(b[:count].contiguous(), params)
        torch.cuda.synchronize()
        out.append(x[:batch].clone())
        ctx.close()
    assert float(torch.linalg.norm(out[0])) > 0
    assert torch.equal(torch.view_as_real(out[0]), torch.view_as_real(out[1]))
