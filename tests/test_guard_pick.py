"""The guard's one-launch choice: every slice keeps what the two objectives say,
bit for bit, for the smallest and larger images, one and several contrasts, an
unaligned result (copied slice by slice) and a result in place of x1."""
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


@pytest.mark.parametrize("n,batch,psi,levels", [(16, 1, fs.PSI_HAAR, 1), (80, 5, fs.PSI_DB4, 2),
                                                (320, 3, fs.PSI_TV | fs.PSI_DB4, 3)])
@pytest.mark.parametrize("out", ["aligned", "unaligned", "in place"])
def test_guard_follows_the_objectives(F, n, batch, psi, levels, out):
    g = torch.Generator(device="cuda").manual_seed(n)
    crandn = lambda: torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda"))  # noqa: E731
    mask = torch.from_numpy(fs.vd_mask(n, 0.4, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    ctx = F.Context(n, batch=batch)
    ctx.set_operator(mask, psi, levels)
    b = crandn() * mask
    params = F.make_params(1, 1, lam=1.0, lam_tv=1.0 if psi & fs.PSI_TV else 0.0)
    atb = ctx.adjoint(b)
    x1 = atb.clone()
    for s in range(batch):  # better, worse, not finite
        x1[s] = (atb[s] * 0.9, atb[s] + 10 * crandn()[s], atb[s] * float("nan"))[s % 3]
    f1, f0 = ctx.objective(b, params, x1), ctx.objective(b, params, atb)
    want = [bool(np.isfinite(u) and u <= v) for u, v in zip(f1, f0)]
    assert want[0] and not any(want[1:3])
    ref = torch.stack([x1[s] if want[s] else atb[s] for s in range(batch)])
    if out == "unaligned":
        x0 = torch.empty(batch * n * n + 1, dtype=torch.complex64, device="cuda")[1:].view(batch, n, n)
    else:
        x0 = x1 if out == "in place" else torch.empty_like(x1)
    assert ctx.warm_start_guard(b, params, x1, x0) == want
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(x0), torch.view_as_real(ref))
    ctx.close()
