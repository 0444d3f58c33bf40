"""z = P^{-1} r and q = S d from and into complex64 views that start 8 bytes past a 16-byte
boundary, for every preconditioner with TV and without: the same bits as with
aligned arrays."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(16, 1), (48, 3), (256, 2)])
@pytest.mark.parametrize("psi,levels,precond", [(fs.PSI_TV, 0, "paper"), (fs.PSI_TV, 0, "ilu0"), (8, 0, "ilu0"),
                                                (fs.PSI_TV | fs.PSI_DB4, 1, "paper"), (fs.PSI_TV, 0, "jacobi"),
                                                (fs.PSI_HAAR, 1, "paper")])
def test_unaligned_z(n, batch, psi, levels, precond):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n)
    x, d, r = (torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda")) for _ in range(3))
    mask = torch.from_numpy(fs.vd_mask(n, 0.3, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    ctx = F.Context(n, batch=batch)
    ctx.set_operator(mask, psi, levels)
    params = F.make_params(1, 1, lam=1e-2, lam_tv=1e-2 if psi & (fs.PSI_TV | 8) else 0.0, precond=precond)
    out = []
    for off in (0, 1):
        room = [torch.empty(batch * n * n + 2, dtype=torch.complex64, device="cuda") for _ in range(5)]
        for v in room:
            v.fill_(7.0)
        xv, dv, rv, q, z = (v[off:off + batch * n * n].view(batch, n, n) for v in room)
        for v, w in ((xv, x), (dv, d), (rv, r)):
            v.copy_(w)
        assert all(v.data_ptr() % 16 == 8 * off for v in (xv, dv, rv, q, z))
        ctx.apply_S_P(params, xv, dv, q, rv, z)
        torch.cuda.synchronize()
        assert all(torch.equal(v[off + batch * n * n:].real, torch.full((2 - off,), 7.0, device="cuda")) for v in room)
        out.append((q.clone(), z.clone()))
    for a, b in zip(*out):
        assert float(torch.linalg.norm(a)) > 0
        assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    ctx.close()
