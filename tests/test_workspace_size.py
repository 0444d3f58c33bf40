"""The workspace follows the operator: a context without TV does not hold the sweeps'
layout, and one that changes to TV with slots in the middle of their outer step goes
on as if it had had the room from the start."""
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


@pytest.mark.parametrize("n,batch", [(16, 20000), (48, 2000), (256, 1000)])
def test_wavelet_context_holds_natural_sizes(F, n, batch):
    """105 bytes a pixel (ten complex vectors, two half-size ones, five FP32 arrays, the
    mask), 6.7 KB a slice of state and partial sums, and 2 MB a block of rounding."""
    mask = torch.ones(batch, n, n, dtype=torch.uint8, device="cuda")
    F.Context(16).close()  # the library's own device data
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx = F.Context(n, batch=batch)
    ctx.set_operator(mask, F.PSI_HAAR, 1)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    ctx.close()
    assert used <= batch * (105 * n * n + 6700) + 40 * (2 << 20)


@pytest.mark.parametrize("psi", [fs.PSI_TV, 8], ids=["iso", "l1"])
def test_operator_changes_in_the_middle_of_an_outer_step(F, psi):
    n, batch = 48, 3
    p = fs.make_problem(n, 0.3, 0.01, 3, real=False, psi=fs.PSI_HAAR, levels=2, lam=1e-3, lam_tv=1e-3)
    mask, b = torch.from_numpy(p.mask).cuda(), torch.from_numpy(p.b.astype(np.complex64)).cuda()
    masks = mask[None].expand(batch, n, n).contiguous()
    kw = dict(lam=1e-3, lam_tv=1e-3, eps=1e-4)
    outs = []
    for room in (False, True):
        ctx = F.Context(n, batch=batch)
        if room:
            ctx.set_operator(masks, psi, 0)
        ctx.set_operator(masks, fs.PSI_HAAR, 2)
        for s in range(batch):
            ctx.slot_load(s, mask, b, 1e-3, 1e-3, eps=1e-4)
        ctx.run_steps(F.make_params(1, 30, **kw), 7)
        ctx.set_operator(masks, psi | fs.PSI_HAAR, 2)
        ctx.slot_move(0, 1)
        ctx.run_steps(F.make_params(1, 30, precond="none", **kw), 40)
        ctx.run_steps(F.make_params(1, 30, **kw), 200)
        out = [torch.empty(n, n, dtype=torch.complex64, device="cuda") for _ in range(2)]
        ctx.slot_get(1, out[0])
        ctx.slot_get(2, out[1])
        torch.cuda.synchronize()
        outs.append([torch.view_as_real(o).cpu().numpy() for o in out])
        ctx.close()
    assert np.isfinite(outs[0]).all() and np.any(outs[0][0])
    assert np.array_equal(outs[0], outs[1])
    assert np.array_equal(outs[0][0], outs[0][1])


@pytest.mark.parametrize("psi", [fs.PSI_TV | fs.PSI_HAAR, 8 | fs.PSI_HAAR], ids=["iso", "l1"])
def test_solves_after_an_operator_change(F, psi):
    n, batch = 64, 2
    p = fs.make_problem(n, 0.3, 0.01, 3, real=False, psi=fs.PSI_HAAR, levels=2, lam=1e-3, lam_tv=1e-3)
    b = torch.from_numpy(np.stack([p.b, p.b]).astype(np.complex64)).cuda()
    masks = torch.from_numpy(np.stack([p.mask, p.mask])).cuda()
    prm = F.make_params(2, 8, lam=1e-3, lam_tv=1e-3, eps=1e-4)
    fresh, used = F.Context(n, batch=batch), F.Context(n, batch=batch)
    used.set_operator(masks, fs.PSI_HAAR, 2)
    first = used.solve(b, prm).clone()
    for ctx in (fresh, used):
        ctx.set_operator(masks, psi, 2)
    x, y = fresh.solve(b, prm).clone(), used.solve(b, prm).clone()
    used.set_operator(masks, fs.PSI_HAAR, 2)
    again = used.solve(b, prm)
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(x), torch.view_as_real(y))
    assert torch.equal(torch.view_as_real(first), torch.view_as_real(again))
    fresh.close()
    used.close()
