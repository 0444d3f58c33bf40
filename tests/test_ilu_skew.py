"""The TV preconditioner's sweeps as a wavefront over bands of 32 rows, on
arrays in the skewed layout (pair c of row 32 b + L at (b K + c + L) 32 + L).

On the CPU: the layout's indexes (in range, no two alike, consecutive along a
step), and the schedule restated in NumPy against the oracle's triangular
solves.  On the GPU: P^{-1} r at sizes with one band, a part band and many
bands, and a slice that goes on under another preconditioner, whose vectors
change layout."""
import numpy as np
import pytest

import firls_synth as fs
from oracle import firls_oracle as O

SIZES = (16, 32, 48, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512)
TOL_OP = 2e-5  # single operator application, as in the parity tests


def skewed(n):
    """(index of every pair [n][n/2], pairs per slice)."""
    H, K, nb = n // 2, n // 2 + 31, (n + 31) // 32
    row, c = np.meshgrid(np.arange(n), np.arange(H), indexing="ij")
    L = row % 32
    return (row // 32 * K + c + L) * 32 + L, nb * K * 32


@pytest.mark.parametrize("n", SIZES)
def test_skewed_indexes(n):
    idx, total = skewed(n)
    assert idx.min() >= 0 and idx.max() < total
    assert np.unique(idx).size == idx.size
    # one step of a band: its lanes' pairs are consecutive
    rows = min(n, 32)
    k = rows - 1
    step = [idx[L, k - L] for L in range(rows) if 0 <= k - L < n // 2]
    assert np.all(np.diff(step) == 1)


@pytest.mark.parametrize("n", [32, 48, 96])
def test_wavefront_equals_triangular_solves(n):
    """Lane L of a band at step k holds pair k - L; every value it needs from
    the row above comes from the step before (or the band before)."""
    sysm = O.System(fs.vd_mask(n, 0.25, 3), False, O.PSI_TV, 0, 0.0, 8e-4)
    rng = np.random.default_rng(n)
    x = fs.complex_phantom(n, 4) + 0.05 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    sysm.update_weights(x)
    r = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    P = sysm.P.tocsr()
    N, H, K, nb = n * n, n // 2, n // 2 + 31, (n + 31) // 32
    ia = (1.0 / P.diagonal()).reshape(n, n)
    left = np.array([-P[i, i - 1] if i % n else 0.0 for i in range(N)]).reshape(n, n)
    up = np.array([-P[i, i - n] if i >= n else 0.0 for i in range(N)]).reshape(n, n)
    y = np.full((n, n), np.nan, complex)
    for b in range(nb):
        for k in range(K):
            for L in range(32):
                row, c = 32 * b + L, k - L
                if row >= n or not 0 <= c < H:
                    continue
                for j in (2 * c, 2 * c + 1):
                    v = r[row, j]
                    if row:
                        v += up[row, j] * ia[row - 1, j] * y[row - 1, j]
                    if j:
                        v += left[row, j] * ia[row, j - 1] * y[row, j - 1]
                    y[row, j] = v
    z = np.full((n, n), np.nan, complex)
    for b in reversed(range(nb)):
        for k in reversed(range(K)):
            for L in range(32):
                row, c = 32 * b + L, k - L
                if row >= n or not 0 <= c < H:
                    continue
                for j in (2 * c + 1, 2 * c):
                    v = ia[row, j] * y[row, j]
                    if row < n - 1:
                        v += ia[row, j] * up[row + 1, j] * z[row + 1, j]
                    if j < n - 1:
                        v += ia[row, j] * left[row, j + 1] * z[row, j + 1]
                    z[row, j] = v
    ref = sysm.apply_Pinv(r).reshape(n, n)
    assert np.max(np.abs(z - ref)) <= 1e-10 * np.max(np.abs(ref))


@pytest.fixture(scope="module")
def F():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    return F


@pytest.mark.gpu
@pytest.mark.parametrize("precond", ["paper", "ilu0"])
@pytest.mark.parametrize("psi", [O.PSI_TV, 8], ids=["iso", "l1"])
@pytest.mark.parametrize("n", [16, 32, 48, 80, 320, 384, 512])
def test_sweeps_at_band_edges(F, n, psi, precond):
    import torch
    rng = np.random.default_rng(n)
    mask = fs.vd_mask(n, 0.25, 3)
    x, r = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)) for _ in range(2))
    x = 0.05 * x + fs.complex_phantom(n, 4)
    sysm = O.System(mask, False, psi, 0, 0.0, 1e-3, None, precond=precond)
    sysm.update_weights(x)
    ctx = F.Context(n, batch=2)
    ctx.set_operator(torch.from_numpy(np.stack([mask, mask])).cuda(), psi, 0)
    xd, rd = (torch.from_numpy(np.stack([v, v])).to(torch.complex64).cuda() for v in (x, r))
    q, z = torch.empty_like(xd), torch.empty_like(xd)
    ctx.apply_S_P(F.make_params(1, 1, lam_tv=1e-3, precond=precond), xd, rd, q, rd, z)
    torch.cuda.synchronize()
    ref = sysm.apply_Pinv(r).reshape(n, n)
    for s in range(2):
        got = z[s].cpu().numpy().astype(np.complex128)
        assert np.linalg.norm(got - ref) <= TOL_OP * np.linalg.norm(ref)
    ctx.close()


@pytest.mark.gpu
def test_preconditioner_change_keeps_the_vectors(F):
    """A slot that changes between a sweep and a diagonal preconditioner in the
    middle of an outer step and back: r and z move between the layouts and
    arrive bit for bit, so a detour of no macro steps between changes nothing,
    and the slice still converges to what it converges to without one."""
    import torch
    n = 48
    p = fs.make_problem(n, 0.3, 0.01, 3, real=False, psi=fs.PSI_TV, levels=0, lam=0.0, lam_tv=1e-3)
    mask, b = torch.from_numpy(p.mask).cuda(), torch.from_numpy(p.b.astype(np.complex64)).cuda()
    kw = dict(lam_tv=1e-3, eps=1e-4)
    outs = []
    for detour in (False, True):
        ctx = F.Context(n, batch=2)
        ctx.set_operator(mask[None].expand(2, n, n).contiguous(), p.psi, 0)
        for s in range(2):
            ctx.slot_load(s, mask, b, 0.0, 1e-3, eps=1e-4)
        ctx.run_steps(F.make_params(1, 30, **kw), 7)
        if detour:
            ctx.run_steps(F.make_params(1, 30, precond="jacobi", **kw), 5)
        ctx.run_steps(F.make_params(1, 30, **kw), 400)
        out = torch.empty(n, n, dtype=torch.complex64, device="cuda")
        ctx.slot_get(1, out)
        torch.cuda.synchronize()
        outs.append(out.cpu().numpy().astype(np.complex128))
        ctx.close()
    assert np.linalg.norm(outs[0] - outs[1]) <= 1e-4 * np.linalg.norm(outs[0])
