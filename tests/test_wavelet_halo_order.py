"""The one-launch wavelet transform at the shapes whose column steps are not split
into parts: there a column is updated by another thread than the one that sends its
boundary rows to the neighbouring CTA, so the step has to wait until they are sent.

The shapes are taken from the launch table in wavelet.cuh and the kernel's rule for
parts.  Both forms lift the same values in FP32: at most a few roundings per level
and direction apart, 2 x 5 levels of 2D steps x 6e-8 each, below 5e-6 of the norm."""
import os
import re

import numpy as np
import pytest

import firls_synth as fs

TOL = 5e-6
SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1411_5057_gb300", "csrc",
                   "wavelet.cuh")


def launch_table():
    """(side, rows per CTA) -> threads per CTA."""
    src = open(SRC).read()
    wide = int(re.search(r"WCL_WIDE_R = (\d+);", src).group(1))
    t = {(int(n), int(r)): int(h) for n, r, h in re.findall(r"\bX\((\d+), (\d+), (\d+)\)", src)}
    t.update({(int(n), wide): int(h) for n, h in re.findall(r"\bX\((\d+), (\d+)\)", src)})
    return t


def undivided():
    """(side, levels, level) whose column step keeps whole columns."""
    out = []
    table = launch_table()
    for n in sorted({n for n, _ in table}):
        for L in range(1, 6):
            if n % (1 << L) or (n >> L) % 4:
                continue
            if n > 256:
                R = 32
            else:
                R = next((n // C for C in range(8, 0, -1) if n % (C << L) == 0 and n // C <= 32), 0)
            if (n, R) not in table:
                continue
            for level in range(1, L + 1):
                m, pairs, parts = n >> (level - 1), (R >> (level - 1)) // 2, 1
                while parts * 2 * m <= table[n, R] and pairs % (parts * 2) == 0:
                    parts *= 2
                if parts == 1:
                    out.append((n, L, level))
    return out


def test_undivided_shapes():
    """More than a warp's columns: the shapes at which the order is between warps."""
    many = {(n, L, level) for n, L, level in undivided() if n >> (level - 1) > 32}
    assert many == {(48, 1, 1), (80, 1, 1), (96, 2, 2), (160, 2, 2), (192, 3, 3)} | {(512, L, 1) for L in range(1, 6)}


@pytest.mark.gpu
@pytest.mark.parametrize("n,levels", sorted({(n, L) for n, L, _ in undivided()}))
@pytest.mark.parametrize("batch", [1, 40])
def test_halo_rows_leave_before_they_change(n, levels, batch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n + levels)
    x, d, r = (torch.view_as_complex(torch.randn(batch, n, n, 2, generator=g, device="cuda")) for _ in range(3))
    mask = torch.from_numpy(fs.vd_mask(n, 0.3, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    out = []
    for rows in (0, 8):
        ctx = F.Context(n, batch=batch)
        ctx.set_operator(mask, fs.PSI_DB4, levels)
        ctx.set_tuning(rows_per_cta=rows)
        q, z = torch.empty_like(d), torch.empty_like(d)
        ctx.apply_S_P(F.make_params(1, 1, lam=1e-2), x, d, q, r, z)
        torch.cuda.synchronize()
        out.append((q, z))
        ctx.close()
    for a, b in zip(*out):
        assert float(torch.linalg.norm(b)) > 0
        worst = torch.linalg.norm((a - b).flatten(1), dim=1) / torch.linalg.norm(b.flatten(1), dim=1)
        assert float(worst.max()) <= TOL
