"""A tuning file with an entry from before the wide clusters (tiled levels at 512^2): it
no longer decides, the shapes are timed again and the new entry does."""
import numpy as np
import pytest

import firls_synth as fs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_entry_of_replaced_kernels_is_timed_again(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    n, batch, levels = 512, 2, 5
    path = tmp_path / "tune.txt"
    old = f"n={n} batch={batch} psi={fs.PSI_DB4} levels={levels} | 16 32 0\n"
    path.write_text(old)
    mask = torch.from_numpy(fs.vd_mask(n, 0.25, 3).astype(np.uint8)).cuda()[None].repeat(batch, 1, 1).contiguous()
    ctx = F.Context(n, batch=batch)
    ctx.set_operator(mask, fs.PSI_DB4, levels)
    first = ctx.autotune(str(path))
    lines = path.read_text().splitlines(keepends=True)
    assert lines[0] == old and len(lines) == 2
    assert ctx.autotune(str(path)) == first
    assert path.read_text().splitlines(keepends=True) == lines
    ctx.close()
