"""Pixel indexes of the warm-start network on images with more than 2^31 values a
layer: the index function itself, compiled for the host, and one 8320^2 image on the
GPU against crops of its first and last corner.

A pixel of the output depends on the 13 x 13 pixels around it, in the same order of
operations wherever it lies, so crops agree bit for bit 6 pixels from their cut
edges."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import firls_synth as fs

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1411_5057_gb300", "csrc")


def test_pixel_index_has_64_bits(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src = tmp_path / "index.cpp"
    src.write_text('#include "cnn_index.h"\nextern "C" unsigned long long pixel(int y, int x, int n, int c) '
                   "{ return firls::cnn_pixel(y, x, n, c); }\n")
    lib = str(tmp_path / "index.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", lib], check=True)
    f = ctypes.CDLL(lib).pixel
    f.restype = ctypes.c_ulonglong
    for n in (128, 8192, 8320, 16384):
        for c in (16, 32):
            for y, x in ((0, 0), (0, n - 1), (n - 1, 0), (n - 1, n - 1), (n // 2, 3)):
                assert f(y, x, n, c) == (y * n + x) * c


@pytest.mark.gpu
def test_image_beyond_32_bit_indexes():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    n, m, edge = 8320, 256, 6
    if torch.cuda.mem_get_info()[0] < 60e9:
        pytest.skip("needs 60 GB of device memory")
    rng = np.random.default_rng(7)
    params = [((rng.standard_normal(w.shape) * 0.05).astype(np.float32) if l == 5 else w,
               (rng.standard_normal(b.shape) * 0.05).astype(np.float32))
              for l, (w, b) in enumerate(fs.cnn_init_weights(7))]
    g = torch.Generator(device="cuda").manual_seed(7)
    atb = torch.view_as_complex(torch.randn(1, n, n, 2, generator=g, device="cuda"))
    mask = (torch.rand(1, n, n, generator=g, device="cuda") < 0.3).to(torch.uint8)
    whole = F.Cnn(n, 1)
    whole.set_params(params)
    x1 = whole.forward(atb, mask)
    torch.cuda.synchronize()
    whole.close()
    crop = F.Cnn(m, 1)
    crop.set_params(params)
    for at in (0, n - m):
        rows = slice(at, at + m)
        y = crop.forward(atb[:, rows, rows].contiguous(), mask[:, rows, rows].contiguous())
        keep = slice(0, m - edge) if at == 0 else slice(edge, m)
        a, b = x1[:, rows, rows][:, keep, keep], y[:, keep, keep]
        torch.cuda.synchronize()
        assert float(torch.linalg.norm(b - atb[:, rows, rows][:, keep, keep])) > 0
        assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    crop.close()
