"""The dense PCG kernel's inner products against exact ones, through one PCG step
whose other operations are reproduced here in FP32: the relative change of the step
is |alpha d| / |x0| with alpha = <d, d> / <d, A^T A d> rounded to FP32.

The kernel's sums carry three floats (72 bits), so they are as good as exact in FP64:
what is left is alpha's division, a square root and a division in FP64, 3 x 1.1e-16;
1e-14 stands for them.  A sum that loses the low halves of its products is 1e-10 and
more off, and with data that cancel alpha's FP32 value changes."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def exact_dot(a, b):  # products of two floats are exact in FP64, fsum rounds once
    return math.fsum((a.astype(np.float64) * b.astype(np.float64)).tolist())


def well_conditioned(N, rng):
    A = np.eye(N, dtype=np.float32)
    return A, rng.standard_normal(N).astype(np.float32), rng.standard_normal(N).astype(np.float32)


def cancelling(N, rng):
    """2 x 2 blocks [[1, 1], [0, 2^-13]] and d = (u, -u + small): in <d, A^T A d> =
    sum (d1 + d2)^2 + 2^-26 d2^2 the products d_i q_i of a pair cancel to 1e-3 and less."""
    A = np.zeros((N, N), np.float32)
    k = np.arange(0, N, 2)
    A[k, k] = A[k, k + 1] = 1.0
    A[k + 1, k + 1] = 2.0 ** -13
    grid = 2.0 ** -22
    b1 = rng.integers(2 ** 22, 2 ** 23, N // 2) * grid  # [1, 2)
    small = rng.integers(1, 2 ** 10, N // 2) * grid
    x0 = np.zeros(N)
    x0[1::2] = 0.5
    b = np.empty(N)
    b[0::2] = b1
    b[1::2] = ((1.0 - b1 + small) - b1) * 2.0 ** 13  # A^T b = (b1, 1 - b1 + small)
    assert np.array_equal(b, b.astype(np.float32))
    return A, b.astype(np.float32), x0.astype(np.float32)


@pytest.mark.parametrize("N", [64, 1024, 4096])
@pytest.mark.parametrize("data", [well_conditioned, cancelling])
def test_one_step_against_exact_products(N, data):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    A, b, x0 = data(N, np.random.default_rng(N))
    ctx = F.DenseContext(N, N, 1)
    ctx.set_matrix(torch.from_numpy(A).cuda())

    def AtA(v):
        out = torch.empty(1, N, dtype=torch.float32, device="cuda")
        ctx.apply_AtA(torch.from_numpy(v).cuda()[None].contiguous(), out)
        torch.cuda.synchronize()
        return out[0].cpu().numpy()

    atb = (A.astype(np.float64).T @ b.astype(np.float64)).astype(np.float32)
    d = (atb - AtA(x0)).astype(np.float32)
    q = AtA(d)
    dq = exact_dot(d, q)
    assert dq > 0
    if data is cancelling:
        assert math.fsum(np.abs(d.astype(np.float64) * q).tolist()) > 500 * dq
    alpha = np.float32(exact_dot(d, d) / dq)
    dx = (alpha * d).astype(np.float32)
    want = math.sqrt(exact_dot(dx, dx) / exact_dot(x0, x0))
    _, st = ctx.solve(torch.from_numpy(b).cuda()[None].contiguous(), F.make_params(1, 1, lam=0.0, precond="none"),
                      x0=torch.from_numpy(x0).cuda()[None].contiguous(), stats=True)
    assert st["max_rel_change"] == pytest.approx(want, rel=1e-14)
    ctx.close()
