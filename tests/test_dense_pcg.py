"""The dense PCG kernel's register form: the edges of its vector lengths, and
problems scaled out of the range in which its inner products are summed in
compensated FP32.

With x -> s x, b -> s b, eps -> s^2 eps and lambda -> s lambda the iteration
scales by s, and for a power of two every operation scales exactly; what may
differ is the last bits of the inner products, so of alpha and beta (6e-8 each)
over 2 x 4 PCG steps from a system of condition below 1e2: 1e-5 of the
solution's norm."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1411_5057_gb300 as F
    return F


@pytest.mark.parametrize("N", [4, 100, 2048, 2052, 4096, 4100, 8192])
@pytest.mark.parametrize("shared", [False, True])
def test_scaled_problem_scales(F, N, shared):
    M, P = 24, 2
    rng = np.random.default_rng(N)
    A = rng.standard_normal((1 if shared else P, M, N)) / math.sqrt(N)
    ctx = F.DenseContext(M, N, P, shared=shared)
    ctx.set_matrix(torch.from_numpy((A[0] if shared else A).astype(np.float32)).cuda())
    b = torch.from_numpy(rng.standard_normal((P, M)).astype(np.float32)).cuda()

    def solve(s):
        x = ctx.solve(b * s, F.make_params(2, 4, lam=0.05 * s, eps=1e-2 * s * s))
        return (x / s).cpu().numpy().astype(np.float64)

    ref = solve(1.0)
    assert np.linalg.norm(ref) > 0
    for s in (2.0 ** -50, 2.0 ** 50):
        got = solve(s)
        assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref), (s, np.linalg.norm(got - ref))
