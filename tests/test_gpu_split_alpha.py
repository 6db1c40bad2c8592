"""C += alpha A B of the split product is one rounding of alpha (A B) + C where
A B is exact in the digits, whatever alpha: with C = -fl(alpha A B) the result is
the rounding error of that product, not zero."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_02011_gb300 import build
    build.build()
    import paper_1701_02011_gb300 as g
    g.load_library()
    return g


@pytest.mark.parametrize("M,N,K", [(130, 70, 40), (40, 30, 300), (4500, 28, 8), (28, 200, 700)])
@pytest.mark.parametrize("alpha", [1.0 / 3.0, -0.3, -0.5])
def test_one_rounding(lib, M, N, K, alpha):
    import torch
    rng = np.random.default_rng(M + K)
    A = rng.integers(-63, 64, (M, K)).astype(np.float64)
    B = rng.integers(-63, 64, (K, N)).astype(np.float64)
    t = A @ B  # integers below 2^53
    C0 = -(alpha * t)
    C = torch.from_numpy(C0).cuda()
    lib.dsrg_split_gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, alpha, 2)
    got = C.cpu().numpy()
    for m in range(0, M, max(1, M // 25)):
        for n in range(N):
            want = float(Fraction(alpha) * int(t[m, n]) + Fraction(C0[m, n]))
            assert got[m, n] == want, (m, n, got[m, n], want)
