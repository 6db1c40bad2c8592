"""The split product where a CTA takes several tiles and a tile several exact
windows: outputs of more than 152 tiles at both tile widths without a k split,
at slice counts with one and with two sets of accumulators, and operands whose
digits are all 63 (2 * 0.(63)(63)... in base 128: the level sums of rows and
columns of one sign come to 0.98 or more of the 2^24 up to which they are exact).
k = 2100 is 132 stages; a window of those digits is 37 stages at 8 slices, 52 at
5, 66 at 4 and 88 at 3, all of k at 1 and 2."""
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


def tolerance(S):
    """|error| over K max|A row| max|B column|: the operands are rounded to
    2^(1 - 7 S) of their maxima (4 units of 2^(-7 S) over both), the digit
    pairs beyond level S + 1 left out add 4 (S - 1) 128/127 more, and the
    result is rounded once."""
    return 2.0 ** (-7 * S) * (4 + 4.04 * (S - 1)) + 2.0 ** -52


# 64-column tiles: 21 x 24; 32-column tiles: 305 x 1 (and, the long side along the columns, 1 x 305)
@pytest.mark.parametrize("M,N", [(2563, 1497), (38921, 29), (23, 38921)])
@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 8])
def test_many_tiles_of_many_windows(lib, M, N, S):
    import torch
    K = 2100
    g = torch.Generator(device="cuda").manual_seed(S + N)
    v = sum(126.0 * 128.0 ** -t for t in range(1, min(S, 7) + 1))  # 7 digits are 49 bits

    def operand(rows):
        x = torch.where(torch.rand((rows, K), device="cuda", generator=g) < 0.5, -v, v).double()
        x[: rows // 3] = v
        x[rows // 3: rows // 2] *= torch.exp2(torch.randint(-3, 1, (rows // 2 - rows // 3, K), device="cuda", generator=g).double())
        x[rows - rows // 5:] = torch.randn((rows // 5, K), dtype=torch.float64, device="cuda", generator=g)
        return x

    A, B = operand(M), operand(N).T.contiguous()
    C0 = torch.randn((M, N), dtype=torch.float64, device="cuda", generator=g)
    C = C0.clone()
    lib.dsrg_split_gemm(A, B, C, -0.5, S)
    ma, mb = A.abs().amax(1), B.abs().amax(0)
    bound = K * ma[:, None] * mb[None, :]
    # every element against FP64, whose own sum of K products is off by up to K 2^-53 of the bound
    ref = C0 - 0.5 * (A @ B)
    assert bool(((C - ref).abs() <= (0.5 * tolerance(S) + (K + 2) * 2.0 ** -53) * bound + 2.0 ** -52 * ref.abs()).all())
    # and rows and columns of every tile against more than 64 bits
    ms, ns = range(3, M, max(1, M // 40)), range(1, N, max(1, N // 40))
    a, b = A[list(ms)].cpu().numpy().astype(np.longdouble), B[:, list(ns)].cpu().numpy().astype(np.longdouble)
    want = C0[list(ms)][:, list(ns)].cpu().numpy() - np.longdouble(0.5) * (a @ b)
    got = C[list(ms)][:, list(ns)].cpu().numpy()
    lim = 0.5 * tolerance(S) * bound[list(ms)][:, list(ns)].cpu().numpy() + 2.0 ** -51 * np.abs(want).astype(np.float64)
    if np.finfo(np.longdouble).eps > 2.0 ** -60:
        lim = lim + K * 2.0 ** -52 * bound[list(ms)][:, list(ns)].cpu().numpy()
    assert (np.abs(got - want) <= lim).all(), float((np.abs(got - want) / lim).max())
