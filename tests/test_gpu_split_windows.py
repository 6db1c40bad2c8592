"""The split product's exact windows, its one-pass packing and its write-back,
where they can go wrong: k on both sides of a 16-k stage, of the one-pass limit
(256) and of several windows; operands whose digits are all as large as they
get (windows as short as they get) and operands of a few large elements; every
orientation of contiguous rows or k; outputs of fewer rows or columns than a
warp; and factors alpha that are powers of two (folded into the exponent), not,
or zero."""
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


def check(lib, A, B, S, alpha=1.0, C0=None):
    import torch
    C = torch.zeros((A.shape[0], B.shape[1]), dtype=torch.float64, device="cuda") if C0 is None else C0.clone()
    lib.dsrg_split_gemm(A, B, C, alpha, S)
    # the reference in double-double: products and sums of halves are exact enough in 2 x 64 bits
    a, b = A.cpu().numpy().astype(np.longdouble), B.cpu().numpy().astype(np.longdouble)
    ref = a @ b * np.longdouble(alpha) + (0 if C0 is None else C0.cpu().numpy())
    bound = A.abs().amax(1)[:, None] * B.abs().amax(0)[None, :] * A.shape[1]
    err = np.abs(C.cpu().numpy() - ref)
    lim = tolerance(S) * abs(alpha) * bound.cpu().numpy() + 2.0 ** -51 * np.abs(ref) + A.shape[1] * 2.0 ** -52 * abs(
        alpha) * bound.cpu().numpy() * (np.finfo(np.longdouble).eps > 2.0 ** -60)
    assert (err <= lim.astype(np.float64)).all(), float((err / np.maximum(lim, 1e-300)).max())


@pytest.mark.parametrize("K", [1, 15, 16, 17, 31, 255, 256, 257, 1300])
@pytest.mark.parametrize("S", [6, 8])
def test_k_around_stages_and_the_one_pass_limit(lib, K, S):
    import torch
    g = torch.Generator(device="cuda").manual_seed(K)
    A = torch.randn((131, K), dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn((K, 70), dtype=torch.float64, device="cuda", generator=g)
    check(lib, A, B, S)


@pytest.mark.parametrize("S", [1, 5, 6, 7, 8])
@pytest.mark.parametrize("kind", ["full digits", "few large"])
def test_windows_of_extreme_digits(lib, S, kind):
    """Full digits: every element 1 - 2^-53 or its negative (the balanced digits
    of the grid's end) beside 64/127 (every digit 64 or its carry), over k of
    many of the shortest windows.  Few large: one element in a hundred, so
    that almost all digits vanish and a window is the whole k."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(S)
    shape = (150, 2100)
    if kind == "full digits":
        v = torch.tensor([64.0 / 127.0, -64.0 / 127.0, 63.5 / 127.0, 1.0 - 2.0 ** -53], dtype=torch.float64, device="cuda")
        A = v[torch.randint(0, 4, shape, device="cuda", generator=g)]
        B = v[torch.randint(0, 2, (shape[1], 90), device="cuda", generator=g)]
        A[:40] = 64.0 / 127.0
        B[:, :40] = 64.0 / 127.0
    else:
        A = torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
        A *= torch.rand(shape, device="cuda", generator=g) < 0.01
        B = torch.randn((shape[1], 90), dtype=torch.float64, device="cuda", generator=g)
    check(lib, A.contiguous(), B.contiguous(), S)


@pytest.mark.parametrize("M,N,K", [(5, 3, 40), (1, 200, 33), (4500, 28, 8), (28, 5000, 8), (129, 33, 64), (300, 8, 700)])
def test_narrow_outputs(lib, M, N, K):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn((M, K), dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn((K, N), dtype=torch.float64, device="cuda", generator=g)
    C0 = torch.randn((M, N), dtype=torch.float64, device="cuda", generator=g)
    check(lib, A, B, 7, -0.5, C0)


@pytest.mark.parametrize("alpha", [2.0 ** -40, -1.0, 0.3, -1.0 / 6.0, 0.0])
def test_alpha(lib, alpha):
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn((140, 90), dtype=torch.float64, device="cuda", generator=g) * 1e3
    B = torch.randn((90, 77), dtype=torch.float64, device="cuda", generator=g) * 1e-5
    C0 = torch.randn((140, 77), dtype=torch.float64, device="cuda", generator=g)
    check(lib, A, B, 6, alpha, C0)
    C = C0.clone()
    lib.dsrg_split_gemm(A, B, C, 0.0, 6)
    assert torch.equal(C, C0)
