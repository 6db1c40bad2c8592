"""dsrg_cholesky at each CTA size that its rule picks (96 to 256 rows), on both
sides of the sizes where one CTA per SM becomes two and with a ragged last CTA,
bit for bit against the same operations done one by one."""
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


@pytest.mark.parametrize("N", [95, 14592, 14593, 19457, 24321, 29185, 34049, 38911, 38913, 46001])
def test_vectors_and_pivots(lib, N):
    import torch
    most = 19
    g = torch.Generator(device="cuda").manual_seed(N)
    X = torch.randn((most + 3, N), dtype=torch.float64, device="cuda", generator=g)
    V = X.T @ X
    V = torch.tril(V) + torch.tril(V, -1).T
    B, piv = lib.dsrg_cholesky(V, 0.0, most)
    D, ref, want = V.diagonal().clone(), [], []
    for q in range(most):
        J = int(torch.nonzero(D == D.max())[0])  # the smallest index on ties
        acc = torch.zeros(N, dtype=torch.float64, device="cuda")
        for b in ref:
            p = b * b[J]
            acc = acc + p
        L = (V[J] - acc) / torch.sqrt(D[J])
        s = L * L
        D = D - s
        ref.append(L)
        want.append(J)
    assert piv.tolist() == want
    assert torch.equal(B, torch.stack(ref))
