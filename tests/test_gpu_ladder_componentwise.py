"""dsrg_df_ladder element by element: a small L[p,q] beside a large L[q,p] has
an error of its own size.  With B[0] = diag(d) the ladder is L[p,q] = d_p d_q t[p,q],
each element one product of one term, so its error is a few roundings of
that element."""
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


@pytest.mark.parametrize("npart,nh,p0", [(2, 1, 0), (11, 2, 1), (33, 5, 0), (106, 3, 2), (150, 2, 0), (470, 1, 1)])
def test_graded_amplitudes(lib, npart, nh, p0):
    import torch
    n = npart + p0 + 1
    g = torch.Generator(device="cuda").manual_seed(n)
    d = 0.5 + torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
    B = torch.diag(d)[None].contiguous()
    t = 1.0 + torch.rand((npart, npart, nh, nh), dtype=torch.float64, device="cuda", generator=g)
    up = torch.triu(torch.ones((npart, npart), dtype=torch.float64, device="cuda"), 1)
    t = t * (1.0 + (1e-12 - 1.0) * up)[:, :, None, None]  # t[p,q], p < q, 12 orders below t[q,p]
    t[:, :, 0, nh - 1] *= 1e-9
    t = t.contiguous()
    L = torch.empty_like(t)
    lib.dsrg_df_ladder(B, t, L, p0)
    dd = d[p0:p0 + npart]
    ref = dd[:, None, None, None] * dd[None, :, None, None] * t
    # two products, one rounding each; the reference takes two of its own
    assert bool(((L - ref).abs() <= 4 * 2.0 ** -53 * ref.abs()).all())
