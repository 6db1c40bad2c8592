"""An error is reported by the call it befell and by no other."""
import pytest

pytestmark = pytest.mark.gpu

GIB = 1 << 30


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


def test_an_error_is_reported_once(lib):
    """the calls after one that ran out of memory succeed"""
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    a = torch.randn((64, 64), dtype=torch.float64, device="cuda", generator=g)
    calls = [lambda: lib.dsrg_split_gemm(a, a, torch.zeros_like(a), 1.0, 6),
             lambda: lib.dsrg_df_ladder(a[None], a.reshape(8, 8, 8, 8), torch.empty_like(a).reshape(8, 8, 8, 8), 3),
             lambda: lib.dsrg_cholesky(a @ a.T, 1e-9, 70)]
    M, K = 16384, 8192  # a product whose digits (2.1 GB per operand) do not fit the 3 GiB left free
    row = torch.ones((1, M), dtype=torch.float64, device="cuda")
    A, B, C = row[:, :K].expand(M, K), row.expand(K, M), torch.zeros_like(row).expand(M, M)
    for f in calls:
        f()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 3 * GIB, dtype=torch.uint8, device="cuda")
    try:
        for f in calls:
            code = 0
            try:
                lib.dsrg_split_gemm(A, B, C, 1.0, 8)
            except lib.DsrgError as e:
                code = e.code
            assert code == lib.DSRG_ERR_OOM
            f()
    finally:
        del fill
        torch.cuda.empty_cache()
