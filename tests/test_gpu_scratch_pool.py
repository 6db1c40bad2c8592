"""The scratch of the calls without a handle: the library's memory pool keeps
at most 1 GiB once a call has returned, whether the call succeeded or ran out
of device memory, and a later call gets what an earlier failed one had taken."""
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


def _free(torch):
    return torch.cuda.mem_get_info()[0]


def test_a_large_call_leaves_at_most_a_gib(lib):
    import torch
    n = 9216  # 8 slices: 1.4 GB of digits per operand
    A = torch.ones((1, n), dtype=torch.float64, device="cuda").expand(n, n)
    C = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    lib.dsrg_split_gemm(A[:256], A, C[:256], 1.0, 8)
    torch.cuda.synchronize()
    before = _free(torch)
    lib.dsrg_split_gemm(A, A, C, 1.0, 8)
    assert before - _free(torch) <= GIB + (64 << 20)
    assert bool((C[256:] == n).all()) and bool((C[:256] == 2 * n).all())


def test_out_of_memory_gives_back_what_was_taken(lib):
    import torch
    M, K = 16384, 8192  # 2.1 GB of digits per operand, 3 GiB left free
    row = torch.ones((1, M), dtype=torch.float64, device="cuda")
    A, B, C = row[:, :K].expand(M, K), row.expand(K, M), torch.zeros_like(row).expand(M, M)
    a = torch.ones((1, 4096), dtype=torch.float64, device="cuda").expand(4096, 4096)
    c = torch.zeros((4096, 4096), dtype=torch.float64, device="cuda")
    lib.dsrg_split_gemm(a[:128], a, c[:128], 1.0, 8)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(_free(torch) - 3 * GIB, dtype=torch.uint8, device="cuda")
    try:
        before = _free(torch)
        for _ in range(3):
            code = 0
            try:
                lib.dsrg_split_gemm(A, B, C, 1.0, 8)
            except lib.DsrgError as e:
                code = e.code
            assert code == lib.DSRG_ERR_OOM
            torch.cuda.synchronize()  # the pool gives back at a synchronisation
            assert before - _free(torch) <= GIB + (64 << 20)
        lib.dsrg_split_gemm(a, a, c, 1.0, 8)
        assert bool((c[128:] == 4096).all())
    finally:
        del fill
        torch.cuda.empty_cache()


@pytest.mark.parametrize("small_call_after", [False, True])
@pytest.mark.parametrize("own_stream", [False, True])
def test_a_handle_gets_what_the_pool_keeps(lib, own_stream, small_call_after):
    """0.5 GB of scratch per operand stay in the pool, 0.2 GB are free, and a
    handle's inputs take 0.42 GB; nothing synchronises in between."""
    import numpy as np
    import synth
    import torch
    inst = synth.make_instance(1, 2, 2, 717, 4, 0.5, seed=1)
    inst["naux"], inst["B"] = 100, np.zeros((100, 720, 720))
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() if isinstance(v, np.ndarray) else v for k, v in inst.items()}
    n = 5600
    A = torch.ones((1, n), dtype=torch.float64, device="cuda").expand(n, n)
    C = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    st = [torch.cuda.Stream().cuda_stream if own_stream else None for _ in range(2)]
    lib.dsrg_split_gemm(A, A, C, 1.0, 8, st[0])
    if small_call_after:
        lib.dsrg_split_gemm(A[:64, :64], A[:64, :64], C[:64, :64], 1.0, 6, st[1])
    fill = torch.empty(_free(torch) - (200 << 20), dtype=torch.uint8, device="cuda")
    try:
        lib.Dsrg(dev).close()
    finally:
        del fill
        torch.cuda.empty_cache()
