"""FP64 energies at sizes whose contractions take the narrow kernel (a short
side of 3 to 48, here 3, 5, 6, 8, 9, 32 and 50 beside, and a long one past
4864 that is no multiple of its 128-row blocks) and the element-wise kernels'
runs of 4, 2 and 1 elements (innermost extents 12, 10 and 5), against the
block-restricted oracle."""
import pytest

import synth
from oracle import dsrg_df

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


@pytest.mark.parametrize("shape", [(2, 3, 2, 47, 24), (4, 5, 4, 27, 30), (4, 6, 6, 24, 28), (6, 6, 6, 17, 20)], ids=str)
def test_fp64_energies_match_the_block_oracle(lib, shape):
    nc, na, nel, nv, naux = shape
    inst = synth.make_instance(nc, na, nel, nv, naux, 0.5, seed=sum(shape))
    ref = dsrg_df.dsrg_pt3(inst)
    h = lib.Dsrg(inst)
    try:
        e = h.pt3()
    finally:
        h.close()
    for k in ("e2", "e3a", "e3b", "e3"):
        assert abs(e[k] - ref[k]) < 1e-9 * max(1.0, abs(ref[k])), (k, e[k], ref[k])
