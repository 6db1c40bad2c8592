"""FP64 energies whose contractions take the narrow kernel (six CTAs per SM or
more) with 4, 6, 9, 11 and 13 columns, padded to 4, 6, 10, 12 and 14 of them,
over 4 to 13 k, against the block-restricted oracle."""
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


@pytest.mark.parametrize("shape", [(4, 5, 4, 45, 24), (5, 6, 6, 40, 20), (9, 4, 4, 44, 20)], ids=str)
def test_energies_match_the_block_oracle(lib, shape):
    nc, na, nel, nv, naux = shape
    inst = synth.make_instance(nc, na, nel, nv, naux, 0.5, seed=3)
    ref = dsrg_df.dsrg_pt3(inst)
    h = lib.Dsrg(inst)
    try:
        e = h.pt3()
    finally:
        h.close()
    for k in ("e2", "e3a", "e3b", "e3"):
        assert abs(e[k] - ref[k]) < 1e-9 * max(1.0, abs(ref[k])), (k, e[k], ref[k])
