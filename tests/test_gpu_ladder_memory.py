"""The energy's ladder where the matrix of (pr|qs) over pairs does not fit the
device: the energy runs in batches of rows instead, with the result that a
budget too small for the matrix (DSRG_LADDER_BUDGET_MB) gives, alone and as one
of several in dsrg_pt3_batch; and handles at rest keep one matrix between them,
not one each."""
import os

import pytest

import synth

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


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


class Batched:
    """(pr|qs) in batches within 1 GiB (or as much as is said)"""

    def __init__(self, mb=1024):
        self.mb = mb

    def __enter__(self):
        os.environ["DSRG_LADDER_BUDGET_MB"] = str(self.mb)

    def __exit__(self, *a):
        os.environ.pop("DSRG_LADDER_BUDGET_MB", None)


class Filled:
    """Device memory taken so that `leave` bytes stay free."""

    def __init__(self, leave):
        import torch
        self.t = torch.empty(_free() - leave, dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *a):
        self.t = None
        _free()


def _instance(nv):
    return synth.make_instance(2, 2, 2, nv, 40, 0.5, seed=7)


def test_energy_falls_back_to_batches(lib):
    inst = _instance(158)  # the matrix of 160 particles: 1.33 GB
    with Batched():
        h = lib.Dsrg(inst)
        e, peak = h.pt3(), lib.dsrg_peak_bytes(h.h)
        h.close()
    with Filled(peak + GIB // 2):
        h = lib.Dsrg(inst)
        try:
            assert h.pt3() == e
            assert h.pt3() == e
        finally:
            h.close()


def test_batch_falls_back_to_batches(lib):
    insts = [_instance(nv) for nv in (158, 160, 163)]
    with Batched():
        before = _free()
        hs = [lib.Dsrg(i) for i in insts]
        e = lib.dsrg_pt3_batch(hs)
        used = before - _free()
        for h in hs:
            h.close()
    with Filled(used + GIB // 2):
        hs = [lib.Dsrg(i) for i in insts]
        try:
            assert lib.dsrg_pt3_batch(hs) == e
            assert lib.dsrg_pt3_batch(hs) == e
            hs[1].load(insts[1])
            assert lib.dsrg_pt3_batch(hs) == e
        finally:
            for h in hs:
                h.close()


def test_idle_handles_keep_one_matrix_between_them(lib):
    insts = [_instance(nv) for nv in (198, 196, 194)]  # matrices of 3.2 GB and less
    lib.Dsrg(insts[0]).close()
    used = []
    for batched in (True, False):
        before = _free()
        hs = []
        for i in insts:
            hs.append(lib.Dsrg(i))
            if batched:
                with Batched():
                    hs[-1].pt3()
            else:
                hs[-1].pt3()
        used.append(before - _free())
        for h in hs:
            h.close()
        assert before - _free() <= GIB + (64 << 20)
    assert used[1] <= used[0] + 3230 * 10 ** 6 + GIB + (256 << 20)


def test_capture_without_the_blocks_of_earlier_calls(lib):
    """An energy in batches of 4 GiB leaves a block that batches of 1 GiB do not
    use; with half a GiB free the capture fits only without it."""
    inst = _instance(216)  # 218 particles: the matrix would take 4.5 GB
    with Batched():
        h = lib.Dsrg(inst)
        e = h.pt3()
        h.close()
    with Batched(4096):
        h = lib.Dsrg(inst)
        h.pt3()
    try:
        with Filled(GIB // 2), Batched():
            assert lib.dsrg_pt3_batch([h]) == [e]
            assert lib.dsrg_pt3_batch([h]) == [e]
    finally:
        h.close()
