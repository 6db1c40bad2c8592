"""A batch that fails after some of its handles have been captured leaves those
handles usable: whatever they compute next equals a fresh handle's result.
The small zeroed tensors of a handle come out of arenas cleared as a whole;
an arena opened inside a capture is cleared by the graph alone, which a
failed batch never launches."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

KEYS = ("e2", "e3a", "e3b", "e3")


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


def _failed_batch(lib, h):
    """A batch of h, captured first, and a handle whose bounded waits run out."""
    bad = lib.Dsrg(synth.make_instance(2, 4, 4, 30, 120, 0.5, seed=5), precision=lib.DSRG_PREC_SPLIT, slices=6,
                   wait_limit=1)
    try:
        with pytest.raises(lib.DsrgError) as ex:
            lib.dsrg_pt3_batch([h, bad])
        assert ex.value.code == lib.DSRG_ERR_TIMEOUT
    finally:
        bad.close()


def _used_handle(lib, inst):
    h = lib.Dsrg(inst)
    e = h.pt3()
    for _ in range(400):  # small zeroed tensors, written and given back: the arenas' memory holds old values
        h.fetch("T1")
    assert h.pt3() == e
    return h


def test_load_after_a_failed_batch(lib):
    a, b = (synth.make_instance(2, 4, 4, 12, 60, 0.5, seed=s) for s in (31, 32))
    b["f1"] = (lambda x: 0.01 * (x + x.T))(np.random.default_rng(3).standard_normal((18, 18)))
    ref = lib.Dsrg(b)
    h = _used_handle(lib, a)
    try:
        _failed_batch(lib, h)
        h.load(b)
        want, got = ref.pt3(), h.pt3()
        for k in KEYS:
            assert got[k] == want[k], (k, got[k], want[k])
        assert h.relaxed(2, 2) == ref.relaxed(2, 2)
    finally:
        h.close()
        ref.close()


def test_dyall_after_a_failed_batch(lib):
    inst = synth.make_instance(2, 4, 4, 7, 40, 0.5, seed=33)
    ref = lib.Dsrg(inst)
    h = _used_handle(lib, inst)
    try:
        want = ref.dyall_aavv(1e-12, 300)
        for _ in range(2):
            _failed_batch(lib, h)
            got = h.dyall_aavv(1e-12, 300)
            assert got["converged"] == want["converged"] and got["iterations"] == want["iterations"]
            assert np.array_equal(h.fetch("Taavv"), ref.fetch("Taavv"))
        assert lib.dsrg_pt3_batch([h]) == lib.dsrg_pt3_batch([ref])
    finally:
        h.close()
        ref.close()
