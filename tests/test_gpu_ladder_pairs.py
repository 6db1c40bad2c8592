"""The ladder in pair form (sums and differences over pairs p >= q, r >= s):
the general entry point for a B that is not symmetric in its last two
indices, at pair counts around its batches and at the smallest sizes, and the
energy's symmetric form against its batched form, which a small
DSRG_LADDER_BUDGET_MB selects (0.05 MB; 1 MB keeps the pair form in several
batches of rows)."""
import os

import numpy as np
import pytest

import synth

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


@pytest.mark.parametrize("n,naux,p0,npart,nh", [(1, 1, 0, 1, 1), (3, 2, 1, 2, 1), (12, 7, 1, 11, 2), (34, 19, 1, 33, 5),
                                                (64, 24, 0, 64, 3), (90, 16, 2, 87, 4)])
def test_general_ladder_unsymmetric_factor(lib, n, naux, p0, npart, nh):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n + naux)
    B = torch.randn((naux, n, n), dtype=torch.float64, device="cuda", generator=g)
    t = torch.randn((npart, npart, nh, nh), dtype=torch.float64, device="cuda", generator=g)
    L = torch.full_like(t, 7.0)
    lib.dsrg_df_ladder(B, t, L, p0)
    b = B[:, p0:p0 + npart, p0:p0 + npart]
    X = torch.einsum("Qqs,rsij->Qqrij", b, t)
    ref = torch.einsum("Qpr,Qqrij->pqij", b, X)
    # |G| |t| summed with every product and sum rounded once: K = naux + np^2 roundings at most
    A = torch.einsum("Qqs,rsij->Qqrij", b.abs(), t.abs())
    bound = torch.einsum("Qpr,Qqrij->pqij", b.abs(), A) * (naux + npart * npart + 8) * 2.0 ** -53
    assert bool(((L - ref).abs() <= 2 * bound).all())


@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("budget", ["0.05", "1"])
def test_pair_form_equals_batched_form(lib, split, budget):
    inst = synth.make_instance(2, 4, 4, 17, 40, 0.5, seed=11)
    kw = dict(precision=lib.DSRG_PREC_SPLIT, slices=7) if split else {}
    out = []
    for env in (None, budget):
        if env is not None:
            os.environ["DSRG_LADDER_BUDGET_MB"] = env
        try:
            h = lib.Dsrg(inst, **kw)
            try:
                h.pt3()
                out.append(h.fetch("O2"))
            finally:
                h.close()
        finally:
            os.environ.pop("DSRG_LADDER_BUDGET_MB", None)
    scale = np.abs(out[0]).max()
    # FP64: summation order; 7 slices: 2^-49 of the row and column maxima times K = 21^2
    assert np.abs(out[0] - out[1]).max() <= (1e-11 if split else 1e-12) * scale
