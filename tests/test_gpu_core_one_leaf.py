"""Alg. 2 steps 9-10 with one leaf per CholQR pass (ranks up to 128) against
the blocked form (the tuned key core_leaf at 16), which they replace: same
rank, the same basis Q bit for bit, U, D, V and Q C equal up to rounding, for
ranks at the leaf's edges, FP64, FP32 and mixed, and an A^T Q too
ill-conditioned for an unshifted Cholesky, which both hand to the shifted
passes.

Bounds: the two forms differ by the rounding of FP64 Cholesky factors of the
same Grams, u64 cond(G) relative, and (FP32 data) of FP32 products, u32 times
the condition of C; the matrices have cond(C) <= 1e2."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


def _factors(eod, A, tol, **kw):
    f = eod.factor(A, tol, 5, **kw)
    out = {"rank": f.rank, "Q": f.Q.clone(), "U": f.U.clone().double(), "D": f.D.clone(), "V": f.V.clone().double(),
           "tdiag": list(f.tdiag), "err": f.rel_err}
    f.close()
    return out


def _both(eod, tmp_path, A, tol, **kw):
    path = tmp_path / "t.txt"
    path.write_text("core_leaf 1 1000000 0 0 0 0 16\n")
    got = _factors(eod, A, tol, **kw)
    assert eod.eod_abe_tuning_load(str(path).encode()) == eod.EOD_OK
    try:
        ref = _factors(eod, A, tol, **kw)
    finally:
        eod.eod_abe_tuning_load(None)
    return got, ref


@pytest.mark.parametrize("r", [1, 2, 17, 63, 64, 65, 100, 127, 128])
@pytest.mark.parametrize("form,bound", [("f64", 1e-9), ("f32", 1e-3), ("mixed", 1e-3)])
def test_one_leaf_core_matches_the_blocked_form(eod, tmp_path, r, form, bound):
    w = W.exact_rank(m=1040, n=301, r=r, seed=r)
    A = torch.from_numpy(np.asfortranarray(w.A.astype(np.float64 if form == "f64" else np.float32))).cuda()
    kw = {"precision": "mixed" if form == "mixed" else "plain", "block_k": 48, "tol_mode": "rel"}
    got, ref = _both(eod, tmp_path, A, 1e-4, **kw)
    assert got["rank"] == ref["rank"] == r
    assert torch.equal(got["Q"], ref["Q"]) and got["tdiag"] == ref["tdiag"]
    assert got["err"] == ref["err"]
    assert bool(torch.equal(torch.triu(got["D"]), got["D"])) and bool((torch.diagonal(got["D"]) > 0).all())
    for k in ("U", "V", "D"):
        assert torch.linalg.norm(got[k] - ref[k]).item() <= bound * torch.linalg.norm(ref[k]).item(), k
    eye = torch.eye(r, dtype=torch.float64, device="cuda")
    tol = 1e-12 if form == "f64" else 1e-4
    assert (got["U"].t() @ got["U"] - eye).abs().max().item() <= tol
    assert (got["V"].t() @ got["V"] - eye).abs().max().item() <= tol


def test_ill_conditioned_core_takes_the_shifted_passes(eod, tmp_path):
    """sigma from 1 to 1e-12 with eps = 1e-13: the Gram of A^T Q has condition
    1e24, beyond an FP64 Cholesky."""
    rng = np.random.default_rng(2)
    A = torch.from_numpy(W.low_rank(rng, 400, 300, np.geomspace(1.0, 1e-12, 60))).cuda()
    got, ref = _both(eod, tmp_path, A, 1e-13, block_k=32)
    assert got["rank"] == ref["rank"]
    assert torch.equal(got["Q"], ref["Q"])
    Ag, Ar = (x["U"] @ x["D"] @ x["V"].t() for x in (got, ref))
    assert torch.linalg.norm(Ag - A).item() <= 1e-11 and torch.linalg.norm(Ag - Ar).item() <= 1e-11
    eye = torch.eye(got["rank"], dtype=torch.float64, device="cuda")
    assert (got["V"].t() @ got["V"] - eye).abs().max().item() <= 1e-10
