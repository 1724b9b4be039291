"""Alg. 2 steps 9-11 against their definition in 64 bits, from the call's own
Q and C: C^T = V R, R^T = Qh D, U = Q Qh (diagonals positive), for ranks at the
edges of the leaf that runs on one CTA (16) and of the one that takes a whole
factor (128).

Bounds: an entry's perturbation of a QR factorisation by rounding u in the data's
precision, at most 20 r u cond(C) relative to the factor (Stewart 1977), with
cond(C) <= 1e2 here."""
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


def _qr(X):
    Q, R = torch.linalg.qr(X)
    s = torch.where(torch.diagonal(R) < 0, -1.0, 1.0).to(X.dtype)
    return Q * s, R * s.unsqueeze(1)


@pytest.mark.parametrize("r", [1, 2, 3, 15, 16, 17, 128, 129])
@pytest.mark.parametrize("form", ["f64", "f32"])
def test_core_factors(eod, r, form):
    w = W.exact_rank(m=700, n=301, r=r, seed=r)
    A = torch.from_numpy(np.asfortranarray(w.A.astype(np.float64 if form == "f64" else np.float32))).cuda()
    f = eod.factor(A, 1e-4, 5, tol_mode="rel", block_k=48)
    assert f.rank == r
    V, R = _qr(f.Ct.double())
    Qh, D = _qr(R.t())
    s = torch.linalg.svdvals(f.Ct.double())
    u = 2.0 ** -53 if form == "f64" else 2.0 ** -24
    bound = 20 * r * u * float(s[0] / s[-1])
    for got, ref in ((f.V, V), (f.D, D), (f.U, f.Q.double() @ Qh)):
        assert float((got.double() - ref).norm()) <= bound * float(ref.norm())
