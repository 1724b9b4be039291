"""The leaf factorisation over a cluster of CTAs (widths above 64; blocks of 32
columns, 8 columns at a time) against the one-CTA schedule with two barriers
per pivot (decide | 256) and LAPACK, at the edges of its blocks, and rank-test
stops inside each of them.

Bounds: a Cholesky factorisation's backward error, O(w u) ||G|| (Higham,
Accuracy and Stability, Thm 10.3: gamma_{w+1} |R^T| |R|, whose norm is at most
w gamma ||G||), taken as 20 w u ||G|| as for the one-CTA leaf."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


def _run(eod, G, decide=0, eps2=0.0, coef=0.0, rho=0.0, pad=0, shift=0.0):
    w = G.shape[0]
    Gd = torch.from_numpy(np.asfortranarray(np.vstack([G, np.full((pad, w), np.nan)]))).cuda()
    R = torch.full((w, w + pad), float("nan"), dtype=torch.float64, device="cuda").t()
    Ri = torch.full((w, w + pad), float("nan"), dtype=torch.float64, device="cuda").t()
    info = torch.zeros(2, dtype=torch.int32, device="cuda")
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    st = eod.eod_abe_debug_chol(P(Gd), w + pad, w, decide, eps2, coef, rho, shift, P(R), P(Ri), w + pad, P(info),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == eod.EOD_OK
    p, code = info.tolist()
    R, Ri = R.cpu().numpy(), Ri.cpu().numpy()
    assert np.all(np.isnan(R[w:])) and np.all(np.isnan(Ri[w:]))   # nothing beyond the block's rows
    return p, code, R[:p, :p], Ri[:p, :p]


def _spd(w, cond, seed):
    rng = np.random.default_rng(seed)
    Q, _ = np.linalg.qr(rng.standard_normal((w, w)))
    return (Q * np.geomspace(1.0, 1.0 / cond, w)) @ Q.T


@pytest.mark.parametrize("w", [65, 71, 72, 73, 95, 96, 97, 104, 121, 127, 128])
@pytest.mark.parametrize("cond,pad", [(1e2, 0), (1e8, 3)])
def test_block_leaf(eod, w, cond, pad):
    G = _spd(w, cond, w)
    p, code, R, Ri = _run(eod, G, pad=pad)
    assert (p, code) == (w, 0)
    assert np.array_equal(np.tril(R, -1), np.zeros((w, w))) and np.array_equal(np.tril(Ri, -1), np.zeros((w, w)))
    assert np.all(np.diag(R) > 0)
    assert np.linalg.norm(R.T @ R - G) <= 20 * w * U64 * np.linalg.norm(G)
    assert np.linalg.norm(Ri @ R - np.eye(w)) <= 50 * w * U64 * cond
    p2, code2, R2, _ = _run(eod, G, decide=256, pad=pad)
    assert (p2, code2) == (p, code)
    assert np.linalg.norm(R - R2) <= 50 * w * U64 * cond * np.linalg.norm(R2)


@pytest.mark.parametrize("stop", [0, 1, 7, 8, 9, 31, 32, 33, 40, 63, 64, 70, 96, 97])
def test_block_leaf_stops_at_the_same_column(eod, stop):
    """Column `stop` nearly dependent on the ones before it: its pivot falls
    below eps^2 and both schedules keep the same columns, their factor and its
    inverse."""
    w = 104
    rng = np.random.default_rng(stop)
    X = rng.standard_normal((300, w))
    X[:, stop] = (X[:, :stop] @ rng.standard_normal(stop) if stop else 0.0) + 1e-7 * rng.standard_normal(300)
    G = X.T @ X
    coef = 64.0 * (w + np.sqrt(300.0)) * U64
    for decide in (1, 257):
        p, code, R, Ri = _run(eod, G, decide=decide, eps2=1e-6, coef=coef, rho=1e-10)
        assert p == stop and code in (1, 2)
        if stop:
            assert np.linalg.norm(R.T @ R - G[:p, :p]) <= 20 * p * U64 * np.linalg.norm(G)
            assert np.linalg.norm(Ri @ R - np.eye(p)) <= 1e-9


def test_block_leaf_not_positive_and_shift(eod):
    G = _spd(100, 10.0, 7)
    p, code, R, _ = _run(eod, G, shift=0.5)
    assert (p, code) == (100, 0)
    assert np.linalg.norm(R.T @ R - (G + 0.5 * np.eye(100))) <= 20 * 100 * U64 * np.linalg.norm(G + 0.5 * np.eye(100))
    G[77, 77] = -1.0
    p, code, _, _ = _run(eod, G)
    assert code == 3 and p <= 77


@pytest.mark.parametrize("w", [17, 24, 25, 31, 32, 33, 39, 40, 41, 57, 63, 64])
@pytest.mark.parametrize("cond,pad", [(1e2, 0), (1e8, 3)])
def test_block_leaf_of_one_and_two_blocks(eod, w, cond, pad):
    """Widths of one or two blocks, whole and ragged, with the same bounds."""
    test_block_leaf(eod, w, cond, pad)


@pytest.mark.parametrize("w,stop", [(24, 0), (24, 8), (32, 15), (32, 31), (40, 33), (64, 20), (64, 32), (64, 63)])
def test_narrow_block_leaf_stops_at_the_same_column(eod, w, stop):
    rng = np.random.default_rng(100 * w + stop)
    X = rng.standard_normal((300, w))
    X[:, stop] = (X[:, :stop] @ rng.standard_normal(stop) if stop else 0.0) + 1e-7 * rng.standard_normal(300)
    G = X.T @ X
    coef = 64.0 * (w + np.sqrt(300.0)) * U64
    for decide in (1, 257):
        p, code, R, Ri = _run(eod, G, decide=decide, eps2=1e-6, coef=coef, rho=1e-10)
        assert p == stop and code in (1, 2)
        if stop:
            assert np.linalg.norm(R.T @ R - G[:p, :p]) <= 20 * p * U64 * np.linalg.norm(G)
            assert np.linalg.norm(Ri @ R - np.eye(p)) <= 1e-9
