"""The pivot reciprocal of the cluster leaf (widths from 17) against CUDA's
division, seen through the leaf: for 2 x 2 blocks [d u; u 1] along the diagonal
with u a power of two so small that 1 - u^2 / d rounds to 1, the inverse factor's
entry is -u / d to the reciprocal's own rounding.  Within 2 ulp, as the one-CTA
leaf's; and a subnormal pivot ends the factorisation behind it."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


def _leaf(eod, G):
    w = G.shape[0]
    Gd = torch.from_numpy(np.asfortranarray(G)).cuda()
    R, Ri = (torch.zeros(w, w, dtype=torch.float64, device="cuda").t() for _ in range(2))
    info = torch.zeros(2, dtype=torch.int32, device="cuda")
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    assert eod.eod_abe_debug_chol(P(Gd), w, w, 0, 0.0, 0.0, 0.0, 0.0, P(R), P(Ri), w, P(info), None) == eod.EOD_OK
    return info.tolist(), Ri.cpu().numpy()


@pytest.mark.parametrize("w", [18, 64, 128])
def test_reciprocals(eod, w):
    rng = np.random.default_rng(w)
    worst = 0.0
    for _ in range(2 * 2042 // w):
        e = rng.integers(-1021, 1021, w // 2)
        m = rng.uniform(1.0, 2.0, w // 2)
        m[:3] = 1.0, 1.5, np.nextafter(2.0, 0.0)
        d, u = np.ldexp(m, e), np.ldexp(1.0, (e - 57) // 2)
        G = np.eye(w)
        i = 2 * np.arange(w // 2)
        G[i, i] = d
        G[i, i + 1] = G[i + 1, i] = u
        (p, code), Ri = _leaf(eod, G)
        assert (p, code) == (w, 0)
        r, ref = -Ri[i, i + 1] / u, 1.0 / d
        worst = max(worst, float((np.abs(r - ref) / np.spacing(ref)).max()))
    assert worst <= 2.0


@pytest.mark.parametrize("w", [16, 17, 64])
def test_subnormal_pivot(eod, w):
    G = np.eye(w)
    G[5, 5] = 2.0 ** -1030
    (p, code), _ = _leaf(eod, G)
    assert (p, code) == (6, 3)   # not positive (or not finite) behind it
