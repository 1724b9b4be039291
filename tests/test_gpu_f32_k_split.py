"""The FP32 product on digits where its K is split over the SMs (fewer than 152
tiles of 128 x 64): exact integer sums, added in FP64 and rounded once to FP32,
through `eod_abe_reconstruct` with U, V of integers below 2^12 and D a diagonal
of powers of two."""
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


@pytest.mark.parametrize("m,n,r,pad", [(600, 600, 2112, 0), (257, 1000, 3001, 3), (1100, 1030, 700, 1)])
def test_split_sums_are_rounded_once(eod, m, n, r, pad):
    rng = np.random.default_rng(m)
    U, V = (rng.integers(-4095, 4096, (k, r)) for k in (m, n))
    d = 2 ** rng.integers(0, 6, r)
    Ud, Dd, Vd = (torch.from_numpy(np.asfortranarray(X)).cuda()
                  for X in (U.astype(np.float32), np.diag(d.astype(np.float64)), V.astype(np.float32)))
    f = eod.EodFactors(m=m, n=n, rank=r, precision=eod.EOD_PLAIN, f_dtype=eod.EOD_F32)
    f.U, f.D, f.V = Ud.data_ptr(), Dd.data_ptr(), Vd.data_ptr()
    out = torch.full((n, m + pad), -7.0, dtype=torch.float32, device="cuda")
    o = eod.make_opts(dtype=eod.EOD_F32)
    eod.eod_abe_debug_profile(1)
    st = eod.eod_abe_reconstruct(ctypes.byref(f), ctypes.c_void_p(out.data_ptr()), m + pad, ctypes.byref(o))
    emulated, fma = (eod.profile_read(k)["launches"] for k in (5, 7))
    eod.eod_abe_debug_profile(0)
    assert st == eod.EOD_OK and (emulated, fma) == (1, 1)   # A_hat; W alone by FMAs
    ref = ((U * d).astype(np.float64) @ V.T.astype(np.float64)).astype(np.float32)
    assert np.array_equal(out[:, :m].t().cpu().numpy(), ref)
    assert torch.all(out[:, m:] == -7.0)
