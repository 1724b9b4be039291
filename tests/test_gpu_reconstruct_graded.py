"""A_hat = U D V^T entry by entry where the terms of an entry differ much in size,
at sizes whose products run on the tensor cores: D graded over 2^40, V or U the
identity, rows of V that are zero against the large columns.  The bound is that
of FMA products for every entry, 2 (r + 2) u |U| |D| |V|^T, the reference's own on
top.  The digits alone are accurate to row scale x column scale; such factors
have to take the FMA kernels, dense ones need not."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

F64, F32 = torch.float64, torch.float32
SIMT = {F64: 0, F32: 7}   # the profile counters' kinds


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


def _factors(kind, m, n, r, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda a, b: torch.randn(b, a, generator=g, device="cuda", dtype=F64).t()
    U, V = rnd(m, r) / m ** 0.5, rnd(n, r) / n ** 0.5
    at = torch.arange(r, device="cuda", dtype=F64)
    D = torch.diag(1.0 / (1.0 + at)) if kind == "dense" else torch.diag(2.0 ** (40.0 * (1.0 - at / r)).round())
    D = D + 0.01 * torch.triu(rnd(r, r), 1) * torch.diagonal(D)
    if kind == "v_identity":
        V = torch.eye(n, r, device="cuda", dtype=F64)
    elif kind == "u_identity":
        U = torch.eye(m, r, device="cuda", dtype=F64)
    elif kind == "v_zeros":
        V[::3, : r // 2] = 0.0
    elif kind == "w_zero":     # a row of W that cancels, and rows of zeros
        U[5] = 0.0
        V[7] = 0.0
        D[:, 1:] = 0.0
        D[0, 0] = 0.0
    return U, D, V


@pytest.mark.parametrize("kind", ["dense", "v_identity", "u_identity", "v_zeros", "w_zero"])
@pytest.mark.parametrize("m,n,r,dtype", [(700, 401, 390, F64), (2049, 130, 129, F64), (1500, 811, 805, F32)])
def test_every_entry(eod, kind, m, n, r, dtype):
    U, D, V = _factors(kind, m, n, r, m)
    U, V = (X.to(dtype).t().contiguous().t() for X in (U, V))
    D = D.to(dtype).double().t().contiguous().t()
    f = eod.EodFactors(m=m, n=n, rank=r, precision=eod.EOD_PLAIN, f_dtype=eod.EOD_F64 if dtype == F64 else eod.EOD_F32)
    f.U, f.D, f.V = U.data_ptr(), D.data_ptr(), V.data_ptr()
    out = torch.full((n, m), 3.0, dtype=dtype, device="cuda").t()
    o = eod.make_opts(dtype=f.f_dtype)
    eod.eod_abe_debug_profile(1)
    st = eod.eod_abe_reconstruct(ctypes.byref(f), ctypes.c_void_p(out.data_ptr()), m, ctypes.byref(o))
    fma = eod.profile_read(SIMT[dtype])["launches"]
    eod.eod_abe_debug_profile(0)
    assert st == eod.EOD_OK
    U, V = U.double(), V.double()
    size = U.abs() @ D.abs() @ V.abs().t()
    u = 2.0 ** -53 if dtype == F64 else 2.0 ** -24
    assert bool(((out.double() - U @ D @ V.t()).abs() <= 4 * (r + 2) * u * size).all())
    if kind == "dense":   # W alone in FP32
        assert fma == (0 if dtype == F64 else 1)
