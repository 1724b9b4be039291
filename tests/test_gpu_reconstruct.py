"""A_hat = U D V^T (eod_abe_reconstruct) on factor sets that a program fills
itself, FP64 below and above the size from which its products run on the
tensor cores (2^25 multiply-adds): odd sizes, a padded leading dimension, rank
1, and factors that hold NaN and infinities (those propagate as with FP64
FMAs).

Bound: FP64 dot products of length r, twice: |error| <= 2 (r + 2) u |U| |D| |V|^T
entry by entry for FP64 FMAs; the emulation's one rounding and 2^-63 of the
row x column scales per term lie below it on these operands, whose entries
along a row differ by less than 2^8."""
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


def _factors(m, n, r, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda a, b: (torch.rand(b, a, generator=g, device="cuda", dtype=torch.float64) + 0.01).t() * (
        1 - 2 * torch.randint(0, 2, (b, a), generator=g, device="cuda").t())
    return rnd(m, r), torch.triu(rnd(r, r)).t().contiguous().t(), rnd(n, r)


def _run(eod, U, D, V, ld):
    m, n, r = U.shape[0], V.shape[0], D.shape[0]
    f = eod.EodFactors(m=m, n=n, rank=r, precision=eod.EOD_PLAIN, f_dtype=eod.EOD_F64)
    f.U, f.D, f.V = U.data_ptr(), D.data_ptr(), V.data_ptr()
    out = torch.full((n, ld), -7.0, dtype=torch.float64, device="cuda")
    o = eod.make_opts(dtype=eod.EOD_F64)
    assert eod.eod_abe_reconstruct(ctypes.byref(f), ctypes.c_void_p(out.data_ptr()), ld, ctypes.byref(o)) == eod.EOD_OK
    torch.cuda.synchronize()
    assert torch.all(out[:, m:] == -7.0)      # the padding is not written
    return out.t()[:m]


@pytest.mark.parametrize("m,n,r,pad", [(65, 33, 1, 0), (300, 257, 40, 3), (641, 513, 129, 0), (1025, 777, 200, 5),
                                       (128, 4099, 65, 1), (2049, 130, 127, 0)])
def test_reconstruct_f64(eod, m, n, r, pad):
    U, D, V = _factors(m, n, r, m + r)
    got = _run(eod, U, D, V, m + pad)
    ref = U @ D @ V.t()
    # the reference's own error is within the same bound
    bound = 4 * (r + 2) * U64 * (U.abs() @ D.abs() @ V.abs().t())
    assert bool(((got - ref).abs() <= bound).all())


@pytest.mark.parametrize("where", ["U", "D", "V"])
def test_non_finite_factors_propagate(eod, where):
    m, n, r = 700, 600, 150
    U, D, V = _factors(m, n, r, 5)
    {"U": U, "D": D, "V": V}[where][3, 4] = float("nan") if where != "V" else float("inf")
    got = _run(eod, U, D, V, m)
    ref = (U @ D) @ V.t()
    assert bool(torch.equal(torch.isnan(got), torch.isnan(ref)))
    assert bool(torch.equal(torch.isinf(got), torch.isinf(ref)))
    ok = torch.isfinite(ref)
    assert not bool(ok.all())
    assert bool(torch.allclose(got[ok], ref[ok], rtol=1e-10, atol=1e-8))
