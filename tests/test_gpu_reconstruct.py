"""A_hat = U D V^T (eod_abe_reconstruct) on factor sets that a program fills
itself: FP32 integers, whose product has to be rounded once where it runs on
the tensor cores (narrowest side 256, K above 256, 2^29.5 multiply-adds), and FP64 below and above the size from which its products run on the
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
    dt = eod.EOD_F64 if U.dtype == torch.float64 else eod.EOD_F32
    f = eod.EodFactors(m=m, n=n, rank=r, precision=eod.EOD_PLAIN, f_dtype=dt)
    f.U, f.D, f.V = U.data_ptr(), D.data_ptr(), V.data_ptr()
    out = torch.full((n, ld), -7.0, dtype=U.dtype, device="cuda")
    o = eod.make_opts(dtype=dt)
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


@pytest.mark.parametrize("m,n,r,pad", [(300, 8500, 300, 1), (1281, 1153, 515, 0), (257, 11600, 257, 3),
                                       (5003, 300, 511, 0)])
def test_reconstruct_f32_integers_are_rounded_once(eod, m, n, r, pad):
    """U, V of integers below 2^12, D a diagonal of powers of two: the exact
    sums (below 2^40) rounded to FP32."""
    rng = np.random.default_rng(m)
    U, V = (rng.integers(-4095, 4096, (k, r)) for k in (m, n))
    d = 2 ** rng.integers(0, 6, r)
    col = lambda X: torch.from_numpy(np.asfortranarray(X)).cuda()
    got = _run(eod, col(U.astype(np.float32)), col(np.diag(d.astype(np.float64))), col(V.astype(np.float32)), m + pad)
    ref = ((U * d).astype(np.float64) @ V.T.astype(np.float64)).astype(np.float32)
    assert np.array_equal(got.cpu().numpy(), ref)


@pytest.mark.parametrize("where", ["U", "D", "V"])
@pytest.mark.parametrize("m,n,r,dtype", [(700, 600, 150, torch.float64), (1400, 1300, 500, torch.float32)])
def test_non_finite_factors_propagate(eod, where, m, n, r, dtype):
    U, D, V = _factors(m, n, r, 5)
    U, V = (X.to(dtype).t().contiguous().t() for X in (U, V))
    {"U": U, "D": D, "V": V}[where][3, 4] = float("nan") if where != "V" else float("inf")
    got = _run(eod, U, D, V, m)
    ref = (U @ D.to(dtype)) @ V.t()
    assert bool(torch.equal(torch.isnan(got), torch.isnan(ref)))
    assert bool(torch.equal(torch.isinf(got), torch.isinf(ref)))
    ok = torch.isfinite(ref)
    assert not bool(ok.all())
    size = (U.abs().double() @ D.abs() @ V.abs().double().t())[ok]
    u = U64 if dtype == torch.float64 else 2.0 ** -24
    assert bool(((got[ok].double() - ref[ok].double()).abs() <= 4 * (r + 2) * u * size).all())
