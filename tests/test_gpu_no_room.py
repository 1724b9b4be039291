"""Without room for the operands' digit slices a product runs on the FMA kernels:
plain FP32 factorisations (the projection and U on the tensor cores) and A_hat,
with the n-th allocation of the call refused, for every n.  Either the call
reports EOD_ENOMEM (its own buffers) or it returns the result; the slices' turn
shows as an emulated product less.

Bounds: the factorisation's residual 100 n u ||A||_F, n the longer side; A_hat
entry by entry 2 (r + 2) u |U| |D| |V|^T, the reference's own on top."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

OZ_GEMM = 5   # the profile counters' kind


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


def _counted(eod, call, refuse):
    """The call's outcome with the refuse-th allocation failing (0: none), and its emulated products."""
    n, ms, fl, by = ctypes.c_int64(), ctypes.c_double(), ctypes.c_double(), ctypes.c_double()
    eod.eod_abe_debug_profile(1)
    eod.eod_abe_debug_fail_alloc_after(refuse)
    try:
        out = call()
    except eod.EodError as e:
        assert e.status == eod.EOD_ENOMEM
        out = None
    finally:
        eod.eod_abe_debug_fail_alloc_after(0)
        torch.cuda.synchronize()
        assert eod.eod_abe_debug_profile_read(OZ_GEMM, ctypes.byref(n), ctypes.byref(ms), ctypes.byref(fl),
                                              ctypes.byref(by)) == eod.EOD_OK
        eod.eod_abe_debug_profile(0)
    return out, n.value


def _sweep(eod, call, check):
    _, every = _counted(eod, call, 0)
    assert every >= 1
    fewer = refused = 0
    for n in range(1, 120):
        out, done = _counted(eod, call, n)
        if out is None:
            refused += 1
            continue
        check(out)
        fewer += done < every
    assert refused >= 1 and fewer >= 2 * every   # both operands of each product, their exponents


def test_fp32_factorisation(eod):
    g = torch.Generator(device="cuda").manual_seed(4)
    m, n, r = 1600, 1300, 700
    rnd = lambda a, b: torch.randn(b, a, generator=g, device="cuda", dtype=torch.float64)
    A = (rnd(n, r).t() @ rnd(m, r)).float().t()

    def call():
        f = eod.factor(A, 1e-3, 5, tol_mode="rel", compute_err=False, block_k=128)
        out = f.rank, f.U.clone(), f.D.clone(), f.V.clone()
        f.close()
        return out

    def check(out):
        rank, U, D, V = out
        assert rank == r
        assert float((U.double() @ D @ V.double().t() - A.double()).norm()) <= 100 * m * 2.0 ** -24 * float(A.double().norm())
    _sweep(eod, call, check)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_reconstruct(eod, dtype):
    g = torch.Generator(device="cuda").manual_seed(7)
    m, n, r = 1400, 1300, 500
    rnd = lambda a, b: (0.5 - torch.rand(b, a, generator=g, device="cuda", dtype=torch.float64)).t()
    U, V = rnd(m, r).to(dtype).t().contiguous().t(), rnd(n, r).to(dtype).t().contiguous().t()
    D = torch.triu(rnd(r, r)).t().contiguous().t()
    f = eod.EodFactors(m=m, n=n, rank=r, precision=eod.EOD_PLAIN,
                       f_dtype=eod.EOD_F64 if dtype == torch.float64 else eod.EOD_F32)
    f.U, f.D, f.V = U.data_ptr(), D.data_ptr(), V.data_ptr()
    ref = U.double() @ D @ V.double().t()
    bound = 4 * (r + 2) * (2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24) * (U.double().abs() @ D.abs() @ V.double().abs().t())

    def call():
        out = torch.empty(n, m, dtype=dtype, device="cuda").t()
        o = eod.make_opts(dtype=f.f_dtype)
        st = eod.eod_abe_reconstruct(ctypes.byref(f), ctypes.c_void_p(out.data_ptr()), m, ctypes.byref(o))
        if st != eod.EOD_OK:
            raise eod.EodError(st, "eod_abe_reconstruct")
        return out

    def check(out):
        assert bool(((out.double() - ref).abs() <= bound).all())
    _sweep(eod, call, check)
