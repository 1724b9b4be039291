"""Operands of more rows than a grid's second dimension holds in tiles of 32
(65535 x 32 = 2,097,120): slicing for the tensor-core products, through the
calls that reach it.

Bounds: A_hat entry by entry as two dot products of length r in the data's
precision, 2 (r + 2) u |U| |D| |V|^T, the reference's own error on top; the
factorisation's residual 100 n u ||A||_F with n the longer side of the core."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

F64, F32 = torch.float64, torch.float32
U = {F64: 2.0 ** -53, F32: 2.0 ** -24}
LONG = 2_200_003


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


@pytest.mark.parametrize("m,n,r,dtype", [(LONG, 9, 8, F64), (9, LONG, 8, F64), (LONG, 256, 257, F32),
                                         (256, LONG, 257, F32)])
def test_reconstruct(eod, m, n, r, dtype):
    g = torch.Generator(device="cuda").manual_seed(r)
    rnd = lambda a, b: (0.5 - torch.rand(b, a, generator=g, device="cuda", dtype=F64)).to(dtype).t()
    A, D, B = rnd(m, r), torch.triu(rnd(r, r)).double().t().contiguous().t(), rnd(n, r)
    f = eod.EodFactors(m=m, n=n, rank=r, precision=eod.EOD_PLAIN, f_dtype=eod.EOD_F64 if dtype == F64 else eod.EOD_F32)
    f.U, f.D, f.V = A.data_ptr(), D.data_ptr(), B.data_ptr()
    out = torch.empty(n, m, dtype=dtype, device="cuda").t()
    o = eod.make_opts(dtype=f.f_dtype)
    assert eod.eod_abe_reconstruct(ctypes.byref(f), ctypes.c_void_p(out.data_ptr()), m, ctypes.byref(o)) == eod.EOD_OK
    for c in range(0, m if m > n else n, 1 << 18):   # a part of the long side at a time
        rows, cols = (slice(c, c + (1 << 18)), slice(None)) if m > n else (slice(None), slice(c, c + (1 << 18)))
        L, R = A[rows].double(), B[cols].double()
        size = L.abs() @ D.abs() @ R.abs().t()
        assert bool(((out[rows, cols].double() - L @ D @ R.t()).abs() <= 4 * (r + 2) * U[dtype] * size).all())


def test_fp64_factorisation(eod):
    m, n, r = 4_300_001, 12, 5
    g = torch.Generator(device="cuda").manual_seed(1)
    rnd = lambda a, b: torch.randn(b, a, generator=g, device="cuda", dtype=F64).t()
    A = (rnd(n, r) @ rnd(m, r).t()).t()
    f = eod.factor(A, 1e-10, 3, tol_mode="rel")
    assert f.rank == r
    eye = torch.eye(r, dtype=F64, device="cuda")
    assert (f.U.t() @ f.U - eye).norm() <= 1e-12
    assert (f.U @ f.D @ f.V.t() - A).norm() <= 100 * n * U[F64] * A.norm()
