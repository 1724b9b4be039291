"""The emulated FP64 product where the sums of its later digit groups are the
largest they can be: row and column digits of extreme size whose signs agree
across one group g = s + t, while all the others cancel and do not hide an error
in it.  The result has to be the
exact sum of the products kept (s + t below the number of digits: seven in
`eod_abe_debug_f64_gemm`, eight in `eod_abe_reconstruct`), rounded once.
K around the chunks of 128 and 256 terms.  (Outputs of at least 152 tiles of
128 x 64: smaller ones split K.)"""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

M, N = 1311, 997   # 176 tiles


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


def _digits(rng, K, group):
    """A row of signed digits a[k][s] and a column b[k][t] over positions 0..6 (the
    last a multiple of 4: 53 bits).  Eight k at a time share their sizes, and
    the signs are rows of a Hadamard matrix: a_s b_t sums to zero over them unless
    s + t = group, where all products are positive.  k in a random order inside
    each 256 (an MMA's partial sums are then odd and even)."""
    H = np.array([[1]])
    for _ in range(3):
        H = np.block([[H, H], [H, -H]])
    pos = np.arange(7)
    a, b = (np.concatenate([rng.integers(121, 128, (K // 8, 6)), np.full((K // 8, 1), 124)], axis=1).repeat(8, axis=0)
            for _ in range(2))
    u = group - pos
    a *= np.tile(H[:, pos], (K // 8, 1)) * (pos <= group)
    b *= np.tile(H[:, u % 8], (K // 8, 1)) * (u >= 0)
    order = np.concatenate([c + rng.permutation(min(256, K - c)) for c in range(0, K, 256)])
    return a[order], b[order]


def _values(d):
    return (d * (256.0 ** (6 - np.arange(7)))).sum(-1)   # below 2^55, multiples of 4 where above 2^53: exact


def _case(K, group, slices):
    """A, B^T and their product over s + t < slices, rounded once: one value, the
    rows and columns at different powers of two and signs."""
    rng = np.random.default_rng(100 * K + group)
    a, b = _digits(rng, K, group)
    tot = sum(int(a[:, s] @ b[:, t]) * 256 ** (12 - s - t) for s in range(7) for t in range(7) if s + t < slices)
    r, c = (rng.choice([-1.0, 1.0], x) * 2.0 ** rng.integers(-40, 41, x) for x in (M, N))
    return r[:, None] * _values(a), c[:, None] * _values(b), np.outer(r, c) * float(tot)


@pytest.mark.parametrize("K", [64, 128, 192, 256, 264, 320, 704])
@pytest.mark.parametrize("group", [4, 5, 6])
def test_seven_digits(eod, K, group):
    A, Bt, ref = _case(K, group, 7)
    Ad, Bd = (torch.from_numpy(np.asfortranarray(X)).cuda() for X in (A, Bt))
    out = torch.zeros(N, M, dtype=torch.float64, device="cuda").t()
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    st = eod.eod_abe_debug_f64_gemm(1, 0, 1, M, N, K, 1.0, P(Ad), M, P(Bd), N, 0.0, P(out), M,
                                    ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == eod.EOD_OK
    assert np.array_equal(out.cpu().numpy(), ref)


@pytest.mark.parametrize("K", [64, 192, 256, 264, 704])
@pytest.mark.parametrize("group", [4, 6, 7])
def test_eight_digits(eod, K, group):
    A, Bt, ref = _case(K, group, 8)
    U, V = (torch.from_numpy(np.asfortranarray(X)).cuda() for X in (A, Bt))
    D = torch.eye(K, dtype=torch.float64, device="cuda")
    f = eod.EodFactors(m=M, n=N, rank=K, precision=eod.EOD_PLAIN, f_dtype=eod.EOD_F64)
    f.U, f.D, f.V = U.data_ptr(), D.data_ptr(), V.data_ptr()
    out = torch.zeros(N, M, dtype=torch.float64, device="cuda").t()
    o = eod.make_opts(dtype=eod.EOD_F64)
    assert eod.eod_abe_reconstruct(ctypes.byref(f), ctypes.c_void_p(out.data_ptr()), M, ctypes.byref(o)) == eod.EOD_OK
    assert np.array_equal(out.cpu().numpy(), ref)
