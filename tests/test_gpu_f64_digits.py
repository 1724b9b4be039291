"""The emulated FP64 product on integers, where it has to be the exact sum
rounded once: entries below 2^26 take four base-256 digits, every pair of them
is among the products kept, and the digit sums are integers.  K around the
256-term chunks and 64-term blocks, rows of extreme equal-signed digits, a
wide spread of row scales, and the rounding of sums beyond 53 bits.  (Outputs
of at least 152 tiles of 128 x 64: smaller ones split K and add the rounded
partial sums.)"""
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


def _product(eod, A, B, ta=0, alpha=1.0, beta=0.0, C=None):
    """alpha op(A) B + beta C through the emulation, column-major."""
    M, K, N = (A.shape[1], A.shape[0], B.shape[1]) if ta else (A.shape[0], A.shape[1], B.shape[1])
    Ad, Bd = (torch.from_numpy(np.asfortranarray(X)).cuda() for X in (A, B))
    out = torch.from_numpy(np.asfortranarray(np.zeros((M, N)) if C is None else C)).cuda()
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    st = eod.eod_abe_debug_f64_gemm(1, ta, 0, M, N, K, alpha, P(Ad), A.shape[0], P(Bd), B.shape[0], beta, P(out), M,
                                    ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == eod.EOD_OK
    return out.cpu().numpy()


def _exact(A, B):
    """The integer product rounded once to double: entries in two parts of 14
    bits and less, whose products sum exactly in double, joined in int64."""
    Ah, Bh = np.round(A / 8192.0), np.round(B / 8192.0)
    Al, Bl = A - 8192.0 * Ah, B - 8192.0 * Bh
    hi, mid, lo = Ah @ Bh, Ah @ Bl + Al @ Bh, Al @ Bl
    return ((hi.astype(np.int64) << 26) + (mid.astype(np.int64) << 13) + lo.astype(np.int64)).astype(np.float64)


M, N = 1311, 997   # 176 tiles


@pytest.mark.parametrize("K", [8, 63, 64, 65, 255, 256, 257, 300, 511, 513, 1025])
@pytest.mark.parametrize("ta", [0, 1])
def test_integer_products_are_rounded_once(eod, K, ta):
    rng = np.random.default_rng(K)
    A = rng.integers(-2**26 + 1, 2**26, (M, K)).astype(np.float64)
    B = rng.integers(-2**26 + 1, 2**26, (K, N)).astype(np.float64)
    A[3] = 0.0
    B[:, 5] = 0.0
    A[7] = np.sign(A[7])
    assert np.array_equal(_product(eod, A.T if ta else A, B, ta), _exact(A, B))


@pytest.mark.parametrize("digit", [128, 127, -128, 85])
@pytest.mark.parametrize("K", [256, 260, 700])
def test_equal_extreme_digits(eod, digit, K):
    """Every entry the same four digits: all partial sums run one way."""
    x = sum(digit * 256 ** i for i in range(3)) + (abs(digit) // 2) * 256 ** 3
    A, B = np.full((M, K), float(x)), np.full((K, N), float(x))
    A[1] *= -1.0
    ref = np.full((M, N), float(K * x * x))
    ref[1] *= -1.0
    assert np.array_equal(_product(eod, A, B), ref)


def test_scales_and_accumulation(eod):
    """Row scales from 2^-300 to 2^300 (exact powers), C = -A B + C."""
    rng = np.random.default_rng(3)
    A = rng.integers(-2**20, 2**20, (140, 330)).astype(np.float64)
    B = rng.integers(-2**20, 2**20, (330, 70)).astype(np.float64)
    s = np.ldexp(1.0, rng.integers(-300, 301, 140))[:, None]
    ref = _exact(A, B)
    assert np.array_equal(_product(eod, A * s, B), ref * s)
    C = rng.integers(-2**40, 2**40, ref.shape).astype(np.float64)
    assert np.array_equal(_product(eod, A, B, alpha=-1.0, beta=1.0, C=C), C - ref)   # |ref| < 2^49: exact
