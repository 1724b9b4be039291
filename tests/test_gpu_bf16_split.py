"""The BF16 split of a matrix whose columns do or do not start on 16 bytes,
through the sketch contraction against FP64 products.

Bound per entry, relative to |X| |Y|: FP32 accumulation of exact products, whose
rounding walks with the number of terms: 2^-24 sqrt(K), taken eight times."""
import ctypes
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


def _matrix(rows, cols, ld, off, g, exact=False):
    """rows x cols, column-major with leading dimension ld, `off` floats into its buffer."""
    buf = torch.full((off + cols * ld,), float("nan"), device="cuda")
    x = torch.randn((cols, rows), generator=g)
    x = x.to(torch.bfloat16).float() if exact else x
    v = buf[off:].view(cols, ld).t()[:rows]
    v.copy_(x.t().cuda())
    return v


def _run(eod, form, M, N, K, X, Y):
    D = torch.full((N, M), float("nan"), device="cuda").t()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    st = eod.eod_abe_debug_tc_gemm(form, M, N, K, p(X), X.stride(1), p(Y), Y.stride(1), p(D), M, None,
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == eod.EOD_OK, eod.status_string(st)
    return D


@pytest.mark.parametrize("rows", [1, 3, 4, 5, 2047, 2048, 2049, 4100])
@pytest.mark.parametrize("pad,off", [(0, 0), (4, 0), (1, 0), (4, 1), (2, 2)])
def test_split_of_aligned_and_unaligned_columns(eod, rows, pad, off):
    """The sketch form splits X (rows x K) exactly into three BF16 terms."""
    N, K = 16, 70
    g = torch.Generator().manual_seed(rows + 10 * pad + off)
    X, Y = _matrix(rows, K, (rows + 3) // 4 * 4 + pad, off, g), _matrix(K, N, K, 0, g, exact=True)
    D = _run(eod, 0, rows, N, K, X, Y)
    ref = X.double() @ Y.double()
    scale = X.double().abs() @ Y.double().abs()
    assert torch.isfinite(D).all()
    assert ((D.double() - ref).abs() <= 8 * math.sqrt(K) * 2.0 ** -24 * scale).all()
