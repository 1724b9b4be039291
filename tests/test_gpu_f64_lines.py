"""FP64 factorisations on both sides of the lines where products move to the
tensor-core emulation: slices of A and Q kept from 1.9e7 multiply-adds a block
(m n k), a product with one sliced operand from 1.2e7, with neither from 2.1e7.

Exact rank r with singular values in [1e-2, 1]: the rank is found, U and V are
orthonormal and U D V^T is A to a few units of rounding.  Bounds: CholQR2 leaves
O(n u) of orthogonality (Yamamoto et al. 2015, Thm 3.1), taken as 20 n u; the
residual is at most that of the projections and two factorisations, 100 n u
||A||_F."""
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


@pytest.mark.parametrize("m,n", [(770, 770), (772, 771), (1001, 523), (523, 1001), (1024, 1023), (2049, 300)])
@pytest.mark.parametrize("r,block", [(37, 32), (101, 32), (150, 64), (200, 128)])
def test_factorisation_across_the_lines(eod, m, n, r, block):
    g = torch.Generator(device="cuda").manual_seed(m * 7 + n + r)
    L = torch.linalg.qr(torch.randn(m, r, generator=g, device="cuda", dtype=torch.float64))[0]
    R = torch.linalg.qr(torch.randn(n, r, generator=g, device="cuda", dtype=torch.float64))[0]
    s = torch.logspace(0, -2, r, dtype=torch.float64, device="cuda")
    A = ((R * s) @ L.t()).t()
    f = eod.factor(A, 1e-10, 5, tol_mode="abs", block_k=block)
    assert f.rank == r
    size = max(m, n)
    eye = torch.eye(r, dtype=torch.float64, device="cuda")
    assert (f.U.t() @ f.U - eye).norm() <= 20 * size * U64
    assert (f.V.t() @ f.V - eye).norm() <= 20 * size * U64
    assert (f.U @ f.D @ f.V.t() - A).norm() <= 100 * size * U64 * A.norm()
