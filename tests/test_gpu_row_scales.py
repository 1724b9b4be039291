"""FP64 factorisations of a matrix whose rows differ in scale by up to 2^60, at
sizes where the products with Q's rows (Y -= Q S, U = Q Qh) have between 1.2e7
and 2^25 multiply-adds: Q, C and U, D, V reproduce every row to its own scale.

Each step treats a row apart from the others (A Omega, Y -= Q S, Y R^-1, Q Qh),
with a rounding error relative to that row, amplified by at most the condition
of the kept columns, kappa = ||A||_F / min T(l, l); the bound is 100 m u kappa
per row."""
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


@pytest.mark.parametrize("m,n,r,block", [(1500, 600, 100, 32), (1500, 600, 115, 32), (1100, 900, 160, 64),
                                         (1500, 600, 230, 128)])
def test_every_row_to_its_own_scale(eod, m, n, r, block):
    g = torch.Generator(device="cuda").manual_seed(r)
    rnd = lambda a, b: torch.randn(b, a, generator=g, device="cuda", dtype=torch.float64)
    scale = 2.0 ** -(60.0 * torch.rand(m, generator=g, device="cuda", dtype=torch.float64)).round()
    scale[torch.randperm(m, generator=g, device="cuda")[: 3 * r]] = 1.0
    A = ((rnd(n, r).t() @ rnd(m, r)) * scale).t()
    f = eod.factor(A, 1e-10, 5, tol_mode="rel", block_k=block)
    assert f.rank == r
    rows = A.norm(dim=1)
    bound = 100 * m * U64 * f.norm_a / min(f.tdiag[:r])
    assert bound < 1e-6
    assert float(((f.Q @ f.Ct.t() - A).norm(dim=1) / rows).max()) <= bound
    if m * r * r < 2 ** 25:
        assert float(((f.U @ f.D @ f.V.t() - A).norm(dim=1) / rows).max()) <= bound
