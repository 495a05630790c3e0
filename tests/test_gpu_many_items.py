"""Many small pencils in one call: cluster sizes of the panel kernel and of the diagonal-block
kernels by the item count, waves of items, and products with a large batch."""
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09058_gb300 import gks
    return gks.Context(0)


def _pencils(m, nk, cplx):
    g = torch.Generator(device="cuda").manual_seed(100 * m + nk)
    dt = torch.complex128 if cplx else torch.float64
    a, b = (torch.randn(nk, m, m, dtype=dt, device="cuda", generator=g) for _ in range(2))
    S = torch.eye(m, dtype=dt, device="cuda") + 0.1 / m ** 0.5 * (b + b.mH)  # condition below 10
    return (a + a.mH).contiguous(), S.contiguous()


def _check(H, S, sol, m):
    """Residual and orthonormality of every item within 64 m u of their scales (Householder,
    Cholesky and products: a few m u each), eigenvalues of some against a library's."""
    some = sorted({0, H.shape[0] // 2, H.shape[0] - 1})
    nh = torch.linalg.eigvalsh(H[some]).abs().max()
    R = H @ sol.C - (S @ sol.C) * sol.eps[:, None, :]
    assert R.abs().max() <= 64 * m * U * nh * sol.C.abs().max().clamp_min(1.0)
    assert (sol.C.mH @ S @ sol.C - torch.eye(m, dtype=H.dtype, device="cuda")).abs().max() <= 64 * m * U
    Li = torch.linalg.inv(torch.linalg.cholesky(S[some]))
    ref = torch.linalg.eigvalsh(Li @ H[some] @ Li.mH)
    assert (sol.eps[some] - ref).abs().max() <= 64 * m * U * nh


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m", [3, 40, 104, 161, 170])
@pytest.mark.parametrize("nk", [5, 17, 70, 310])
def test_items(ctx, m, nk, cplx):
    H, S = _pencils(m, nk, cplx)
    _check(H, S, ctx.solve(H, S, 0.05, 0.6 * m), m)


def test_more_merges_than_a_grid_holds(ctx):
    """20000 tridiagonals of order 34: 80000 products in the first merges."""
    m, nk = 34, 20000
    g = torch.Generator(device="cuda").manual_seed(3)
    d, e = (torch.randn(nk, m, dtype=torch.float64, device="cuda", generator=g) for _ in range(2))
    lam, Z = ctx.stedc(d, e)
    T = torch.diag_embed(d) + torch.diag_embed(e[:, :-1], 1) + torch.diag_embed(e[:, :-1], -1)
    assert (T @ Z - Z * lam[:, None, :]).abs().max() <= 32 * m * U * T.abs().sum(-1).max()
    assert (Z.mT @ Z - torch.eye(m, dtype=torch.float64, device="cuda")).abs().max() <= 32 * m * U
