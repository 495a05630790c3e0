"""Split products at the edges of their launch rules: tiles and residue groups just full and
just over, the one-launch and two-launch splitting (padded inner length 1024 and over), one
chunk and several, the smallest dispatched sizes, and non-finite operands."""
import numpy as np
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


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("ops", [("N", "C"), ("C", "N")])
@pytest.mark.parametrize("shape", [(32, 32, 32), (128, 256, 512), (129, 257, 513), (256, 128, 1024), (130, 70, 1025),
                                   (1000, 40, 65), (40, 1300, 1)])
def test_split_product_edges(ctx, cplx, ops, shape):
    """Within 54 bits below the row and column scales plus the FP64 rounding of the reference
    (K terms) and of the final sum."""
    M, N, K = shape
    rng = np.random.default_rng(M + 3 * N + 7 * K)

    def rnd(r, c):
        x = rng.standard_normal((r, c)) * 2.0 ** rng.integers(-9, 9, (r, c))
        return x + 1j * rng.standard_normal((r, c)) if cplx else x
    A = rnd(*((M, K) if ops[0] == "N" else (K, M)))
    B = rnd(*((K, N) if ops[1] == "N" else (N, K)))
    C0 = rnd(M, N)
    a = A if ops[0] == "N" else A.conj().T
    b = B if ops[1] == "N" else B.conj().T
    Cd = torch.as_tensor(C0).cuda()
    ctx.gemm(torch.as_tensor(A).cuda(), torch.as_tensor(B).cuda(), Cd, ops[0], ops[1], -1.0, 1.0, "split")
    Ke = 2 * K if cplx else K
    bound = 4 * Ke * 2.0 ** -54 * 2 * np.abs(a).max(1, keepdims=True) * 2 * np.abs(b).max(0, keepdims=True)
    bound = bound + 4 * U * (Ke * (np.abs(a) @ np.abs(b)) + np.abs(C0))
    err = np.abs(Cd.cpu().numpy() - (C0 - a @ b))
    assert np.all(err <= bound), (err / bound).max()


@pytest.mark.parametrize("form", ["residues", "digits"])
@pytest.mark.parametrize("K", [100, 1100])
def test_non_finite_operands_stay_visible(form, K):
    """A NaN or an infinity in a row of A or a column of B makes that row or column of the
    product NaN, and nothing else (as on the FP64 pipe, up to inf there)."""
    from paper_2606_09058_gb300 import gks
    c2 = gks.Context(0, split=form)
    A = torch.randn(150, K, dtype=torch.float64, device="cuda")
    B = torch.randn(K, 140, dtype=torch.float64, device="cuda")
    A[3, 7], B[K - 1, 11] = float("nan"), float("inf")
    C = c2.gemm(A, B, torch.zeros(150, 140, dtype=torch.float64, device="cuda"), mode="split")
    bad = torch.zeros_like(C, dtype=torch.bool)
    bad[3], bad[:, 11] = True, True
    assert torch.equal(torch.isnan(C), bad)
