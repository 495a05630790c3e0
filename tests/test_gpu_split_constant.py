"""Split products of constant operands, whose chunk sums of residues are far larger than those
of random signs: dyadic entries, so that the product is an integer the residues carry exactly
and FP64 holds exactly."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09058_gb300 import gks
    return gks.Context(0)


# the single fold of these sums is 128 for modulus 255 (K' = 832 and 1024)
PAIRS = {1024: [(1.31640625, 1.01171875), (1.671875, 1.9765625), (1.48046875, 1.19921875), (1.43359375, 1.36328125)],
         832: [(1.55078125, 1.69140625), (1.35546875, 1.203125), (1.5390625, 1.65625)],
         64: [(1.99609375, 1.99609375)], 1025: [(1.31640625, 1.01171875)]}


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("Kp", sorted(PAIRS))
def test_constant_operands(ctx, Kp, sign, cplx):
    dt = torch.complex128 if cplx else torch.float64
    K = Kp // 2 if cplx else Kp
    for a, b in PAIRS[Kp]:
        A = torch.full((130, K), sign * a, dtype=dt, device="cuda")
        B = torch.full((K, 70), b, dtype=dt, device="cuda")
        if cplx:  # the embedded row (Re, Im) meets (Re, Im) and (-Im, Re)
            A, B = A * (1 + 1j), B * (1 + 1j)
        C = ctx.gemm(A, B, torch.zeros(130, 70, dtype=dt, device="cuda"), mode="split")
        want = sign * K * a * b * ((1 + 1j) ** 2 if cplx else 1.0)
        assert torch.equal(C, torch.full_like(C, want))
