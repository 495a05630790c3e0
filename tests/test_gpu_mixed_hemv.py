"""Mixed precision follows opts.hemv: with "fp64" the single-precision steps run at every order
(two launches per step), with "digits" small orders take the digit form (one per panel)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cplx", [False, True])
def test_mixed_keeps_the_chosen_step(cplx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09058_gb300 import gks
    n = 200
    g = torch.Generator(device="cuda").manual_seed(7)
    dt = torch.complex128 if cplx else torch.float64
    a = torch.randn(n, n, dtype=dt, device="cuda", generator=g)
    H, S = (a + a.mH).contiguous()[None], torch.eye(n, dtype=dt, device="cuda")[None].contiguous()
    launches = {}
    for hemv in ("digits", "fp64"):
        ctx = gks.Context(0, precision="mixed", hemv=hemv)
        before = gks.launch_count()
        sol = ctx.solve(H, S, 0.1, 0.6 * n)
        launches[hemv] = gks.launch_count() - before
        ref = torch.linalg.eigvalsh(H)  # both forms refine to FP64: 8 n u ||H|| each
        assert (sol.eps - ref).abs().max() <= 16 * n * 2.0 ** -53 * ref.abs().max()
    # steps j = n - 1 .. 2 in two launches each; the digit form's whole solve takes fewer
    assert launches["digits"] < 2 * (n - 2) <= launches["fp64"]
