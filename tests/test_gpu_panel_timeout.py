"""The panel kernel's bounded waits run out: a barrier waits for an arrival that nothing makes, every CTA
leaves within the limit, gks_sync reports GKS_ETIMEOUT, and the next solve on the context is whole again."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gks():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09058_gb300 import gks as g
    return g


# clusters of 16, 8 and one CTA, and the grid form
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,nk", [(40, 1), (104, 5), (40, 160), (418, 1), (300, 3)])
def test_expires_and_recovers(gks, n, nk, cplx):
    g = torch.Generator(device="cuda").manual_seed(n)
    dt = torch.complex128 if cplx else torch.float64
    a = torch.randn(nk, n, n, dtype=dt, device="cuda", generator=g)
    H, S = (a + a.mH).contiguous(), torch.eye(n, dtype=dt, device="cuda").repeat(nk, 1, 1).contiguous()
    ctx = gks.Context(0, debug=gks.GKS_DEBUG_LATE_ARRIVAL, wait_limit=1 << 28)
    t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    t0.record()
    with pytest.raises(gks.GKSError) as ei:
        ctx.solve(H, S, 0.1, 0.6 * n)
    t1.record()
    torch.cuda.synchronize()
    assert ei.value.code == gks.GKS_ETIMEOUT
    assert t0.elapsed_time(t1) < 10e3  # the limit is a seventh of a second; two waves of items at most
    sol = ctx.solve(H, S, 0.1, 0.6 * n)
    ref = gks.Context(0).solve(H, S, 0.1, 0.6 * n)
    assert all(torch.equal(getattr(sol, f), getattr(ref, f)) for f in ("eps", "C", "mu", "rho", "e_band"))
