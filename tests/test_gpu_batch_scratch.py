"""Device memory of a large batch: the problems of one worker stream run one after another and
share their split-product scratch, so each further problem adds its workspace only."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("graph", [False, True])
def test_memory_per_problem(graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09058_gb300 import gks
    n = 416
    g = torch.Generator(device="cuda").manual_seed(1)
    a = torch.randn(1, n, n, dtype=torch.complex128, device="cuda", generator=g)
    H, S = (a + a.mH).contiguous(), torch.eye(n, dtype=torch.complex128, device="cuda")[None].contiguous()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        alone = gks.Context(0, stream, gemm="fp64")  # no split products: the workspace
        ref = gks.Context(0, stream).solve(H, S, 0.02, 0.6 * n)
        before = _used()
        out = alone.solve(H, S, 0.02, 0.6 * n)
        ws = _used() - before
        del out
        ctx = gks.Context(0, stream, graph=graph)

        def run(count):
            outs = [gks.Solution(torch.empty(1, n, dtype=torch.float64, device="cuda"), torch.empty_like(H),
                                 torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(H),
                                 torch.empty(1, dtype=torch.float64, device="cuda")) for _ in range(count)]
            before = _used()
            probs = [{"H": H, "S": S, "kT": 0.02, "n_elec": 0.6 * n}] * count
            for _ in range(3 if graph else 1):
                ctx.solve_batched(probs, out=outs)
            for s in outs:
                assert all(torch.equal(getattr(s, f), getattr(ref, f)) for f in ("eps", "C", "mu", "rho", "e_band"))
            return _used() - before
        run(4)       # scratch of their own
        run(160)     # about 13 GB if each had its own
        more = run(240)
        run(4)
        ctx.close()
        # a quarter for the captured graph's and the streams' own memory
        assert more <= 80 * 1.25 * ws, (more, ws)
    stream.synchronize()
