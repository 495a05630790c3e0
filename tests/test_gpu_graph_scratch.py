"""A graph-mode context between other calls: a captured solve holds the addresses of the
split-product scratch, which larger calls on the same context replace.  Every call equals the
one of a context without graphs bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09058_gb300 import gks
    return gks


KT = 0.02


def _pencil(n, cplx, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.complex128 if cplx else torch.float64
    a, b = (torch.randn(1, n, n, dtype=dt, device="cuda", generator=g) for _ in range(2))
    return (a + a.mH).contiguous(), (torch.eye(n, dtype=dt, device="cuda") + 0.1 / n ** 0.5 * (b + b.mH)).contiguous()


class _Case:
    """A graph-mode context and an eager one on a stream, and one set of buffers."""

    def __init__(self, lib, n, cplx, **opts):
        self.stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(self.stream):
            self.graph = lib.Context(0, self.stream, graph=True, **opts)
            self.eager = lib.Context(0, self.stream, **opts)
            self.n, self.ne = n, 0.6 * n
            self.H, self.S = _pencil(n, cplx, n)
            self.out = self._buffers()
            self.ref_out = self._buffers()

    def _buffers(self):
        r = {"eps": torch.empty(1, self.n, dtype=torch.float64, device="cuda"), "C": torch.empty_like(self.H),
             "rho": torch.empty_like(self.H)}
        r["mu"], r["e_band"] = (torch.empty(1, dtype=torch.float64, device="cuda") for _ in range(2))
        return r

    def solve(self, eigen_only, **kw):
        for ctx, out in ((self.graph, self.out), (self.eager, self.ref_out)):
            for t in out.values():
                t.zero_()
            ctx.solve_into(self.H, self.S, KT, self.ne, eigen_only=eigen_only, **out, **kw)
        assert all(torch.equal(self.out[k], self.ref_out[k]) for k in self.out)

    def occupy(self):
        a, b = (ctx.occupy(self.ref_out["eps"], self.ref_out["C"], KT, self.ne, edm=True)
                for ctx in (self.graph, self.eager))
        assert all(torch.equal(x, y) for x, y in zip(a, b))

    def gemm(self, m):
        g = torch.Generator(device="cuda").manual_seed(m)
        A = torch.randn(m, m, dtype=self.H.dtype, device="cuda", generator=g)
        a, b = (ctx.gemm(A, A, torch.zeros_like(A)) for ctx in (self.graph, self.eager))
        assert torch.equal(a, b)


# the largest product of an eigen-only solve needs less scratch than the density matrix
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n", [416, 832])
def test_captured_eigenpairs_between_larger_calls(lib, n, cplx):
    c = _Case(lib, n, cplx)
    with torch.cuda.stream(c.stream):
        for _ in range(3):  # eager, captured, replayed
            c.solve(True)
        c.occupy()
        for _ in range(2):  # captured anew, replayed
            c.solve(True)
        c.gemm(2 * n)
        c.solve(True)
        c.occupy()
        c.solve(True)
    c.stream.synchronize()


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n", [416, 832])
def test_full_solve_after_captured_eigenpairs(lib, n, cplx):
    """Another path on the same buffers runs eagerly before it is captured, also after other
    entry points have replaced the workspace."""
    c = _Case(lib, n, cplx)
    with torch.cuda.stream(c.stream):
        for _ in range(3):
            c.solve(True)
        for _ in range(3):
            c.solve(False)
        for _ in range(3):
            c.solve(False, reuse_s=True)
        c.solve(True)
        c.graph.potrf(c.S.clone())
        c.graph.potrf(torch.eye(40, dtype=c.S.dtype, device="cuda")[None].contiguous())
        c.graph.potrf(c.S.clone())
        for _ in range(3):
            c.solve(True)
    c.stream.synchronize()


def test_workspace_of_another_form_between_solves(lib):
    c = _Case(lib, 160, False)
    with torch.cuda.stream(c.stream):
        for _ in range(3):
            c.solve(False)
        c.graph.he2hb(c.H.clone(), 16)
        for _ in range(3):
            c.solve(False)
    c.stream.synchronize()


@pytest.mark.parametrize("n", [70, 260])
def test_tridiagonal_entry_between_solves(lib, n):
    """gks_stedc shares the merges' product lists with the solve."""
    c = _Case(lib, n, False)
    d, e = (torch.rand(1, n, dtype=torch.float64, device="cuda") for _ in range(2))
    with torch.cuda.stream(c.stream):
        lam, Z = c.eager.stedc(d, e)
        for _ in range(3):
            c.solve(False)
        lam2, Z2 = c.graph.stedc(d, e)
        keep = Z2.clone()
        assert torch.equal(lam2, lam) and torch.equal(Z2, Z)
        for _ in range(3):
            c.solve(False)
        assert torch.equal(Z2, keep)
        c.graph.solve_into(c.H, c.S, KT, c.ne, sync=False, **c.out)  # in flight
        lam2, Z2 = c.graph.stedc(d, e)
        assert torch.equal(lam2, lam) and torch.equal(Z2, Z)
        assert all(torch.equal(c.out[k], c.ref_out[k]) for k in c.out)
    c.stream.synchronize()
