"""Reduction and eigenvalue kernels at the edges of their launch rules: the persistent panel's
cluster and grid forms, one CTA per item and more items than SMs, panel lengths at their
limits; the triangular solves' lanes and warps; the chemical potential in gaps and at steps;
the mixed path's digit reduction."""
import math

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2606_09058_gb300 import inputs as I

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def gks():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09058_gb300 import gks as g
    return g


@pytest.fixture(scope="module")
def ctx(gks):
    return gks.Context(0)


def _pencils(m, nk, cplx):
    H, S = zip(*(I.random_pencil(m, 40 * m + k, cplx, cond=10.0) for k in range(nk)))
    return np.stack(H), np.stack(S)


def _check_eigenpairs(H, S, eps, C):
    """Eigenvalues against LAPACK's on the reduced pencil (both backward stable: condition 10),
    scaled orthonormality and backward error within the parity gates."""
    for k in range(H.shape[0]):
        m = H.shape[1]
        Li = np.linalg.inv(np.linalg.cholesky(S[k]))
        ref = np.linalg.eigvalsh(Li @ H[k] @ Li.conj().T)
        assert np.abs(eps[k] - ref).max() <= 1e-10 * max(1.0, np.abs(ref).max()), k
        cn = np.linalg.norm(C[k], axis=0)
        G = C[k].conj().T @ S[k] @ C[k] - np.eye(m)
        R = H[k] @ C[k] - (S[k] @ C[k]) * eps[k]
        nh = np.linalg.norm(H[k], 2)
        assert np.abs(G / np.outer(cn, cn)).max() <= 1e-12 * math.sqrt(m), k
        assert (np.linalg.norm(R, axis=0) / ((nh + np.abs(eps[k])) * cn)).max() <= 1e-12 * math.sqrt(m), k


# order - 1 <= 160 runs one cluster, above a grid; panels take 64 steps; digit tiles are 32 x 16.
# 80 items share the SMs one CTA each (corrections behind the product from order 250 complex),
# 160 items are more than the SMs.
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m,nk", [(2, 1), (3, 2), (4, 1), (17, 1), (32, 3), (33, 1), (64, 1), (65, 2), (66, 1), (97, 1),
                                  (128, 1), (129, 1), (161, 1), (162, 2), (225, 1), (418, 1), (260, 80), (40, 160)])
def test_panel_edges(ctx, cplx, m, nk):
    H, S = _pencils(m, nk, cplx)
    sol = ctx.solve(torch.as_tensor(H).cuda(), torch.as_tensor(S).cuda(), 0.1, 0.8 * m)
    _check_eigenpairs(H, S, sol.eps.cpu().numpy(), sol.C.cpu().numpy())


@pytest.mark.parametrize("cplx,m", [(True, 66), (True, 300), (False, 640)])
@pytest.mark.parametrize("shift", [-61, 60])
def test_deferred_update_scales(ctx, cplx, m, shift):
    """The deferred update as one product with balanced columns: H and 2^shift H give the same
    eigenvalues up to the scale, within 8 m u ||H|| each."""
    H, S = _pencils(m, 1, cplx)
    a, b = (ctx.solve(torch.as_tensor(H * f).cuda(), torch.as_tensor(S).cuda(), 0.1 * f, 0.8 * m).eps.cpu().numpy()[0]
            for f in (1.0, 2.0 ** shift))
    assert np.abs(a - b / 2.0 ** shift).max() <= 16 * m * U * 10.0 * np.linalg.norm(H[0], 2)
    _check_eigenpairs(H, S, a[None], ctx.solve(torch.as_tensor(H).cuda(), torch.as_tensor(S).cuda(), 0.1,
                                               0.8 * m).C.cpu().numpy())


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m,count", [(65, 1), (70, 151), (129, 7), (192, 40), (200, 9), (321, 30)])
def test_triangular_solves_by_lanes_and_warps(ctx, cplx, m, count):
    """|L L^H - S| within the Cholesky bound (m + 1) 8 u max S_ii; L^-1 H L^-H as the oracle's
    gate."""
    H, S = _pencils(m, min(count, 4), cplx)
    idx = np.arange(count) % H.shape[0]
    L = ctx.potrf(torch.as_tensor(S[idx]).cuda()).cpu().numpy()
    R, _ = ctx.reduce(torch.as_tensor(H[idx]).cuda(), torch.as_tensor(S[idx]).cuda())
    R = R.cpu().numpy()
    ref = [O.reduce_standard(O.cholesky(S[k]), H[k]) for k in range(H.shape[0])]
    for i, k in enumerate(idx):
        l = np.tril(L[i])
        assert np.abs(l @ l.conj().T - S[k]).max() <= 8 * U * (m + 1) * np.abs(np.diagonal(S[k])).max()
        assert np.abs(np.tril(R[i]) - np.tril(ref[k])).max() <= 1e-12 * m * max(1.0, np.abs(ref[k]).max())


def _levels(kind, nk, m, rng):
    if kind == "spread":
        return np.sort(rng.uniform(-1.0, 1.0, (nk, m)), axis=1), 0.02, 0.7 * m
    if kind == "gap":  # no level within 100 kT of mu
        e = np.concatenate([rng.uniform(-2.0, -1.0, (nk, m // 2)), rng.uniform(1.0, 2.0, (nk, m - m // 2))], axis=1)
        return np.sort(e, axis=1), 0.01, 2.0 * (m // 2)
    if kind == "cold":  # steps far below the level spacing
        return np.sort(rng.uniform(-1.0, 1.0, (nk, m)), axis=1), 1e-9, 0.9 * m
    if kind == "hot":
        return np.sort(rng.uniform(-1.0, 1.0, (nk, m)), axis=1), 50.0, 0.3 * m
    return np.zeros((nk, m)) + 0.25, 0.05, 1.3 * m  # one degenerate level


@pytest.mark.parametrize("kind", ["spread", "gap", "cold", "hot", "level"])
@pytest.mark.parametrize("nk,m", [(1, 2), (1, 1023), (3, 1025), (8, 400)])
def test_chemical_potential(ctx, kind, nk, m):
    """The electron count changes sign across mu +- 8 u max(1, |mu|) up to the rounding of its
    sum (u per term and 200 terms per lane at most, so 256 u n); a root outside the bracket
    [min eps - 1, max eps + 1] gives its end, as in the oracle."""
    rng = np.random.default_rng(5 + nk + m)
    eps, kT, ne = _levels(kind, nk, m, rng)
    w = rng.uniform(0.5, 1.5, nk)
    w /= w.sum()
    mu = ctx.occupy(torch.as_tensor(eps).cuda(), None, kT, ne, kweights_all=torch.as_tensor(w).cuda())[0].item()

    def count(x):
        return 2.0 * math.fsum((w[:, None] / (1.0 + np.exp(np.clip((eps - x) / kT, -700, 700)))).ravel())
    d = 8 * U * max(1.0, abs(mu))
    if kind == "hot":
        ref = O.chemical_potential(eps, w, 2.0, kT, ne)
        assert ref == pytest.approx(eps.min() - 1.0, abs=d)
        assert abs(mu - ref) <= d
        return
    assert count(mu - d) <= ne * (1 + 256 * U) and count(mu + d) >= ne * (1 - 256 * U)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m,nk", [(65, 1), (193, 2)])
def test_mixed_digit_reduction(gks, cplx, m, nk):
    H, S = _pencils(m, nk, cplx)
    c2 = gks.Context(0, precision="mixed")
    sol = c2.solve(torch.as_tensor(H).cuda(), torch.as_tensor(S).cuda(), 0.1, 0.8 * m)
    _check_eigenpairs(H, S, sol.eps.cpu().numpy(), sol.C.cpu().numpy())
