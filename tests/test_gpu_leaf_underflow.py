"""Leaves of the divide and conquer with couplings whose squares underflow, beside zero and equal
diagonal entries."""
import numpy as np
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


C = [5e-324, 1e-300, 1e-170, 1.4e-162, 1e-155, 1e-150, 1e-140]


def _check(ctx, m, scale, c):
    d, e = np.zeros(m), np.full(m, c)
    d[-1] = 1.0
    e[m - 1:] = 0.0
    d, e = d * scale, e * scale
    lam, Z = (t.cpu().numpy()[0] for t in ctx.stedc(torch.as_tensor(d).cuda(), torch.as_tensor(e).cuda()))
    T = np.diag(d / scale) + np.diag(e[:-1] / scale, 1) + np.diag(e[:-1] / scale, -1)
    ref = np.linalg.eigvalsh(T)
    u = 2.0 ** -53
    assert np.abs(lam / scale - ref).max() <= 8 * m * u
    assert np.abs(Z.T @ Z - np.eye(m)).max() <= 16 * m * u
    assert np.abs(T @ Z - Z * (lam / scale)).max() <= 16 * m * u


@pytest.mark.parametrize("c", C)
@pytest.mark.parametrize("scale", [1.0, 1e100, 1e-100])
@pytest.mark.parametrize("m", [3, 7, 16])
def test_tiny_couplings(ctx, m, scale, c):
    _check(ctx, m, scale, c)


@pytest.mark.parametrize("c", C)
@pytest.mark.parametrize("scale", [1.0, 1e100, 1e-100])
@pytest.mark.parametrize("m", [17, 40, 70, 300])
def test_tiny_blocks_beside_a_large_one(ctx, m, scale, c):
    """Merges whose whole spectrum lies far below the rest of T."""
    _check(ctx, m, scale, c)
