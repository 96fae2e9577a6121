"""Blocked factorisation at the edges of its blocks: 16-column steps and 128-column panels of the
diagonal kernel, outer panels of 512, halves of the triangular inverse.  Backward errors against
the inputs in FP64: 8 n u relative to the norms (the standard bound of Cholesky and of products
with a triangular inverse, with room for the digit products' 2^-48)."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
SIZES = [1, 15, 16, 17, 33, 112, 127, 128, 129, 144, 255, 257, 384, 511, 513, 641, 700]


def _cgauss(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / np.sqrt(2.0)


def _hpd(rng, n):
    G = _cgauss(rng, n, n)
    return G.conj().T @ G / n + 0.5 * np.eye(n)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", SIZES)
def test_cholesky_and_reduction_at_block_edges(n, precision):
    rng = np.random.default_rng(n)
    B = _hpd(rng, n)
    A = _cgauss(rng, n, n)
    A = A + A.conj().T
    junk = np.triu(np.full((n, n), np.nan), 1)  # the upper triangles are not read
    with cb.Solver(700, 160, precision=precision) as s:
        L = cb.chfsi_cholesky(s.ctx, torch.from_numpy(np.tril(B) + junk).cuda()).cpu().numpy()
        assert not np.triu(L, 1).any()
        assert np.linalg.norm(L @ L.conj().T - B) <= 8 * n * U * np.linalg.norm(B)
        Lc = torch.from_numpy(np.tril(L) + junk).cuda()
        H = cb.chfsi_reduce(s.ctx, torch.from_numpy(np.tril(A) + junk).cuda(), Lc).cpu().numpy()
        k = np.linalg.cond(L)
        assert np.linalg.norm(L @ H @ L.conj().T - A) <= 8 * n * U * k * k * np.linalg.norm(A)


@pytest.mark.parametrize("bad", [0, 15, 16, 130, 300])
def test_failed_pivot_is_named(bad):
    n = 400
    B = np.eye(n, dtype=complex)
    B[bad, bad] = -1.0
    with cb.Solver(n, 130) as s:
        with pytest.raises(cb.ChfsiError, match=rf"pivot {bad}\b") as e:
            cb.chfsi_cholesky(s.ctx, torch.from_numpy(B).cuda())
        assert e.value.code == cb.CHFSI_ENOTPD
        L = cb.chfsi_cholesky(s.ctx, torch.eye(n, dtype=torch.complex128).cuda())
        assert torch.equal(L.cpu(), torch.eye(n, dtype=torch.complex128))
