"""Blocked factorisation where its panel products change form: from 1024 rows below a 128-column panel
(n = 1152) the panel is multiplied in place by digit products (operands sliced before the result is
written), below through a copy in FP64; one and two panels in place.  Backward errors against the
inputs in FP64, 8 n u relative to the norms (the bound of the smaller sizes' test)."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _cgauss(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / np.sqrt(2.0)


@pytest.mark.parametrize("n", [1151, 1152, 1153, 1281])
def test_cholesky_and_reduction_around_the_first_panel_in_place(n):
    rng = np.random.default_rng(n)
    G = _cgauss(rng, n, n)
    B = G.conj().T @ G / n + 0.5 * np.eye(n)
    A = _cgauss(rng, n, n)
    A = A + A.conj().T
    junk = np.triu(np.full((n, n), np.nan), 1)  # the upper triangles are not read
    with cb.Solver(1281, 160) as s:
        L = cb.chfsi_cholesky(s.ctx, torch.from_numpy(np.tril(B) + junk).cuda()).cpu().numpy()
        assert not np.triu(L, 1).any()
        assert np.linalg.norm(L @ L.conj().T - B) <= 8 * n * U * np.linalg.norm(B)
        H = cb.chfsi_reduce(s.ctx, torch.from_numpy(np.tril(A) + junk).cuda(),
                            torch.from_numpy(np.tril(L) + junk).cuda()).cpu().numpy()
    k = np.linalg.cond(L)
    assert np.linalg.norm(L @ H @ L.conj().T - A) <= 8 * n * U * k * k * np.linalg.norm(A)
