"""What a bound on the device waits covers, as the header states it: with a bound set the eigensolver
runs over its grid barrier at every size (by default up to 64 columns run in one cluster, whose
hardware barrier has no limit), and the panel factorisation, a cluster always, has no wait to run out."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu


def _herm(m):
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    return 0.5 * (A + A.conj().T)


@pytest.mark.parametrize("m", [30, 64])
def test_small_eigenproblems_have_bounded_waits_once_a_bound_is_set(m):
    A = _herm(m)
    with cb.Solver(256, 130) as s:
        cb.chfsi_set_wait_limit(s.ctx, 1)
        with pytest.raises(cb.ChfsiError) as e:
            cb.chfsi_heev(s.ctx, torch.from_numpy(A).cuda())
        assert e.value.code == cb.CHFSI_ETIMEOUT
        for limit in (10 ** 7, 0):  # over the grid, in a cluster
            cb.chfsi_set_wait_limit(s.ctx, limit)
            w, _ = cb.chfsi_heev(s.ctx, torch.from_numpy(A).cuda())
            assert np.max(np.abs(w.cpu().numpy() - np.linalg.eigvalsh(A))) <= 40 * m * 2.0 ** -53 * np.linalg.norm(A)


def test_factorisation_under_the_smallest_bound():
    n = 200  # FP64 products: the panel kernel and its inverse have no bounded wait
    A = _herm(n)
    B = A @ A / n + np.eye(n)
    with cb.Solver(n, 130, precision=0) as s:
        cb.chfsi_set_wait_limit(s.ctx, 1)
        L = cb.chfsi_cholesky(s.ctx, torch.from_numpy(B).cuda()).cpu().numpy()
    assert np.linalg.norm(L @ L.conj().T - B) <= 8 * n * 2.0 ** -53 * np.linalg.norm(B)
