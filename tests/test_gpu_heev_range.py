"""The FP64 Jacobi eigensolver over the range of FP64: entries near its ends scale like any other matrix
(results equal those of the matrix scaled by a power of two, bit for bit, where nothing is subnormal),
and a matrix with a NaN or infinity has NaN results in every place, none left from a call before."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu


def _matrix(m):
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    return 0.5 * (A + A.conj().T)


@pytest.mark.parametrize("m", [9, 100])
@pytest.mark.parametrize("power", [-1000, -600, 600, 1015])
def test_powers_of_two_near_the_ends_of_the_range(m, power):
    A = _matrix(m)  # entries below 2^3
    with cb.Solver(160, 160) as s:
        w0, V0 = (x.cpu().numpy() for x in cb.chfsi_heev(s.ctx, torch.from_numpy(A).cuda()))
        w, V = (x.cpu().numpy() for x in cb.chfsi_heev(s.ctx, torch.from_numpy(np.ldexp(1.0, power) * A).cuda()))
    assert np.array_equal(w, np.ldexp(w0, power)) and np.array_equal(V, V0)


@pytest.mark.parametrize("m", [9, 100])
def test_subnormal_entries(m):
    A = _matrix(m)
    A = np.round(A * 2.0 ** 30)  # integers, units of the smallest subnormal below
    with cb.Solver(160, 160) as s:
        w0, V0 = (x.cpu().numpy() for x in cb.chfsi_heev(s.ctx, torch.from_numpy(A).cuda()))
        w, V = (x.cpu().numpy() for x in cb.chfsi_heev(s.ctx, torch.from_numpy(A * 2.0 ** -537 * 2.0 ** -537).cuda()))
    assert np.array_equal(V, V0) and np.max(np.abs(w * 2.0 ** 537 * 2.0 ** 537 - w0)) <= 0.5


@pytest.mark.parametrize("m", [9, 100])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("at", [(0, 0), (3, 5)])
def test_no_finite_result_for_a_matrix_that_is_not(m, bad, at):
    A = _matrix(m)
    with cb.Solver(160, 160) as s:
        cb.chfsi_heev(s.ctx, torch.from_numpy(A).cuda())
        B = A.copy()
        B[at] = B[at[::-1]] = bad
        w, V = (x.cpu().numpy() for x in cb.chfsi_heev(s.ctx, torch.from_numpy(B).cuda()))
        assert np.all(np.isnan(w)) and np.all(np.isnan(V))
        w, _ = cb.chfsi_heev(s.ctx, torch.from_numpy(A).cuda())
    assert np.max(np.abs(w.cpu().numpy() - np.linalg.eigvalsh(A))) <= 40 * m * 2.0 ** -53 * np.linalg.norm(A)
