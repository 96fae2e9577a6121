"""The FP64 Jacobi eigensolver where its work division changes: one cluster up to 32 pairs, a grid of
one CTA per pair up to the number of SMs, several rows and blocks per CTA above, rotations formed
ahead or after the barrier (128 pairs), odd and even pair counts; and its scaling by powers of two.
Bounds: each of the m rotations an entry meets in a sweep adds a few ulps, over about ten sweeps."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _check(s, A, scale=1.0):
    m = A.shape[0]
    w, V = (x.cpu().numpy() for x in cb.chfsi_heev(s.ctx, torch.from_numpy(A * scale).cuda()))
    nrm = np.linalg.norm(A)
    ref = np.linalg.eigvalsh(A)
    assert np.all(np.diff(w) >= 0)
    assert np.max(np.abs(w / scale - ref)) <= 40 * m * U * nrm
    assert np.linalg.norm(V.conj().T @ V - np.eye(m)) <= 40 * m * U * np.sqrt(m)
    assert np.linalg.norm(A @ V - V * (w / scale)) <= 40 * m * U * nrm


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 17, 31, 33, 62, 63, 65, 66, 81, 129, 255, 257, 303, 305, 307])
@pytest.mark.parametrize("kind", ["random", "near"])
def test_heev_at_the_edges_of_its_work_division(m, kind):
    rng = np.random.default_rng([m, kind == "near"])
    A = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    A = 0.5 * (A + A.conj().T)
    if kind == "near":
        A = np.diag(np.sort(rng.uniform(-2.0, 2.0, m))) + 1e-4 * A
    with cb.Solver(320, 320) as s:
        _check(s, A)


@pytest.mark.parametrize("m", [10, 150])
@pytest.mark.parametrize("power", [-300, -40, 40, 300])
def test_heev_scales(m, power):
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    with cb.Solver(160, 160) as s:
        _check(s, 0.5 * (A + A.conj().T), 2.0 ** power)


def test_heev_of_diagonal_and_zero_matrices():
    with cb.Solver(160, 160) as s:
        for m in (7, 100):
            d = np.random.default_rng(m).standard_normal(m)
            for A in (np.diag(d).astype(complex), np.zeros((m, m), complex), np.eye(m, dtype=complex)):
                w, V = (x.cpu().numpy() for x in cb.chfsi_heev(s.ctx, torch.from_numpy(A).cuda()))
                assert np.array_equal(w, np.sort(A.diagonal().real))
                assert np.array_equal(np.abs(V).sum(0), np.ones(m)) and np.array_equal(A @ V, V * w)


@pytest.mark.parametrize("m", [15, 37, 64, 97, 217])
def test_heev_leaves_no_more_than_its_threshold(m):
    # close eigenvalues turn what is left off the diagonal of V^H A V into eigenvector errors.  A pair is
    # rotated while it is above 1e-16 ||A||_F, so the mean square stays below that; V^H (A V) itself is
    # evaluated to about 2 U ||A||_2, of the order of 2 U ||A||_F / sqrt(m) here (all eigenvalues near -1)
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    A = np.diag(-1.0 + 0.05 * rng.uniform(size=m)) + 0.5e-7 * (A + A.conj().T)
    with cb.Solver(320, 320) as s:
        V = cb.chfsi_heev(s.ctx, torch.from_numpy(A).cuda())[1].cpu().numpy()
    left = V.conj().T @ (A @ V)
    np.fill_diagonal(left, 0.0)
    assert np.linalg.norm(left) / m <= (1e-16 + 2 * U / np.sqrt(m)) * np.linalg.norm(A)
