"""Lanczos at the block edges of its product (256 and 512 entries of a row, one step or many) and of
its vector kernels (64 rows, four lanes a row), and the FP64 product at shapes that take each of its
tiles (64 x 32, 32 x 16, 16 x 8) with one and several K splits.

Bounds.  A Lanczos run of k steps on H v with relative error eps per product moves the extreme
values of T_k by at most k eps ||H||: eps = 2^-22 sqrt(n) for the FP32 form (truncated operands, sums
of eight), n 2^-52 for FP64.  A product entry is off by at most (K + 4) 2^-52 sum |a||b| times 3 (three
real products)."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu

U = 2.0 ** -52


def _cgauss(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / np.sqrt(2.0)


def _lanczos(H, v, k):
    V = [v / np.linalg.norm(v)]
    al, be = [], []
    for j in range(k):
        w = H @ V[j]
        al.append(np.vdot(V[j], w).real)
        Q = np.stack(V, 1)
        for _ in range(2):
            w = w - Q @ (Q.conj().T @ w)
        be.append(np.linalg.norm(w))
        V.append(w / be[-1])
    th = np.linalg.eigvalsh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
    return th[-1] + be[-1], th[0], th[-1]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,k", [(33, 1), (64, 2), (65, 5), (255, 8), (256, 8), (257, 8), (511, 10), (513, 10),
                                 (768, 40), (1025, 33)])
def test_lanczos_at_block_edges(n, k, precision):
    rng = np.random.default_rng([n, k])
    H = _cgauss(rng, n, n)
    H = (H + H.conj().T) * 3.0
    v = _cgauss(rng, n)
    want = _lanczos(H, v, k)
    with cb.Solver(1100, 130, precision=precision) as s:
        got = cb.chfsi_lanczos(s.ctx, torch.from_numpy(H).cuda(), k, torch.from_numpy(v).cuda())
    eps = 2.0 ** -22 * np.sqrt(n) if precision else n * U
    assert np.max(np.abs(np.array(got) - want)) <= k * eps * np.linalg.norm(H, 2)


@pytest.mark.parametrize("scale", [1e-100, 1e-3, 1e100])
def test_extremes_of_scaled_diagonals(scale):
    # FP64 form; a diagonal matrix and a start vector over a few entries: T_k has their values
    d = np.linspace(-1.0, 3.0, 200) * scale
    v = np.zeros(200, complex)
    v[[0, 50, 199]] = [1.0, 1.0j, -1.0]
    with cb.Solver(200, 130, precision=0) as s:
        _, lo, hi = cb.chfsi_lanczos(s.ctx, torch.from_numpy(np.diag(d).astype(complex)).cuda(), 3,
                                     torch.from_numpy(v).cuda())
    assert abs(lo - d[0]) <= 1e-13 * scale and abs(hi - d[199]) <= 1e-13 * scale


SHAPES = [(30, 30, 512), (512, 30, 30), (30, 30, 31), (1, 1, 7), (17, 9, 33), (16, 8, 32), (15, 7, 65), (100, 30, 512),
          (33, 17, 1000), (200, 100, 50), (640, 64, 640), (700, 130, 90), (64, 32, 16), (129, 65, 257)]


@pytest.mark.parametrize("opa", ["N", "C"])
@pytest.mark.parametrize("opb", ["N", "C"])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_fp64_product_tiles_and_splits(M, N, K, opa, opb):
    rng = np.random.default_rng([M, N, K])
    A = _cgauss(rng, *((M, K) if opa == "N" else (K, M)))
    B = _cgauss(rng, *((K, N) if opb == "N" else (N, K)))
    C = _cgauss(rng, M, N)
    a = A if opa == "N" else A.conj().T
    b = B if opb == "N" else B.conj().T
    with cb.Solver(700, 160) as s:
        got = cb.chfsi_zgemm(s.ctx, opa, opb, 0.7, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), -1.3,
                             torch.from_numpy(C).cuda()).cpu().numpy()
    want = 0.7 * (a @ b) - 1.3 * C
    bound = 3 * (K + 4) * U * (2 * np.abs(a) @ np.abs(b) + np.abs(C))
    assert np.all(np.abs(got - want) <= bound)


@pytest.mark.parametrize("M,N,K", [(427, 59, 427), (562, 12, 562), (700, 30, 1100)])
def test_fp64_product_sums_in_short_pieces(M, N, K):
    # Sums of K positive terms.  One after another their rounding errors add up to about U / 2 sqrt(K) / 3
    # of the sum (3.4 U at K = 427, 5.5 U at 1100); in S pieces of at most 128 terms to U / 2
    # (sqrt(128 / S) / 3 + sqrt(S) / 3), below 1.5 U for S = 4 .. 18.
    rng = np.random.default_rng([M, N, K])
    a, b = rng.uniform(0.5, 1.0, (M, K)), rng.uniform(0.5, 1.0, (K, N))
    with cb.Solver(1100, 130, precision=0) as s:
        got = cb.chfsi_zgemm(s.ctx, "N", "N", 1.0, torch.from_numpy(a.astype(complex)).cuda(),
                             torch.from_numpy(b.astype(complex)).cuda(), 0.0,
                             torch.zeros(M, N, dtype=torch.complex128).cuda()).cpu().numpy().real
    want = np.matmul(a.astype(np.longdouble), b.astype(np.longdouble))
    assert np.sqrt(np.mean(((got - want) / want) ** 2)) <= 1.5 * U
