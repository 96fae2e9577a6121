"""Re-orthonormalisation in plain FP64 past the width from which the triangular inverse solves its columns
in place instead of in shared memory (1500 rows; a column and its reciprocals beyond 7168 rows fit
no shared memory).  Cholesky QR twice: || Q^H Q - I ||_F within 8 n u sqrt(m), the rounding of m inner
products of length n per column; Q spans the columns of Y (of norm below 4)."""
import torch
import pytest

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def test_orthonormalize_past_the_inverse_s_shared_memory_form():
    n, m = 1510, 1501
    g = torch.Generator(device="cuda").manual_seed(m)
    Y = torch.view_as_complex(torch.randn(n, m, 2, dtype=torch.float64, device="cuda", generator=g)) / n ** 0.5 / 2
    Y[:m] += 2.0 * torch.eye(m, dtype=Y.dtype, device="cuda")
    with cb.Solver(n, m, precision=0) as s:
        Q = cb.chfsi_orthonormalize(s.ctx, Y, None)
    eye = torch.eye(m, dtype=Y.dtype, device="cuda")
    assert float(torch.linalg.norm(Q.mH @ Q - eye)) <= 8 * n * U * m ** 0.5
    assert float(torch.linalg.norm(Y - Q @ (Q.mH @ Y))) <= 8 * n * U * m ** 0.5 * 4
