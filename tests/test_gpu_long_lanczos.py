"""Lanczos runs of thousands of steps, as many as the context's options allow: a Gram-Schmidt pass takes
1024 coefficients at a time and the tridiagonal matrix is in shared memory up to 2048 rows (all of
either beyond 14,500 would fit no shared memory).  A diagonal matrix with known extremes: the FP32
product (entries truncated, one term a row) is off by 2^-22 of its norm at most, and a run of n steps
has the whole spectrum."""
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1025, 2049, 3070])
def test_extremes_after_n_steps(n):
    d = torch.linspace(-1.0, 3.0, n, dtype=torch.float64, device="cuda")
    H = cb.fortran_empty(n, n, d.device)
    H.zero_()
    H.diagonal().copy_(d)
    v = torch.ones(n, dtype=torch.complex128, device="cuda")
    with cb.Solver(n, 1, lanczos_k_cold=n) as s:
        _, lo, hi = cb.chfsi_lanczos(s.ctx, H, n, v)
    assert abs(lo + 1.0) <= 4 * 2.0 ** -22 and abs(hi - 3.0) <= 4 * 2.0 ** -22
