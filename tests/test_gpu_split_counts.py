"""The split counts measured for the products of one context under another with less room for split
partials (partials hold 32 splits of a block, so a narrow context holds one split of an n x n
product where a wide one holds ten)."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1088, 1152, 1280, 1472, 1664])
def test_a_narrow_context_reduces_after_a_wide_one(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.view_as_complex(torch.randn(n, n, 2, dtype=torch.float64, device="cuda", generator=g))
    A = A + A.mH
    L = torch.tril(A) / (4.0 * n) + 2.0 * torch.eye(n, dtype=A.dtype, device="cuda")
    L.diagonal().imag.zero_()
    H = []
    for blk in (512, 16):
        with cb.Solver(n, blk) as s:
            H.append(cb.chfsi_reduce(s.ctx, A, L))
    # the same sums in other pieces: both within the reduction's error of n u cond(L)^2 ||H||
    u = 2.0 ** -53
    assert float(torch.linalg.norm(H[0] - H[1])) <= 2 * n * u * float(np.linalg.cond(L.cpu().numpy())) ** 2 * float(
        torch.linalg.norm(H[0]))
