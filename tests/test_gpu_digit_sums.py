"""Sums of digit products past 2^24 on every level: the chunks of a level add into double-float sums
without rounding while high and low word hold the value (48 bits), the smallest levels among them."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,ss", [(6, 4), (7, 3), (7, 4), (7, 6), (8, 5), (8, 8)])
def test_long_sums_of_one_level_are_exact(S, ss):
    # one digit per entry (slice ss of H, the highest kept slices of Y), all products positive: an
    # entry is an odd or even integer up to 2^24.1 times one power of two, exact in FP64 here
    n, m = 4600, 6
    rng = np.random.default_rng([S, ss])
    d = np.triu(rng.integers(61, 64, (n, n)))
    d = d + np.triu(d, 1).T
    t = np.maximum(1, S + 1 - ss - np.arange(m) % 3)
    H = d * 2.0 ** (1 - 7 * ss)   # the anchors set the scale 2^1 of every row and column
    H[0, :] = H[:, 0] = 1.0
    H[1, :] = H[:, 1] = 0.0
    H[0, 1] = H[1, 0] = 0.0
    Y = rng.integers(61, 64, (n, m)) * 2.0 ** (1.0 - 7 * t)[None, :]
    Y[0, :] = 0.0
    Y[1, :] = 1.0
    with cb.Solver(n, m) as s:
        # degree 1 on [-1, 1] normalised at -2: out = -H Y / 2
        out = cb.chfsi_filter_split(s.ctx, torch.from_numpy(H).to(torch.complex128).cuda(),
                                    torch.from_numpy(Y).to(torch.complex128).cuda(), [1] * m, -2.0, -1.0, 1.0, S)
    got, want = out.cpu().numpy(), -0.5 * (H @ Y)
    assert np.array_equal(got.real, want) and not got.imag.any(), np.max(np.abs(got - want) / np.abs(want).max(0))
