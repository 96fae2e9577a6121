"""Slice pairs of the tensor-core digit products, one pair at a time and exactly.

Every entry of H and Y but one anchor per row and column is a single digit at a chosen slice, so
that the product is a sum of one slice pair per column whose value fits FP32 exactly: a pair that
is missing, counted twice, added at another level or taken from another K-block, row or column
changes the result.  Sizes sit at the edges of row tiles (128), column tiles (16 .. 64 wide),
K-blocks (64), exact chunks (6 to 15 K-blocks) and of the one- and two-region issue loops."""
import numpy as np
import pytest
import torch

from paper_1206_3768_gb300 import binding as cb

pytestmark = pytest.mark.gpu

CASES = [(n, m, S)
         for S in range(1, 9)
         for n, m in [(63, 1), (129, 17), (448, 48), (500, 64), (961, 65), (1025, 130)]]


@pytest.mark.parametrize("n,m,S", CASES)
def test_every_kept_slice_pair_is_exact(n, m, S):
    rng = np.random.Generator(np.random.PCG64([n, m, S]))
    d = np.triu(rng.integers(-63, 64, (n, n)))
    d = d + np.triu(d, 1).T
    f = rng.integers(-63, 64, (n, m))
    with cb.Solver(max(n, 200), m) as s:
        for ss in range(1, S + 1):
            t = 1 + (np.arange(m) % (S + 1 - ss))  # slice of each column: the pair is kept
            H = d * 2.0 ** (1 - 7 * ss)            # the anchors set the scale 2^1 of every row
            H[0, :] = H[:, 0] = 1.0
            H[1, :] = H[:, 1] = 0.0
            H[0, 1] = H[1, 0] = 0.0
            Y = f * 2.0 ** (1.0 - 7 * t)[None, :]
            Y[0, :] = 0.0
            Y[1, :] = 1.0                          # meets the zero column of H
            # degree 1 on [-1, 1] normalised at -2: out = -H Y / 2
            out = cb.chfsi_filter_split(s.ctx, torch.from_numpy(H).to(torch.complex128).cuda(),
                                        torch.from_numpy(Y).to(torch.complex128).cuda(), [1] * m, -2.0, -1.0, 1.0, S)
            want = -0.5 * (H @ Y)                  # integers below 2^53 times one power of two
            got = out.cpu().numpy()
            assert np.array_equal(got.real, want) and not got.imag.any(), (ss, np.max(np.abs(got - want)))
