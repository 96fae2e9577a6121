"""Whole solves whose Rayleigh-Ritz blocks are wide enough for the double-float eigensolver (512 columns
by default).  That they reach it is shown by the same sequence in a process that sets the threshold
above the block (CHFSI_JACOBI_DF_MIN, read once per process): with split counts not measured, a
sequence repeats bit for bit within a process, and the FP64 eigensolver gives other bits."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_1206_3768_gb300 import binding as cb  # noqa: E402
from paper_1206_3768_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


def _sequence():
    return inputs.planted_sequence("c5", n=1100, N=1, nev=400, blk=520, device="cuda", keep_vectors=False)


def _solve(seq):
    As = [cb.fortran(torch.tril(p.A)) for p in seq.problems]
    Bs = [cb.fortran(torch.tril(p.B)) for p in seq.problems]
    with cb.Solver(seq.n, seq.blk, deg_min=seq.deg_min, deg_max=seq.deg_max) as s:
        return cb.chfsi_solve_sequence(s.ctx, As, Bs, seq.nev, seq.blk, seq.deg, seq.tol)


def test_solve_with_blocks_in_the_double_float_eigensolver(tmp_path):
    seq = _sequence()
    evals, evecs, stats = _solve(seq)
    scale = max(float(np.max(np.abs(p.lam))) for p in seq.problems)
    for ell, p in enumerate(seq.problems):
        lam = evals[ell]
        assert stats[ell]["converged"] == seq.nev
        assert np.max(np.abs(lam.numpy() - p.lam[:seq.nev])) <= 1e-10 * scale
        A, B, X = p.A, p.B, evecs[ell]
        R = A @ X - (B @ X) * lam.to(A.device).to(torch.complex128)[None, :]
        assert float((torch.linalg.vector_norm(R, dim=0) / torch.linalg.vector_norm(X, dim=0)).max()) <= 1e-10 * scale
        E = X.mH @ (B @ X) - torch.eye(seq.nev, dtype=torch.complex128, device=A.device)
        assert float(E.abs().max()) < 1e-10
    runs = {}
    for name, threshold in (("double-float", {}), ("fp64", {"CHFSI_JACOBI_DF_MIN": str(seq.blk + 1)})):
        out = tmp_path / f"{name}.npz"
        subprocess.run([sys.executable, os.path.abspath(__file__), str(out)], check=True, timeout=300,
                       env={**os.environ, "CHFSI_OZ_AUTOTUNE": "0", **threshold})
        runs[name] = np.load(out)
        assert np.array_equal(runs[name]["first"], runs[name]["again"])
    a, b = runs["double-float"], runs["fp64"]
    assert np.array_equal(a["inputs"], b["inputs"])
    assert not np.array_equal(a["first"], b["first"]) and np.max(np.abs(a["first"] - b["first"])) <= 1e-10 * scale


if __name__ == "__main__":
    seq_ = _sequence()
    np.savez(sys.argv[1], inputs=np.stack([x.cpu().numpy() for p_ in seq_.problems for x in (p_.A, p_.B)]),
             **{k: np.stack([e.numpy() for e in _solve(seq_)[0]]) for k in ("first", "again")})
