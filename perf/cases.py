"""Performance cases of the eigensolver library: the calls its users make, over the sizes they
make them with.

Whole solves of a warm-started sequence go through chfsi_solve_sequence; the other cases are the
steps of one solve through their own entry points (the Chebyshev filter above all, which takes
most of the time of a solve), for callers that assemble their own loop.  Inputs are planted: a
Hermitian matrix H = U diag(lam) U^H whose dense unitary U is a product of discrete Fourier
transforms and random phases, so that it is built in O(n^2 log n) operations and its eigenpairs
are known.  Every matrix is complex128 and column-major on the GPU, as a program has it that
calls this library; the context is the program's own, kept over its calls.
"""
import math

import torch

from paper_1206_3768_gb300 import binding as cb

DEV = "cuda"
Z = torch.complex128
TOL = 1e-10


# ---------------------------------------------------------------- cases
def listed():
    return [
        # smallest whole sequence of the test workloads (three correlated problems, the first
        # cold): bound by launches, read-backs and the small dense steps
        dict(name="solve_n512", kind="solve", n=512, nev=20, blk=30, deg=10, N=3),
        # one small k-point of the batched workload (nev = 4 % of n, blk = 1.3 nev), its cold
        # problem and one warm one
        dict(name="solve_n3039", kind="solve", n=3039, nev=122, blk=159, deg=20, N=2),
        # the filter of the benchmark's n = 9300 workload at its full block: one loop's products
        dict(name="filter_n9300_m320", kind="filter", n=9300, m=320, deg_min=20, deg_max=20, slices=7),
        # the n = 2600 workload's adaptive degrees (8 to 25 per column, so that the active width
        # shrinks within a loop) at an intermediate accuracy
        dict(name="filter_n2600_m130", kind="filter", n=2600, m=130, deg_min=8, deg_max=25, slices=5),
        # late loop of a large k-point: most columns are locked, a narrow odd block remains
        dict(name="filter_n5957_m37", kind="filter", n=5957, m=37, deg_min=20, deg_max=20, slices=7),
        # the smallest call: a few columns of a small problem, where launches count
        dict(name="filter_n256_m16", kind="filter", n=256, m=16, deg_min=10, deg_max=10, slices=7),
        # the plain FP64 option (precision 0)
        dict(name="filter_fp64_n1024_m64", kind="filter", n=1024, m=64, deg_min=10, deg_max=10, slices=0),
        # factorisation of a new overlap matrix, once per sequence (n = 2600 workload)
        dict(name="cholesky_n2600", kind="cholesky", n=2600, cond=1e4),
        # reduction to standard form, once per problem
        dict(name="reduce_n4096", kind="reduce", n=4096, cond=3.0),
        # upper spectral bound of a cold problem (40 steps)
        dict(name="lanczos_n9300", kind="lanczos", n=9300, k=40),
        # re-orthonormalisation of a filtered block against the locked columns, mid-solve
        dict(name="orthonormalize_n9300_m192", kind="orthonormalize", n=9300, m=192, k=128),
        # Rayleigh-Ritz step of a mean k-point's full block
        dict(name="rayleigh_ritz_n4500_m234", kind="rayleigh_ritz", n=4500, m=234),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "filter", "filter", "filter", "filter_fp64", "cholesky", "reduce", "lanczos",
                       "orthonormalize", "rayleigh_ritz"])
    if kind == "solve":
        n = _log_int(rng, 256, 3000)
        nev = max(8, math.ceil(0.04 * n))
        return dict(kind="solve", n=n, nev=nev, blk=math.ceil(1.5 * nev), deg=rng.randint(12, 20), N=2)
    if kind == "filter":
        n = _log_int(rng, 200, 8000)
        lo = rng.randint(4, 20)
        return dict(kind="filter", n=n, m=_log_int(rng, 8, min(320, n // 4)), deg_min=lo,
                    deg_max=min(25, lo + rng.choice([0, 0, 7, 15])), slices=rng.randint(4, 7))
    if kind == "filter_fp64":
        n = _log_int(rng, 200, 1400)
        return dict(kind="filter", n=n, m=_log_int(rng, 8, 96), deg_min=8, deg_max=rng.randint(8, 12), slices=0)
    if kind == "cholesky":
        return dict(kind="cholesky", n=_log_int(rng, 200, 4000), cond=rng.choice([3.0, 100.0, 1e4]))
    if kind == "reduce":
        return dict(kind="reduce", n=_log_int(rng, 200, 4096), cond=rng.choice([3.0, 100.0, 1e4]))
    if kind == "lanczos":
        return dict(kind="lanczos", n=_log_int(rng, 200, 9300), k=rng.choice([10, 20, 40]))
    if kind == "orthonormalize":
        n = _log_int(rng, 400, 9300)
        return dict(kind="orthonormalize", n=n, m=_log_int(rng, 12, min(320, n // 4)),
                    k=rng.choice([0, _log_int(rng, 8, min(256, n // 4))]))
    n = _log_int(rng, 256, 5000)
    return dict(kind="rayleigh_ritz", n=n, m=_log_int(rng, 12, min(320, n // 4)))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _randn(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device=DEV, generator=g)) / math.sqrt(2.0)


def _uniform(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, dtype=torch.float64, device=DEV, generator=g)


def _unitary(g, n):
    """X -> U X for a dense unitary U = F P1 F P2 (F the unitary DFT, P1, P2 random phases)."""
    p1, p2 = (torch.polar(torch.ones(n, dtype=torch.float64, device=DEV), _uniform(g, n, 0.0, 2 * math.pi))
              for _ in range(2))

    def apply(X):
        for p in (p2, p1):
            X = torch.fft.fft(p[:, None] * X, dim=0, norm="ortho")
        return X

    return apply


def _conjugated(apply, M):
    """U M U^H for Hermitian M, made exactly Hermitian."""
    X = apply(apply(M).conj().T).conj().T
    return 0.5 * (X + X.conj().T)


def _spectrum(g, n):
    """The test workloads' spectrum, 95 % spread over [-2, 2] and 5 % within 1e-3 of -1, ascending;
    neighbours repel as the levels of a Hermitian matrix do, so that every wanted vector is defined."""
    nc = max(1, round(0.05 * n))
    k = n - nc
    spread = -2.0 + 4.0 * (torch.arange(k, dtype=torch.float64, device=DEV) + _uniform(g, k, 0.15, 0.85)) / k
    return torch.sort(torch.cat([spread, _uniform(g, nc, -1.001, -0.999)])).values


def _planted(g, n):
    """(H, its ascending eigenvalues, X -> U X): column j of U belongs to eigenvalue j."""
    lam = _spectrum(g, n)
    U = _unitary(g, n)
    return _conjugated(U, torch.diag(lam).to(Z)), lam, U


def _columns(U, n, j0, j1):
    E = torch.zeros(n, j1 - j0, dtype=Z, device=DEV)
    E[j0:j1] = torch.eye(j1 - j0, dtype=Z, device=DEV)
    return U(E)


def _overlap(g, n, cond):
    """B = V diag(mu) V^H with mu spread over [1, cond] (logarithmically)."""
    mu = torch.exp(_uniform(g, n, 0.0, math.log(cond)))
    return _conjugated(_unitary(g, n), torch.diag(mu).to(Z))


def _gauge_vector(g, n):
    return _randn(g, n)


def _fix_gauge(r, X, *more):
    """Eigenvectors are defined up to a phase: makes r^H x_j real and positive for every column."""
    c = r.conj() @ X
    ph = (c.conj() / c.abs())[None, :]
    return [x * ph for x in (X, *more)]


def _inputs(case, seed):
    """The arrays of a case, from the seed alone."""
    g, n, kind = _gen(seed), case["n"], case["kind"]
    if kind == "solve":
        B = _overlap(g, n, 3.0)
        L = torch.linalg.cholesky(B)
        lam, U = _spectrum(g, n), _unitary(g, n)
        d = dict(B=B, A=[], lam=[], X=[], r=_gauge_vector(g, n))
        turns = []  # eigenvectors turn by about 1e-2 from one problem to the next, then half of that
        for l in range(case["N"]):
            if l:
                # eigenvalues drift by about 1e-3
                lam = (1.0 + 1e-3 * float(_uniform(g, 1, -1.0, 1.0))) * lam + 1e-3 * float(_uniform(g, 1, -1.0, 1.0))
                turns.append(torch.polar(torch.ones(n, dtype=torch.float64, device=DEV),
                                         0.5**l * 1e-2 * torch.randn(n, dtype=torch.float64, device=DEV, generator=g)))

            def V(X, turns=tuple(turns)):
                X = U(X)
                for t in turns:
                    X = torch.fft.ifft(t[:, None] * torch.fft.fft(X, dim=0, norm="ortho"), dim=0, norm="ortho")
                return X

            A = L @ _conjugated(V, torch.diag(lam).to(Z)) @ L.conj().T
            d["A"].append(0.5 * (A + A.conj().T))
            d["lam"].append(lam[: case["nev"]])
            d["X"].append(torch.linalg.solve_triangular(L.conj().T, _columns(V, n, 0, case["nev"]), upper=True))
        return d
    if kind == "filter":
        H, lam, U = _planted(g, n)
        m = case["m"]
        # carried vectors: near the lowest eigenvectors, with a part in all others
        Y = _columns(U, n, 0, m) + 0.1 / math.sqrt(n) * _randn(g, n, m)
        degs = torch.randint(case["deg_min"], case["deg_max"] + 1, (m,), device=DEV, generator=g).tolist()
        return dict(H=H, Y=Y, degs=degs, a0=float(lam[0]), a=float(lam[m]), b=2.02)
    if kind == "cholesky":
        return dict(B=_overlap(g, n, case["cond"]))
    if kind == "reduce":
        return dict(A=_planted(g, n)[0], L=torch.linalg.cholesky(_overlap(g, n, case["cond"])))
    if kind == "lanczos":
        return dict(H=_planted(g, n)[0], v0=_randn(g, n))
    if kind == "orthonormalize":
        m, k = case["m"], case["k"]
        U = _unitary(g, n)
        # a filtered block: columns of very different length near orthogonal directions, each
        # with a part of the others, of the locked columns and of everything else
        Y = _columns(U, n, k, k + m) + 0.05 / math.sqrt(n) * _randn(g, n, m)
        Y = Y @ (torch.eye(m, dtype=Z, device=DEV) + 0.2 / math.sqrt(m) * _randn(g, m, m))
        Y = Y * torch.exp(_uniform(g, m, -3.0, 3.0))[None, :]
        return dict(Y=Y, YL=_columns(U, n, 0, k) if k else None)
    if kind == "rayleigh_ritz":
        H, lam, U = _planted(g, n)
        m = case["m"]
        # an orthonormal basis near the lowest eigenvectors, as after filter and QR
        Y = torch.linalg.qr(_columns(U, n, 0, m) + 0.03 / math.sqrt(n) * _randn(g, n, m)).Q
        return dict(H=H, Y=Y, r=_gauge_vector(g, n))
    raise ValueError(kind)


def _widest(case):
    return max(case.get("blk", 0), case.get("m", 0), case.get("k", 0) if case["kind"] == "orthonormalize" else 0, 1)


def prepare(case, seed):
    d = _inputs(case, seed)
    st = {"case": case}
    for key, v in d.items():  # column-major, as the library's callers hold their matrices
        if isinstance(v, list) and v and isinstance(v[0], torch.Tensor):
            st[key] = [cb.fortran(x) for x in v]
        else:
            st[key] = cb.fortran(v) if isinstance(v, torch.Tensor) else v
    fp64 = case["kind"] == "filter" and case["slices"] == 0
    st["solver"] = cb.Solver(case["n"], _widest(case), precision=0 if fp64 else 1)
    return st


# ---------------------------------------------------------------- one pass
def run(st):
    case, ctx = st["case"], st["solver"].ctx
    kind = case["kind"]
    if kind == "solve":
        cb.chfsi_reset_warm_state(ctx)  # the sequence starts cold
        evals, evecs, _ = cb.chfsi_solve_sequence(ctx, st["A"], [st["B"]] * case["N"], case["nev"], case["blk"],
                                                  case["deg"], TOL)
        return {"evals": evals, "evecs": [_fix_gauge(st["r"], X)[0] for X in evecs]}
    if kind == "filter":
        if case["slices"]:
            return cb.chfsi_filter_split(ctx, st["H"], st["Y"], st["degs"], st["a0"], st["a"], st["b"], case["slices"])
        return cb.chfsi_filter(ctx, st["H"], st["Y"], st["degs"], st["a0"], st["a"], st["b"])
    if kind == "cholesky":
        return cb.chfsi_cholesky(ctx, st["B"])
    if kind == "reduce":
        return cb.chfsi_reduce(ctx, st["A"], st["L"])
    if kind == "lanczos":
        return cb.chfsi_lanczos(ctx, st["H"], case["k"], st["v0"])
    if kind == "orthonormalize":
        return cb.chfsi_orthonormalize(ctx, st["Y"], st["YL"])
    theta, Y, HY = cb.chfsi_rayleigh_ritz(ctx, st["H"], st["Y"])
    Y, HY = _fix_gauge(st["r"], Y, HY)
    return {"theta": theta, "Y": Y, "HY": HY}


def exact(case, seed):
    kind = case["kind"]
    if kind == "orthonormalize":
        return None  # any orthonormal basis of the same span is an answer
    d = _inputs(case, seed)
    if kind == "solve":
        return {"evals": torch.stack(d["lam"]), "evecs": [_fix_gauge(d["r"], X)[0] for X in d["X"]]}
    if kind == "filter":
        H, Y, degs = d["H"], d["Y"], torch.tensor(d["degs"], device=DEV)
        e, c = 0.5 * (d["b"] - d["a"]), 0.5 * (d["b"] + d["a"])
        s1 = e / (d["a0"] - c)
        out, s, prev, cur = Y.clone(), s1, None, Y
        for k in range(1, int(degs.max()) + 1):
            if k == 1:
                nxt = (s1 / e) * (H @ cur - c * cur)
            else:
                sn = 1.0 / (2.0 / s1 - s)
                nxt = (2.0 * sn / e) * (H @ cur - c * cur) - (s * sn) * prev
                s = sn
            prev, cur = cur, nxt
            out[:, degs == k] = cur[:, degs == k]
        return out
    if kind == "cholesky":
        return torch.linalg.cholesky(d["B"])
    if kind == "reduce":
        P = torch.linalg.solve_triangular(d["L"], d["A"], upper=False)
        H = torch.linalg.solve_triangular(d["L"], P.conj().T.contiguous(), upper=False)
        return 0.5 * (H + H.conj().T)
    if kind == "lanczos":
        H, k = d["H"], min(case["k"], case["n"])
        v = d["v0"] / torch.linalg.norm(d["v0"])
        V, al, be = [v], [], []
        for j in range(k):
            w = H @ V[j]
            al.append(float(torch.vdot(V[j], w).real))
            Q = torch.stack(V, 1)
            for _ in range(2):
                w = w - Q @ (Q.conj().T @ w)
            be.append(float(torch.linalg.norm(w)))
            V.append(w / be[-1])
        T = torch.diag(torch.tensor(al, dtype=torch.float64))
        for j in range(k - 1):
            T[j, j + 1] = T[j + 1, j] = be[j]
        th = torch.linalg.eigvalsh(T)
        lo, hi = float(th[0]), float(th[-1])
        return hi + be[-1], lo, hi
    H, Y = d["H"], d["Y"]
    W = H @ Y
    G = Y.conj().T @ W
    theta, Q = torch.linalg.eigh(0.5 * (G + G.conj().T))
    Yr, HYr = _fix_gauge(d["r"], Y @ Q, W @ Q)
    return {"theta": theta, "Y": Yr, "HY": HYr}


def work(case):
    """Complex multiply-adds count 8 flops; a Hermitian or triangular matrix is read once as half."""
    n, kind = case["n"], case["kind"]
    half = 8.0 * n * n  # bytes of one triangle
    if kind == "solve":
        # per sequence the factor of B, per problem the reduction, one filter loop and its
        # Rayleigh-Ritz products
        N, blk, nev = case["N"], case["blk"], case["nev"]
        flops = 4.0 / 3.0 * n**3 + N * (4.0 * n**3 + 8.0 * n * n * blk * (case["deg"] + 1) + 24.0 * n * blk * blk)
        return {"bytes": (N + 1) * half + N * 16.0 * n * nev, "flops": flops}
    if kind == "filter":
        mean = 0.5 * (case["deg_min"] + case["deg_max"])
        return {"bytes": half + 32.0 * n * case["m"], "flops": 8.0 * n * n * case["m"] * mean}
    if kind == "cholesky":
        return {"bytes": 2 * half, "flops": 4.0 / 3.0 * n**3}
    if kind == "reduce":
        return {"bytes": 2 * half + 16.0 * n * n, "flops": 4.0 * n**3}
    if kind == "lanczos":
        return {"bytes": half * case["k"], "flops": 8.0 * n * n * case["k"]}
    if kind == "orthonormalize":
        m, k = case["m"], case["k"]
        return {"bytes": 16.0 * n * (2 * m + k), "flops": 8.0 * n * m * (4 * k + 2 * m)}
    m = case["m"]
    return {"bytes": half + 48.0 * n * m, "flops": 8.0 * n * n * m + 24.0 * n * m * m}
