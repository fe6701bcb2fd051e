"""The workloads whose speed this framework is judged by, through its public entry points.

A case is a dict of plain values.  Every solve takes a synthetic system of atoms
on a jittered 2.5 A grid with 8 basis functions and 2 occupied orbitals per
atom, the short-ranged H and S of the repository's synthetic generator, drawn
here on the GPU.  Sizes are those of the repository's configurations, tests and
benchmark: dense m = 144 .. 8192 (n = m / 4), the localised form up to a few
thousand atoms, batches of uneven systems of 32 .. 384 atoms.  `drop_high` and
`drop_low` remove that many unoccupied and occupied orbitals of the last atom,
which makes m and n odd.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2209_05934_gb300 import omm

DEV = "cuda"
F64 = torch.float64
SPACING, JITTER, HS_CUTOFF = 2.5, 0.2, 5.0
COLD_STEPS, WARM_STEPS = 50, 8          # usual CG step counts of a cold and a warm dense solve


# ---------------------------------------------------------------------- the cases
def listed():
    return [
        # a molecule-sized system in the default (FP64) arithmetic: launches and latency decide
        dict(name="fp64_solve_m144", kind="solve", precision="fp64", atoms=18, drop_high=0, drop_low=0),
        # the dense FP64 configuration (64 atoms, m = 512) converged to 1e-10
        dict(name="fp64_solve_m512", kind="solve", precision="fp64", atoms=64, drop_high=0, drop_low=0),
        # an ordinary FP64 solve of a size that fits no tile
        dict(name="fp64_solve_m1996", kind="solve", precision="fp64", atoms=250, drop_high=3, drop_low=1),
        # one SCF step of a served sequence: H changes by 1e-3 eV, S and the previous W stay
        dict(name="mixed_scf_m1856", kind="scf", precision="mixed", atoms=232, drop_high=0, drop_low=0),
        # the benchmark's solve: set_HS and a cold mixed-precision solve at m = 4096
        dict(name="mixed_solve_m4096", kind="solve", precision="mixed", atoms=512, drop_high=0, drop_low=0),
        # the upper end of the served sizes, ragged
        dict(name="mixed_solve_m8171", kind="solve", precision="mixed", atoms=1022, drop_high=4, drop_low=1),
        # the Cholesky-reduced variant: factor, reduce, solve, map back
        dict(name="cholesky_solve_m2048", kind="cholesky", precision="mixed", atoms=256, drop_high=0, drop_low=0),
        # independent spins / k-points / systems solved as one group
        dict(name="batch_16", kind="batch", count=16, lo=32, hi=384, sizes_seed=4),
        # the density matrix an SCF step takes from a converged solve
        dict(name="density_m2880", kind="density", which="rho", atoms=360, drop_high=0, drop_low=0),
        # linear-scaling steps in FP64
        dict(name="sparse_fp64_512", kind="sparse", precision="fp64", atoms=512, radius=6.0, steps=12),
        # linear-scaling steps in mixed precision
        dict(name="sparse_mixed_1728", kind="sparse", precision="mixed", atoms=1728, radius=6.0, steps=24),
        # one FP64-accurate product as a caller of the C ABI runs it: W^T (H W)
        dict(name="op_exact_gemm_tn", kind="op", op="exact", trans_a=1, trans_b=0, M=1024, N=1000, K=4096, digits=7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve64", "solve64", "solve", "solve", "scf", "cholesky", "precon", "batch", "density",
                       "sparse64", "sparse", "op", "op"])
    drops = dict(drop_high=rng.choice([0, 0, 1, 2, 3, 5]), drop_low=rng.choice([0, 0, 1]))
    if kind == "solve64":
        return dict(kind="solve", precision="fp64", atoms=_log_int(rng, 12, 240), **drops)
    if kind == "solve":
        return dict(kind="solve", precision="mixed", atoms=_log_int(rng, 32, 700), **drops)
    if kind == "scf":
        return dict(kind="scf", precision=rng.choice(["mixed", "mixed", "fp64"]), atoms=_log_int(rng, 32, 240), **drops)
    if kind == "cholesky":
        return dict(kind="cholesky", precision=rng.choice(["mixed", "fp64"]), atoms=_log_int(rng, 20, 200), **drops)
    if kind == "precon":
        return dict(kind="precon", precision=rng.choice(["mixed", "fp64"]), atoms=_log_int(rng, 20, 160), **drops)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 16), lo=32, hi=rng.choice([96, 200, 384]),
                    sizes_seed=rng.randrange(1000))
    if kind == "density":
        return dict(kind="density", which=rng.choice(["rho", "rho_E"]), atoms=_log_int(rng, 32, 340), **drops)
    if kind == "sparse64":
        return dict(kind="sparse", precision="fp64", atoms=_log_int(rng, 27, 500), radius=rng.choice([4.5, 6.0]),
                    steps=rng.randint(4, 12))
    if kind == "sparse":
        return dict(kind="sparse", precision="mixed", atoms=_log_int(rng, 64, 1600), radius=rng.choice([4.5, 6.0]),
                    steps=rng.randint(8, 24))
    op = rng.choice(["exact", "split", "dgemm"])
    top = {"exact": 3000, "split": 4000, "dgemm": 1500}[op]
    return dict(kind="op", op=op, trans_a=rng.randint(0, 1), trans_b=rng.randint(0, 1), M=_log_int(rng, 33, top),
                N=_log_int(rng, 33, top), K=_log_int(rng, 64, top),
                digits={"exact": rng.choice([6, 7, 8]), "split": rng.choice([2, 3]), "dgemm": 0}[op])


# ---------------------------------------------------------------------- inputs
def _positions(atoms, gen):
    side = int(math.ceil(round(atoms ** (1.0 / 3.0), 9)))
    idx = torch.arange(atoms, device=DEV)
    grid = torch.stack([idx // (side * side), idx // side % side, idx % side], dim=1).to(F64) * SPACING
    return grid + (torch.rand(atoms, 3, generator=gen, device=DEV, dtype=F64) * 2 - 1) * JITTER


def _distances(pos):
    d = pos[:, None, :] - pos[None, :, :]
    return (d * d).sum(-1).sqrt()


def _blocks(atoms, gen, kinetic=False, geometry=None):
    """Distances and the block arrays H, S (and T) as (N, N, 8, 8); zero beyond the cutoff."""
    r = _distances(_positions(atoms, gen if geometry is None else geometry))
    I, J = torch.nonzero(torch.triu(r <= HS_CUTOFF, diagonal=1), as_tuple=True)
    rij = r[I, J][:, None, None]
    rand = lambda f: f((I.numel(), 8, 8), generator=gen, device=DEV, dtype=F64)
    onsite = torch.tensor([-5.0, -5.0] + [5.0] * 6, device=DEV, dtype=F64)
    onsite = onsite + 0.3 * torch.randn(atoms, 8, generator=gen, device=DEV, dtype=F64)
    diag = torch.arange(atoms, device=DEV)

    def fill(pair, on):
        A = torch.zeros(atoms, atoms, 8, 8, device=DEV, dtype=F64)
        A[I, J] = pair
        A[J, I] = pair.transpose(1, 2)
        A[diag, diag] = torch.diag_embed(on)
        return A

    H = fill(0.8 * torch.exp(-rij / 1.5) * rand(torch.randn), onsite)
    S = fill(0.15 * torch.exp(-rij / 1.2) * (rand(torch.rand) * 2 - 1) / 8, torch.ones(atoms, 8, device=DEV, dtype=F64))
    if not kinetic:
        return r, H, S, None
    on = torch.tensor([2.0, 2.0, 0.5, 20.0, 50.0, 100.0, 200.0, 400.0], device=DEV, dtype=F64)
    on = on + 0.05 * torch.randn(atoms, 8, generator=gen, device=DEV, dtype=F64)
    return r, H, S, fill(0.05 * torch.exp(-rij / 1.2) * (rand(torch.rand) * 2 - 1) / 8, on)


def _dense(case, seed, kinetic=False):
    """H, S, W0 (and T) of a dense case, column-major on the GPU."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    N, dh, dl = case["atoms"], case.get("drop_high", 0), case.get("drop_low", 0)
    _, H, S, T = _blocks(N, gen, kinetic)
    keep = torch.arange(8 * N - dh, device=DEV)
    keep = keep[keep != 8 * (N - 1)] if dl else keep
    n = 2 * N - dl

    def flat(A):
        A = A.permute(0, 2, 1, 3).reshape(8 * N, 8 * N)
        return A[keep][:, keep].T.contiguous().T if (dh or dl) else A.T.contiguous().T

    H, S = flat(H), flat(S)
    T = flat(T) if T is not None else None
    m = H.shape[0]
    W0 = (torch.randn(n, m, generator=gen, device=DEV, dtype=F64) / math.sqrt(m)).T
    return H if T is None else _cm(H + T), S, W0, T


def _cm(A):
    return A.T.contiguous().T


def _perturb(H, seed):
    """An SCF-like change: sym(N(0, 1e-3 eV)) on the nonzeros of H."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 7919)
    R = torch.randn(H.shape, generator=gen, device=DEV, dtype=F64) * 1e-3
    return _cm(H + (R + R.T) / 2 * (H != 0))


def _precision(case):
    return omm.PREC_MIXED if case["precision"] == "mixed" else omm.PREC_FP64


def _batch_sizes(case):
    rng = np.random.Generator(np.random.PCG64(case["sizes_seed"]))
    a = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["count"]))
    return [int(v) for v in np.rint(a)]


def _sparse_inputs(case, seed):
    """Block CSR of H, S (8 x 8) and W (8 x 2 blocks within `radius`), and a localised W0.

    The geometry, hence the block patterns, is that of the case (an SCF cycle
    keeps it); the values are those of the seed."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    N = case["atoms"]
    r, H, S, _ = _blocks(N, gen, geometry=torch.Generator(device=DEV).manual_seed(N))
    hmask, wmask = r <= HS_CUTOFF, r <= case["radius"]
    csr = lambda mask: (np.concatenate([[0], np.cumsum(mask.sum(1).cpu().numpy())]).astype(np.int64),
                        torch.nonzero(mask)[:, 1].cpu().numpy().astype(np.int32))
    at = torch.nonzero(wmask)
    sigma = 1.0 / torch.sqrt(8.0 * wmask.sum(0).to(F64))
    W0 = torch.randn(at.shape[0], 8, 2, generator=gen, device=DEV, dtype=F64) * sigma[at[:, 1]][:, None, None]
    return csr(hmask), csr(wmask), H[hmask].contiguous(), S[hmask].contiguous(), W0.contiguous(), (H, S, at)


# ---------------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "cholesky", "precon"):
        H, S, W0, T = _dense(case, seed, kinetic=kind == "precon")
        m, n = W0.shape
        opts = dict(precision=_precision(case))
        if case["precision"] == "mixed":
            opts["orth_tol"] = 1e-6
        if kind == "cholesky":
            opts["cholesky"] = 1
        if kind == "precon":
            opts["precon"] = -1
        s = omm.Solver(m, n, 8, **opts)
        if T is not None:
            torch.cuda.synchronize()
            s.set_T(T)
        return dict(kind="solve", s=s, H=H, S=S, W0=W0, W=_cm(torch.zeros_like(W0)))
    if kind == "scf":
        H, S, W0, _ = _dense(case, seed)
        m, n = W0.shape
        s = omm.Solver(m, n, 8, precision=_precision(case), orth_tol=1e-6)
        W = _cm(torch.zeros_like(W0))
        torch.cuda.synchronize()
        s.set_HS(H, S)
        s.solve(W0, tol=1e-10, W_out=W)
        return dict(kind="scf", s=s, H=_perturb(H, seed), W0=W, W=_cm(torch.zeros_like(W0)))
    if kind == "batch":
        solvers, Hs, Ss, W0s, Ws = [], [], [], [], []
        for i, atoms in enumerate(_batch_sizes(case)):
            H, S, W0, _ = _dense(dict(atoms=atoms), seed * 64 + i)
            m, n = W0.shape
            solvers.append(omm.Solver(m, n, 8, precision=omm.PREC_MIXED, orth_tol=1e-6))
            Hs.append(H)
            Ss.append(S)
            W0s.append(W0)
            Ws.append(_cm(torch.zeros_like(W0)))
        return dict(kind="batch", s=solvers, H=Hs, S=Ss, W0=W0s, W=Ws)
    if kind == "density":
        H, S, W0, _ = _dense(case, seed)
        m, n = W0.shape
        s = omm.Solver(m, n, 8, precision=omm.PREC_MIXED, orth_tol=1e-6)
        torch.cuda.synchronize()
        s.set_HS(H, S)
        s.solve(W0, tol=1e-12)
        which = omm.DENSITY_RHO_E if case["which"] == "rho_E" else omm.DENSITY_RHO
        return dict(kind="density", s=s, which=which, out=_cm(torch.zeros(m, m, device=DEV, dtype=F64)))
    if kind == "sparse":
        (hrp, hcol), (wrp, wcol), Hv, Sv, W0, _ = _sparse_inputs(case, seed)
        N = case["atoms"]
        s = omm.SparseSolver(8 * N, 2 * N, 8, 2, hrp, hcol, wrp, wcol, precision=_precision(case),
                             max_iter=case["steps"])
        return dict(kind="sparse", s=s, H=Hv, S=Sv, W0=W0, W=torch.zeros_like(W0))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    M, N, K, d = case["M"], case["N"], case["K"], case["digits"]
    normal = lambda rows, cols: torch.randn(cols, rows, generator=gen, device=DEV, dtype=F64).T
    A = normal(K, M) if case["trans_a"] else normal(M, K)
    B = normal(N, K) if case["trans_b"] else normal(K, N)
    nb = {"exact": omm.op_exact_gemm_workspace_bytes, "split": omm.op_split_gemm_workspace_bytes,
          "dgemm": lambda *a: 0}[case["op"]](M, N, K, d)
    return dict(kind="op", case=dict(case), A=A, B=B, C=_cm(torch.zeros(M, N, device=DEV, dtype=F64)),
                ws=torch.zeros(nb // 8 + 64, device=DEV, dtype=F64), nb=nb)


def run(state):
    kind, s = state["kind"], state.get("s")
    if kind == "solve":
        s.set_HS(state["H"], state["S"])
        E, iters, _ = s.solve(state["W0"], tol=1e-10, W_out=state["W"])
        return dict(E=E, iters=iters, W=state["W"])
    if kind == "scf":
        s.set_H(state["H"])
        E, iters, _ = s.solve(state["W0"], tol=1e-10, W_out=state["W"])
        return dict(E=E, iters=iters, W=state["W"])
    if kind == "batch":
        for one, H, S in zip(s, state["H"], state["S"]):
            one.set_HS(H, S)
        E, iters, _, rc = omm.batch_solve_grouped(s, state["W0"], tol=1e-10)
        omm.check(rc, "batch")
        for one, W in zip(s, state["W"]):      # the solutions stay in the handles
            omm.check(omm.lib().omm_get_array(one._h, omm.ARRAY_W, ctypes.c_void_p(W.data_ptr()), 1), "get_array")
        return dict(E=E, iters=iters, W=state["W"])
    if kind == "density":
        return s.get_density(state["which"], out=state["out"])
    if kind == "sparse":
        s.set_HS(state["H"], state["S"])
        E, iters, _ = s.solve(state["W0"], tol=1e-14, W_out=state["W"], raise_on_error=False)
        return dict(E=E, iters=iters, W=state["W"])
    c, A, B, C = state["case"], state["A"], state["B"], state["C"]
    lda, ldb, stream = A.shape[0], B.shape[0], torch.cuda.current_stream().cuda_stream
    args = (c["trans_a"], c["trans_b"], c["M"], c["N"], c["K"])
    if c["op"] == "dgemm":
        st = omm.op_dgemm(*args, 1.0, A, lda, B, ldb, 0.0, None, c["M"], C, c["M"], stream=stream)
    else:
        f = omm.op_exact_gemm if c["op"] == "exact" else omm.op_split_gemm
        st = f(*args, c["digits"], 1.0, A, lda, B, ldb, 0.0, None, c["M"], C, c["M"], state["ws"], state["nb"],
               stream=stream)
    omm.check(st, c["op"])
    return C


# ---------------------------------------------------------------------- work and 64-bit values
def _solve_work(m, n, steps):
    # H'D and SD, the four contractions, the gradient per step; H, S, W0 in, W out
    return dict(bytes=8.0 * (2 * m * m + 2 * m * n), flops=steps * (4.0 * m * m * n + 8.0 * m * n * n + 4.0 * m * n * n))


def _sizes(case):
    dh, dl = case.get("drop_high", 0), case.get("drop_low", 0)
    return 8 * case["atoms"] - dh - dl, 2 * case["atoms"] - dl


def work(case):
    kind = case["kind"]
    if kind == "op":
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=8.0 * (M * K + K * N + M * N), flops=2.0 * M * N * K)
    if kind == "batch":
        w = [_solve_work(8 * a, 2 * a, COLD_STEPS) for a in _batch_sizes(case)]
        return dict(bytes=sum(x["bytes"] for x in w), flops=sum(x["flops"] for x in w))
    if kind == "sparse":
        # neighbours within a radius of the 2.5 A grid (bulk density), blocks of 8 x 8 and 8 x 2
        near = lambda R: min(case["atoms"], 4.0 / 3.0 * math.pi * (R / SPACING) ** 3)
        N, h, w = case["atoms"], near(HS_CUTOFF), near(case["radius"])
        pn = near(2 * case["radius"] + HS_CUTOFF)
        triples = N * (h * w * 2 * 256.0 + w * pn * (3 * 64.0 + 2 * 64.0) / 4)
        return dict(bytes=8.0 * N * (2 * 64 * h + 2 * 16 * w), flops=case["steps"] * triples)
    m, n = _sizes(case)
    if kind == "density":
        e = 1 if case["which"] == "rho_E" else 0
        return dict(bytes=8.0 * (m * n + m * m * (2 + e)),
                    flops=(1 + e) * (2.0 * m * m * n + 2.0 * m * n * n) + 2.0 * m * n * n + 2.0 * m * m * n)
    w = _solve_work(m, n, WARM_STEPS if kind == "scf" else COLD_STEPS)
    if kind == "cholesky":
        w["flops"] += m ** 3 / 3.0 + 2.0 * m ** 3
    if kind == "precon":
        w["flops"] += m ** 3 / 3.0 + m ** 3 + COLD_STEPS * 2.0 * m * m * n
        w["bytes"] += 8.0 * m * m
    if kind == "scf":
        w["bytes"] -= 8.0 * m * m      # S stays
    return w


def _eta(H, S):
    """The Gershgorin bound of the pencil's spectrum (the default shift)."""
    dH, dS = H.diagonal(), S.diagonal()
    g = float((dH + H.abs().sum(1) - dH.abs()).max())
    off = S.abs().sum(1) - dS.abs()
    return g / float((dS - off).min()) if g >= 0 else g / float((dS + off).max())


def _line_min(c):
    roots = np.roots([4 * c[4], 3 * c[3], 2 * c[2], c[1]])
    scale = max(1.0, float(np.abs(roots).max()))
    xs = [float(r.real) for r in roots if abs(r.imag) <= 1e-10 * scale]
    xs = [x for x in xs if 12 * c[4] * x * x + 6 * c[3] * x + 2 * c[2] > 0]
    return min(xs, key=lambda x: (np.polyval(c[::-1], x), abs(x), -x))


def _cg(H, S, W, tol, max_iter, mask=None):
    """The method in plain 64-bit torch: exact line minima along Polak-Ribiere+ directions."""
    eta, n, k = _eta(H, S), W.shape[1], 0
    Hs = H - eta * S
    D = Gp = Ep = None
    HW, SW = Hs @ W, S @ W
    while True:
        h0, s0 = W.T @ HW, W.T @ SW
        E = float(2 * (2 * h0.trace() - (s0 * h0).sum())) + 2 * eta * n
        if k >= 1 and abs(2 * (E - Ep) / (E + Ep)) < tol:
            break
        if k >= max_iter:
            break
        G = 2 * (2 * HW - SW @ h0 - HW @ s0)
        G = G * mask if mask is not None else G
        if D is None:
            D = -G
        else:
            beta = max(0.0, float((G * (G - Gp)).sum() / (Gp * Gp).sum()))
            D = -G + beta * D
            if float((G * D).sum()) >= 0:
                D = -G
        HD, SD = Hs @ D, S @ D
        X, Y, h2, s2 = W.T @ HD, W.T @ SD, D.T @ HD, D.T @ SD
        dot = lambda a, b: float((a * b).sum())
        c = np.array([2 * (2 * float(h0.trace()) - dot(s0, h0)),
                      2 * (4 * float(X.trace()) - 2 * dot(s0, X) - 2 * dot(Y, h0)),
                      2 * (2 * float(h2.trace()) - dot(s0, h2) - 2 * dot(Y, X) - 2 * dot(Y, X.T) - dot(s2, h0)),
                      2 * (-2 * dot(Y, h2) - 2 * dot(s2, X)), -2 * dot(s2, h2)])
        x = _line_min(c)
        W = W + x * D
        HW, SW = HW + x * HD, SW + x * SD
        Ep, Gp, k = E, G, k + 1
    return E, k, W


def exact(case, seed):
    kind = case["kind"]
    if kind == "op":
        s = prepare(case, seed)
        return (s["A"].T if case["trans_a"] else s["A"]) @ (s["B"].T if case["trans_b"] else s["B"])
    if kind == "solve" and case["precision"] == "fp64":
        H, S, W0, _ = _dense(case, seed)
        E, k, W = _cg(H, S, W0, 1e-10, 10000)
        return dict(E=E, iters=k, W=W)
    if kind in ("solve", "cholesky", "precon") and case["atoms"] <= 512:
        # the minimum is twice the sum of the n lowest generalised eigenvalues; W is one of many
        H, S, W0, _ = _dense(case, seed, kinetic=kind == "precon")
        L = torch.linalg.cholesky(S)
        A = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, H, upper=False).T, upper=False)
        lam = torch.linalg.eigvalsh((A + A.T) / 2)
        return dict(E=2.0 * float(lam[: W0.shape[1]].sum()), iters=None, W=None)
    if kind == "density":
        H, S, W0, _ = _dense(case, seed)
        n = W0.shape[1]
        L = torch.linalg.cholesky(S)
        A = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, H, upper=False).T, upper=False)
        lam, U = torch.linalg.eigh((A + A.T) / 2)
        V = torch.linalg.solve_triangular(L.T, U[:, :n], upper=True)
        return 2 * (V * lam[:n]) @ V.T if case["which"] == "rho_E" else 2 * V @ V.T
    if kind == "sparse" and case["precision"] == "fp64" and case["atoms"] <= 600:
        *_, W0, (H, S, at) = _sparse_inputs(case, seed)
        N = case["atoms"]
        flat = lambda A: A.permute(0, 2, 1, 3).reshape(8 * N, 8 * N)
        W = torch.zeros(N, N, 8, 2, device=DEV, dtype=F64)
        mask = torch.zeros_like(W)
        W[at[:, 0], at[:, 1]] = W0
        mask[at[:, 0], at[:, 1]] = 1.0
        thin = lambda A: A.permute(0, 2, 1, 3).reshape(8 * N, 2 * N)
        E, k, W = _cg(flat(H), flat(S), thin(W), 1e-14, case["steps"], thin(mask))
        return dict(E=E, iters=k, W=W.reshape(N, 8, N, 2).permute(0, 2, 1, 3)[at[:, 0], at[:, 1]])
    return None
