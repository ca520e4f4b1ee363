"""The work that a program built on this library has it do, as measurable cases.

Each case calls one public entry point of ``paper_2309_15595_gb300`` on inputs a
caller would have on the GPU: a dense Hermitian matrix, a block of vectors and a
context created once. The sizes are those of the repository's own problems
(``synth/problems.py``: the 512-row parity problem, the warm-start batch of orders
256 to 4096, the 4096-row gradient problem, the 20000-row workload) and the DFT
matrix orders that the paper's Table 2 lists (9273 and 13379).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2309_15595_gb300 as chase

HI = 10.0          # spectra lie in [0, HI]: the repository's uniform problems
REFLECTORS = 8


def listed():
    return [
        # the smallest call: the FP64 filter of the 512-row parity problem on the
        # tensor cores, one call per outer iteration, latency and launches count
        dict(name="filter_512", op="filter", N=512, n=60, dmax=20, tensor=1, mixed=0, dense=0),
        # FP64 filter on the tensor cores with the per-vector degrees that degree
        # optimisation gives, at the order and block width of the 9k DFT matrix
        dict(name="filter_9273", op="filter", N=9273, n=316, dmax=36, tensor=1, mixed=0, dense=0),
        # reduced-precision filter, first iteration (degree 20 for every vector),
        # 13k DFT matrix
        dict(name="filter_mixed_13379", op="filter", N=13379, n=1072, dmax=20, tensor=1, mixed=1,
             dense=0),
        # the library's default options: FP64 filter on the CUDA cores, dense matrix
        dict(name="filter_default_2600", op="filter", N=2600, n=195, dmax=10, tensor=0, mixed=0,
             dense=1),
        # orthonormalisation of a filtered block (CholeskyQR2), 13k DFT matrix
        dict(name="qr_13379", op="qr", N=13379, n=1072, cond=1e4, graded=0, tensor=1),
        # Rayleigh-Ritz with the Jacobi eigensolver on a half-converged block
        dict(name="rr_9273", op="rr", N=9273, n=316, tensor=1),
        # residual norms of all vectors of the 20000-row workload
        dict(name="residuals_20000", op="residuals", N=20000, n=1300, tensor=1, dense=0),
        # backward of the eigenpairs (perturbation theory, complement by CG)
        dict(name="eig_vjp_2048", op="eig_vjp", N=2048, n=64, nex=32, tensor=1),
        # backward of the filter (reversed recurrence with checkpoints)
        dict(name="filter_vjp_1500", op="filter_vjp", N=1500, n=96, deg=20, tensor=1),
        # one iteration of the whole method: Lanczos, reduced-precision filter, QR,
        # Rayleigh-Ritz, residuals, locking (the paper's weak-scaling unit)
        dict(name="step_13379", op="step", N=13379, nev=972, nex=100, tensor=1, mixed=1),
        # the first iteration of eight independent problems solved at once
        dict(name="batch_8", op="batch", sizes="256,700,384,1000,300,2100,1477,611", tensor=1,
             mixed=1),
        # a whole solve to convergence: the 512-row parity problem
        dict(name="solve_512", op="solve", N=512, nev=40, nex=20, tensor=1, mixed=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, N, most):
    """Block widths of the repository's problems: 1/40 to 1/6 of the order."""
    return max(4, min(most, int(N / math.exp(rng.uniform(math.log(6), math.log(40))))))


def draw(rng):
    op = rng.choice(["filter", "filter", "filter", "qr", "rr", "residuals", "lanczos", "eig_vjp",
                     "filter_vjp", "step", "batch", "solve"])
    if op == "filter":
        kind = rng.choice(["tensor", "tensor", "mixed", "default"])
        N = _log(rng, 200, 2600 if kind == "default" else 12000)
        n = _width(rng, N, 195 if kind == "default" else 900)
        return dict(op=op, N=N, n=n, dmax=2 * rng.randint(1, 5 if kind == "default" else 10),
                    tensor=int(kind != "default"), mixed=int(kind == "mixed"),
                    dense=rng.randint(0, 1))
    if op == "qr":
        N = _log(rng, 200, 12000)
        graded = rng.randint(0, 1)
        # 3e9 takes the shifted branch, 10 the single pass
        cond = rng.choice([1e4, 1e6, 3e9]) if graded else rng.choice([10.0, 1e3, 1e4])
        tensor = 1 if N > 2600 else rng.randint(0, 1)
        return dict(op=op, N=N, n=_width(rng, N, 900 if tensor else 200), cond=cond, graded=graded,
                    tensor=tensor)
    if op in ("rr", "residuals"):
        N = _log(rng, 200, 9273)
        tensor = 1 if N > 2600 else rng.randint(0, 1)
        n = _width(rng, N, 500 if op == "rr" else 900)
        if op == "rr":
            return dict(op=op, N=N, n=n, tensor=tensor)
        return dict(op=op, N=N, n=n, tensor=tensor, dense=rng.randint(0, 1))
    if op == "lanczos":
        N = _log(rng, 200, 12000)
        return dict(op=op, N=N, n=_width(rng, N, 900), nvec=rng.choice([4, 4, 1, 6]),
                    tensor=rng.randint(0, 1))
    if op == "eig_vjp":
        N = _log(rng, 256, 2048)
        nev = max(4, N // rng.choice([32, 48, 64]))
        return dict(op=op, N=N, n=nev, nex=nev // 2, tensor=rng.randint(0, 1))
    if op == "filter_vjp":
        N = _log(rng, 256, 1500)
        return dict(op=op, N=N, n=max(4, N // rng.choice([16, 24, 32])), deg=2 * rng.randint(3, 10),
                    tensor=rng.randint(0, 1))
    if op == "step":
        N = _log(rng, 300, 9273)
        return dict(op=op, N=N, nev=-(-N // 25), nex=-(-N // 50), tensor=1, mixed=rng.randint(0, 1))
    if op == "batch":
        k = rng.randint(2, 8)
        return dict(op=op, sizes=",".join(str(_log(rng, 256, 1600)) for _ in range(k)), tensor=1,
                    mixed=rng.randint(0, 1))
    N = _log(rng, 256, 700)
    return dict(op="solve", N=N, nev=-(-N // 14), nex=-(-N // 28), tensor=1, mixed=rng.randint(0, 1))


# ------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 17)
    return g


def _normal(g, rows, cols):
    """Complex Gaussian rows x cols block, E|z|^2 = 1, column-major."""
    z = torch.empty((cols, rows, 2), dtype=torch.float64, device="cuda").normal_(generator=g)
    return torch.view_as_complex(z.mul_(math.sqrt(0.5))).mT


def _apply(vs, X):
    """H X with H = (I - t1 v1 v1^H) ... (I - tr vr vr^H), in place."""
    for v in reversed(vs):
        t = 2.0 / float(torch.vdot(v, v).real)
        X -= t * torch.outer(v, v.conj() @ X)
    return X


def _reflectors(g, N):
    return [_normal(g, N, 1)[:, 0].contiguous() for _ in range(REFLECTORS)]


def _hermitian(lam, vs):
    """H diag(lam) H^H, exactly Hermitian, column-major."""
    N = lam.numel()
    A = torch.zeros((N, N), dtype=torch.complex128, device="cuda").mT
    A.diagonal().copy_(lam)
    for v in reversed(vs):
        t = 2.0 / float(torch.vdot(v, v).real)
        w = A @ v
        u = w - 0.5 * t * torch.vdot(v, w).real * v
        A -= t * torch.outer(v, u.conj())
        A -= t * torch.outer(u, v.conj())
    return _symmetrise(A)


def _symmetrise(A):
    A = chase.colmajor((A + A.mH) * 0.5)
    A.diagonal().imag.zero_()
    return A


def _uniform(N):
    return torch.arange(N, dtype=torch.float64, device="cuda") * (HI / (N - 1))


def _dense(g, N):
    """A dense random Hermitian matrix with its spectrum (a semicircle) in [0, HI]."""
    A = _symmetrise(_normal(g, N, N)) * (HI / (2 * math.sqrt(2 * N)) * 0.98)
    A.diagonal().real.add_(HI / 2)
    return chase.colmajor(A)


def _window(N, n, dense):
    """c, e, mu_1 of a filter that damps everything above the n-th eigenvalue."""
    lo = 0.0
    if dense:  # semicircle: the n-th of N eigenvalues lies about here
        cut = HI / 2 * (3 * math.pi * n / (math.sqrt(32) * N)) ** (2 / 3)
    else:
        cut = HI * (n - 1) / (N - 1)
    b = HI * 1.01
    return (b + cut) / 2, (b - cut) / 2, lo


def _options(case, **over):
    return dict(fp64_tensor=case["tensor"],
                precision=chase.CHASE_MIXED_BF16X3 if case.get("mixed") else chase.CHASE_FP64,
                **over)


def _context(N, nev, nex, case, **over):
    return chase.Context(chase.default_params(N, nev, nex, **_options(case, **over)))


def _matrix(case, g):
    if case.get("dense"):
        return _dense(g, case["N"])
    return _hermitian(_uniform(case["N"]), _reflectors(g, case["N"]))


def _conditioned(g, N, n, cond, graded):
    """A block as the filter leaves it: graded columns (amplified by different
    amounts) or columns that lean towards the strongest ones (condition cond)."""
    Q = torch.linalg.qr(_normal(g, N, n))[0]
    s = torch.logspace(0, -math.log10(cond), n, dtype=torch.float64, device="cuda")
    T = torch.triu(_normal(g, n, n), 1) * (0.3 / math.sqrt(n))
    T = T + torch.eye(n, dtype=T.dtype, device="cuda")
    T = T * s[None, :] if graded else s[:, None] * T
    return chase.colmajor(Q @ T)


def _band(N, n):
    """Spectrum with n low eigenvalues spread over the lower half of the range."""
    lam = torch.empty(N, dtype=torch.float64, device="cuda")
    lam[:n] = torch.arange(n, dtype=torch.float64, device="cuda") * (0.45 * HI / n)
    lam[n:] = torch.linspace(0.5 * HI, HI, N - n, dtype=torch.float64, device="cuda")
    return lam


def _basis(vs, N, n):
    """First n eigenvectors of H diag(.) H^H, column-major."""
    E = torch.zeros((n, N), dtype=torch.complex128, device="cuda").mT
    E.diagonal().fill_(1.0)
    return _apply(vs, E)


def _doubles(n):
    return torch.zeros(n, dtype=torch.float64, device="cuda")


def _raw(case, seed):
    """Inputs alone, without contexts (the exact values use them too)."""
    g, op = _gen(seed), case["op"]
    if op == "filter":
        N, n = case["N"], case["n"]
        A = _matrix(case, g)
        degs = np.sort(2 * np.random.RandomState(seed % (1 << 31)).randint(
            max(1, case["dmax"] // 4), case["dmax"] // 2 + 1, n)).astype(np.int32)
        if case["mixed"]:
            degs[:] = case["dmax"]
        degs[-1] = case["dmax"]
        return dict(A=A, V0=_normal(g, N, n), degs=degs, win=_window(N, n, case["dense"]))
    if op == "qr":
        return dict(X=_conditioned(g, case["N"], case["n"], case["cond"], case["graded"]))
    if op in ("rr", "eig_vjp"):
        N, n = case["N"], case["n"]
        vs = _reflectors(g, N)
        if op == "rr":
            A = _hermitian(_band(N, n), vs)
            Q = _basis(vs, N, n) + 0.1 / math.sqrt(N) * _normal(g, N, n)
            return dict(A=A, Q=chase.colmajor(torch.linalg.qr(Q)[0]), w=_normal(g, N, 1)[:, 0])
        lam = _band(N, n + case["nex"])
        return dict(A=_hermitian(lam, vs), X=_basis(vs, N, n + case["nex"]), lam=lam, vs=vs,
                    lam_bar=_normal(g, n, 1)[:, 0].real.contiguous(), X_bar=_normal(g, N, n))
    if op == "residuals":
        A = _matrix(case, g)
        V = chase.colmajor(torch.linalg.qr(_normal(g, case["N"], case["n"]))[0])
        return dict(A=A, V=V, ritz=(V.conj() * (A @ V[:, :1])).sum(0).real.contiguous())
    if op == "lanczos":
        N = case["N"]
        return dict(A=_hermitian(_uniform(N), _reflectors(g, N)), Q0=_normal(g, N, case["nvec"]))
    if op == "filter_vjp":
        N, n = case["N"], case["n"]
        return dict(A=_hermitian(_uniform(N), _reflectors(g, N)), V=_normal(g, N, n),
                    Ybar=_normal(g, N, n), win=_window(N, n, 0))
    if op in ("step", "solve"):
        N = case["N"]
        vs = _reflectors(g, N)
        return dict(A=_hermitian(_uniform(N), vs), V0=_normal(g, N, case["nev"] + case["nex"]),
                    Q0=_normal(g, N, 4), w=_normal(g, N, 1)[:, 0], vs=vs)
    probs = []
    for N in (int(x) for x in case["sizes"].split(",")):
        nev, nex = -(-N // 20), -(-N // 40)
        vs = _reflectors(g, N)
        probs.append(dict(N=N, nev=nev, nex=nex, A=_hermitian(_uniform(N), vs),
                          V0=_normal(g, N, nev + nex), Q0=_normal(g, N, 4),
                          w=_normal(g, N, 1)[:, 0]))
    return dict(probs=probs)


def prepare(case, seed):
    s, op = _raw(case, seed), case["op"]
    s["op"] = op
    if op == "filter":
        N, n = case["N"], case["n"]
        s.update(ctx=_context(N, n, 0, case), V=torch.empty_like(s["V0"]), n=n,
                 precision=chase.CHASE_MIXED_BF16X3 if case["mixed"] else chase.CHASE_FP64)
    elif op == "qr":
        s.update(ctx=_context(case["N"], case["n"], 0, case), V=torch.empty_like(s["X"]),
                 n=case["n"], cond=float(case["cond"]))
    elif op == "rr":
        s.update(ctx=_context(case["N"], case["n"], 0, case), V=torch.empty_like(s["Q"]),
                 n=case["n"], ritz=_doubles(case["n"]))
    elif op == "residuals":
        s.update(ctx=_context(case["N"], case["n"], 0, case), n=case["n"],
                 resid=_doubles(case["n"]))
    elif op == "lanczos":
        s.update(ctx=_context(case["N"], case["n"], 0, case, lanczos_vecs=case["nvec"]))
    elif op == "eig_vjp":
        N, nev, ne = case["N"], case["n"], case["n"] + case["nex"]
        s.update(ctx=_context(N, nev, case["nex"], case), nev=nev, ne=ne,
                 ritz=s["lam"][:ne].contiguous(), Abar=torch.empty_like(s["A"]))
        del s["lam"], s["vs"]
    elif op == "filter_vjp":
        s.update(ctx=_context(case["N"], case["n"], 0, case), n=case["n"], deg=case["deg"],
                 Abar=torch.empty_like(s["A"]), Vbar=torch.empty_like(s["V"]))
    elif op == "step":
        ne = case["nev"] + case["nex"]
        s.update(ctx=_context(case["N"], case["nev"], case["nex"], case, max_iter=1),
                 V=torch.empty_like(s["V0"]), ritz=_doubles(ne), resid=_doubles(ne))
        del s["vs"]
    elif op == "solve":
        s.update(nev=case["nev"], nex=case["nex"], over=_options(case, tol=1e-12))
        del s["vs"]
    else:
        for p in s["probs"]:
            ne = p["nev"] + p["nex"]
            p["stream"] = torch.cuda.Stream()
            with torch.cuda.stream(p["stream"]):
                p["ctx"] = _context(p["N"], p["nev"], p["nex"], case, max_iter=1)
            p.update(V=torch.empty_like(p["V0"]), ritz=_doubles(ne), resid=_doubles(ne))
    return s


# --------------------------------------------------------------------- runs
def _fix_phase(V, w):
    """Eigenvectors are unique up to a phase: make w^H v real and positive."""
    s = w.conj() @ V
    return V * (s.conj() / s.abs())


def run(state):
    s = state
    op = s["op"]
    if op == "filter":
        s["V"].copy_(s["V0"])
        s["ctx"].chase_filter(s["A"], s["V"], s["n"], s["degs"], *s["win"],
                              precision=s["precision"])
        return s["V"]
    if op == "qr":
        s["V"].copy_(s["X"])
        s["ctx"].chase_qr(s["V"], s["n"], s["cond"])
        return s["V"]
    if op == "rr":
        s["V"].copy_(s["Q"])
        s["ctx"].chase_rayleigh_ritz(s["A"], s["V"], s["n"], s["ritz"])
        return {"ritz": s["ritz"], "V": _fix_phase(s["V"], s["w"])}
    if op == "residuals":
        s["ctx"].chase_residuals(s["A"], s["V"], s["ritz"], s["n"], s["resid"])
        return s["resid"]
    if op == "lanczos":
        return list(s["ctx"].chase_lanczos(s["A"], s["Q0"]))
    if op == "eig_vjp":
        s["ctx"].chase_eig_vjp(s["A"], s["X"], s["ritz"], s["ne"], s["nev"], s["lam_bar"],
                               s["X_bar"], s["Abar"], cg_tol=1e-12)
        return s["Abar"]
    if op == "filter_vjp":
        c, e, mu = s["win"]
        s["ctx"].chase_filter_vjp(s["A"], s["V"], s["n"], s["deg"], c, e, mu, s["Ybar"], s["Abar"],
                                  s["Vbar"])
        return {"Abar": s["Abar"], "Vbar": s["Vbar"]}
    if op == "step":
        s["V"].copy_(s["V0"])
        s["ctx"].chase_solve(s["A"], s["V"], s["ritz"], s["resid"], lanczos_start=s["Q0"],
                             allow_not_converged=True)
        return {"ritz": s["ritz"], "resid": s["resid"], "V": _fix_phase(s["V"], s["w"])}
    if op == "solve":
        # the plain one-call form, context included; the converged pairs' residual
        # norms lie in the rounding noise below the tolerance and are not an output
        ritz, V, _, _ = chase.solve(s["A"], s["nev"], s["nex"], V0=s["V0"], lanczos_start=s["Q0"],
                                    **s["over"])
        return {"ritz": ritz, "V": _fix_phase(V, s["w"])}
    probs = s["probs"]
    main = torch.cuda.current_stream()
    for p in probs:
        p["V"].copy_(p["V0"])
    for p in probs:  # each problem's own stream starts after its inputs are there
        p["stream"].wait_stream(main)
    chase.solve_batch([p["ctx"] for p in probs], [p["A"] for p in probs], [p["V"] for p in probs],
                      [p["ritz"] for p in probs], [p["resid"] for p in probs],
                      lanczos_starts=[p["Q0"] for p in probs], allow_not_converged=True)
    for p in probs:
        main.wait_stream(p["stream"])
    return [{"ritz": p["ritz"], "resid": p["resid"], "V": _fix_phase(p["V"], p["w"])}
            for p in probs]


# --------------------------------------------------------------------- work
def _step_work(N, n, deg):
    flops = 8.0 * N * N * n * (deg + 2) + 32.0 * N * n * n + 36.0 * n ** 3 + 8.0 * N * N * 100
    return {"bytes": 16.0 * (N * N + 2 * N * n) + 16.0 * n, "flops": flops}


def work(case):
    op = case["op"]
    if op == "batch":
        parts = [_step_work(N, -(-N // 20) + -(-N // 40), 20)
                 for N in (int(x) for x in case["sizes"].split(","))]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N, n = case["N"], case.get("n", 0)
    A, B = 16.0 * N * N, 16.0 * N * n
    if op == "filter":
        mean = case["dmax"] if case["mixed"] else 0.75 * case["dmax"]
        return {"bytes": A + 2 * B, "flops": 8.0 * N * N * n * mean}
    if op == "qr":
        return {"bytes": 2 * B, "flops": 8.0 * N * n * n}
    if op == "rr":
        return {"bytes": A + 2 * B + 8.0 * n, "flops": 8.0 * N * N * n + 16.0 * N * n * n + 36.0 * n ** 3}
    if op == "residuals":
        return {"bytes": A + B + 16.0 * n, "flops": 8.0 * N * N * n}
    if op == "lanczos":
        return {"bytes": A + 16.0 * N * case["nvec"] + 32.0, "flops": 8.0 * N * N * case["nvec"] * 25}
    if op == "eig_vjp":
        # about 30 CG steps of one product with A and the projection, then Abar
        return {"bytes": 2 * A + 2 * B, "flops": 30 * (8.0 * N * N * n + 16.0 * N * n * n) + 8.0 * N * N * n}
    if op == "filter_vjp":
        return {"bytes": 2 * A + 3 * B, "flops": 8.0 * N * N * n * 3 * case["deg"]}
    ne = case["nev"] + case["nex"]
    if op == "step":
        return _step_work(N, ne, 20)
    return {"bytes": A + 2 * 16.0 * N * ne, "flops": 6 * _step_work(N, ne, 20)["flops"]}


# -------------------------------------------------------------------- exact
def _coefficients(deg, c, e, mu):
    """alpha_i, beta_i of the filter's three-term recurrence, normalised at mu."""
    s1 = e / (mu - c)
    al, be, s = [0.0, s1 / e], [0.0, 0.0], s1
    for _ in range(2, deg + 1):
        nxt = 1.0 / (2.0 / s1 - s)
        al.append(2.0 * nxt / e)
        be.append(-s * nxt)
        s = nxt
    return al, be


def exact(case, seed):
    op = case["op"]
    if op in ("step", "batch", "lanczos"):
        return None
    s = _raw(case, seed)
    if op == "filter":
        if case["mixed"] and case["N"] > 6000:
            return None  # about 40 s in 64 bits
        c, e, mu = s["win"]
        A, degs, V = s["A"], s["degs"], s["V0"].clone()
        al, be = _coefficients(int(degs[-1]), c, e, mu)
        cur, prev, out = V, None, torch.empty_like(V)
        for i in range(1, int(degs[-1]) + 1):
            j0 = int(np.searchsorted(degs, i))
            if prev is not None:
                k = cur.shape[1] - (len(degs) - j0)
                cur, prev = cur[:, k:], prev[:, k:]
            nxt = al[i] * (A @ cur - c * cur)
            if prev is not None:
                nxt += be[i] * prev
            prev, cur = cur, nxt
            done = int(np.searchsorted(degs, i, side="right")) - j0
            out[:, j0:j0 + done] = cur[:, :done]
        return out
    if op == "qr":
        Q, R = torch.linalg.qr(s["X"])
        d = R.diagonal()
        return Q * (d / d.abs())[None, :]
    if op == "rr":
        G = s["Q"].mH @ (s["A"] @ s["Q"])
        lam, Y = torch.linalg.eigh((G + G.mH) * 0.5)
        return {"ritz": lam, "V": _fix_phase(s["Q"] @ Y, s["w"])}
    if op == "residuals":
        R = s["A"] @ s["V"] - s["V"] * s["ritz"][None, :]
        return torch.linalg.vector_norm(R, dim=0)
    if op == "eig_vjp":
        N, nev = case["N"], case["n"]
        X, lam = _basis(s["vs"], N, N), s["lam"]
        C = X.mH @ s["X_bar"]
        gap = lam[None, :nev] - lam[:, None]
        F = torch.where(gap == 0, torch.zeros_like(gap), 1.0 / gap)
        M = X @ (C * F) + X[:, :nev] * s["lam_bar"][None, :]
        G = M @ X[:, :nev].mH
        return (G + G.mH) * 0.5
    if op == "filter_vjp":
        c, e, mu = s["win"]
        al, be = _coefficients(case["deg"], c, e, mu)
        A, Y = s["A"], [s["V"]]
        for i in range(1, case["deg"] + 1):
            y = al[i] * (A @ Y[-1] - c * Y[-1])
            Y.append(y + be[i] * Y[-2] if i > 1 else y)
        z1, z = torch.zeros_like(s["V"]), s["Ybar"]
        G = torch.zeros_like(A)
        be.append(0.0)
        for i in range(case["deg"], 0, -1):
            G += al[i] * (z @ Y[i - 1].mH)
            z, z1 = al[i] * (A @ z - c * z) + be[i + 1] * z1, z
        return {"Abar": (G + G.mH) * 0.5, "Vbar": z}
    nev = case["nev"]
    X = _basis(s["vs"], case["N"], nev)
    return {"ritz": _uniform(case["N"])[:nev], "V": _fix_phase(X, s["w"])}
