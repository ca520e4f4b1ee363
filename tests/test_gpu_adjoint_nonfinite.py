"""A NaN or an infinity in what the adjoints take reaches Abar, on both sides of the
line (8 N^2 K = 2e8 operations) from which the N x N product runs on the tensor
cores: 0 * inf and sums with NaN are NaN in FP64, so entry (r, k) of Z leaves no
finite entry in row r of Abar, nor, after the Hermitian part, in column r."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BAD = [float("nan"), float("inf")]


def random(lib, rows, cols, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return lib.colmajor(torch.randn(cols, rows, dtype=torch.complex128, device="cuda",
                                    generator=g).mT)


def hermitian(lib, N):
    Z = random(lib, N, N, N)
    return lib.colmajor((Z + Z.mH) / (4 * N ** 0.5))


# 2 parts of K and a ragged column block at N = 700, K = 99; the CUDA cores at N = 200
@pytest.mark.parametrize("N,n", [(700, 33), (200, 12)])
@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("where", ["Ybar", "V"])
def test_filter_adjoint(lib, N, n, bad, where):
    A, V, Yb = hermitian(lib, N), random(lib, N, n, 1), random(lib, N, n, 2)
    r, k = N // 3, n // 2
    (Yb if where == "Ybar" else V)[r, k] = bad
    Ab, Vb = torch.empty_like(A), torch.empty_like(V)
    Ab = lib.colmajor(Ab)
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=1)) as ctx:
        ctx.chase_filter_vjp(A, V, n, 6, 0.3, 0.9, -1.2, Yb, Ab, lib.colmajor(Vb))
    assert not torch.isfinite(Ab[r, :].real).any() or not torch.isfinite(Ab[r, :].imag).any()
    assert not torch.isfinite(Ab[:, r].real).any() or not torch.isfinite(Ab[:, r].imag).any()


@pytest.mark.parametrize("N,n", [(700, 64), (200, 12)])
@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("where", ["lam_bar", "X_bar", "X"])
def test_eigenpair_adjoint(lib, N, n, bad, where):
    H = torch.linalg.qr(random(lib, N, N, 3))[0]
    lam = torch.linspace(1.0, 9.0, N, dtype=torch.float64, device="cuda")
    A = (H * lam) @ H.mH
    A = lib.colmajor((A + A.mH) / 2)
    X, lam_bar = lib.colmajor(H[:, :n]), torch.ones(n, dtype=torch.float64, device="cuda")
    X_bar = random(lib, N, n, 4) if where == "X_bar" else None
    r, k = N // 3, n // 2
    if where == "lam_bar":
        lam_bar[k] = bad
    elif where == "X_bar":
        X_bar[r, k] = bad
    else:
        X[r, k] = bad
    Ab = lib.colmajor(torch.empty_like(A))
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=1)) as ctx:
        ctx.chase_eig_vjp(A, X, lam[:n].contiguous(), n, n, lam_bar, X_bar, Ab, cg_tol=1e-6,
                          allow_not_converged=True)
    # a whole column of M (lam_bar, X_bar) or one row of it
    rows = slice(None) if where != "X" else slice(r, r + 1)
    finite = torch.isfinite(Ab.real) & torch.isfinite(Ab.imag)
    assert not finite[rows, :].any() and not finite[:, rows].any()


def test_finite_result_is_unchanged(lib):
    """The largest finite entries are not taken for infinities."""
    N, n = 700, 64
    X = lib.colmajor(torch.linalg.qr(random(lib, N, n, 5))[0])
    A = lib.colmajor(torch.eye(N, dtype=torch.complex128, device="cuda"))
    out = []
    for s in (1.0, 2.0 ** 1000):
        Ab = lib.colmajor(torch.empty_like(A))
        with lib.Context(lib.default_params(N, n, 0, fp64_tensor=1)) as ctx:
            ctx.chase_eig_vjp(A, X, torch.ones(n, dtype=torch.float64, device="cuda"), n, n,
                              torch.full((n,), s, dtype=torch.float64, device="cuda"), None, Ab)
        out.append(Ab / s)
    assert torch.equal(out[0], out[1]) and bool(torch.isfinite(out[0].real).all())
