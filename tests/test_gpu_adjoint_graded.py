"""The adjoints' N x N product sum_k z_k w_k^H on the tensor cores keeps FP64's
accuracy whatever the sizes of z_k and w_k: only those of their products count.

Columns scaled by 2^s on one side and by 2^-s on the other leave every rounding of an
FP64 product where it was, so Abar has to keep its bits, and a term with a zero
factor has to leave no trace whatever the other one. The product alone is compared
with exact sums: seven digits of two operands leave about sqrt(2K) 2^-55 of the
largest |z_k| |w_k| (digit rounding 2^-57 of scales at most four times the largest
entries, and the pairs below 2^-64); eight times that is the bound, which six digits
(2^-47) or a lost level of pairs (2^-48) exceed."""
from fractions import Fraction

import numpy as np
import pytest

from test_gpu_adjoint_nonfinite import hermitian, random

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def filter_adjoint(lib, A, V, Yb, deg):
    N, n = V.shape
    Ab, Vb = lib.colmajor(torch.empty_like(A)), lib.colmajor(torch.empty_like(V))
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=1)) as ctx:
        ctx.chase_filter_vjp(A, V, n, deg, 0.3, 0.9, -1.2, lib.colmajor(Yb), Ab, Vb)
    return Ab


def powers(n, spread, seed):  # 2^s, s up to +-spread / 2
    s = np.random.default_rng(seed).integers(-(spread // 2), spread // 2 + 1, n)
    return torch.from_numpy(np.ldexp(1.0, s)).cuda()


# one part of K, several with ragged column blocks, the CUDA cores
@pytest.mark.parametrize("N,n,deg", [(700, 33, 6), (1031, 130, 6), (200, 12, 6)])
@pytest.mark.parametrize("spread", [8, 52, 400])
def test_graded_columns(lib, N, n, deg, spread):
    A, V, Yb = hermitian(lib, N), random(lib, N, n, 1), random(lib, N, n, 2)
    p = powers(n, spread, N)
    assert torch.equal(filter_adjoint(lib, A, lib.colmajor(V * p), Yb / p, deg),
                       filter_adjoint(lib, A, V, Yb, deg))


@pytest.mark.parametrize("side", ["V", "Ybar"])
def test_zero_factors(lib, side):
    N, n = 700, 33
    A, V, Yb = hermitian(lib, N), random(lib, N, n, 1), random(lib, N, n, 2)
    other, zero = (V, Yb) if side == "V" else (Yb, V)
    zero[:, 3] = zero[:, 17] = 0.0
    ref = filter_adjoint(lib, A, V, Yb, 6)
    other[:, 3] *= 2.0 ** 60
    other[:, 17] *= 2.0 ** -900
    assert torch.equal(filter_adjoint(lib, A, V, Yb, 6), ref)


@pytest.mark.parametrize("N,n", [(700, 64), (801, 130)])
@pytest.mark.parametrize("kind", ["even", "graded", "balanced", "tiny"])
def test_product_alone(lib, N, n, kind):
    X = torch.linalg.qr(random(lib, N, n, 3))[0]
    lam = torch.ones(n, dtype=torch.float64, device="cuda")
    if kind == "graded":     # terms of very different size
        lam = powers(n, 80, 5)
    if kind == "balanced":   # factors of very different size, terms of one
        p = powers(n, 80, 6)
        X, lam = X * p, p ** -2
    if kind == "tiny":       # rows and columns of different size
        d = powers(N, 40, 7)
        X = X * d[:, None]
    X = lib.colmajor(X)
    Ab = lib.colmajor(torch.empty(N, N, dtype=torch.complex128, device="cuda"))
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=1)) as ctx:
        ctx.chase_eig_vjp(lib.colmajor(torch.eye(N, dtype=torch.complex128, device="cuda")), X,
                          torch.arange(n, dtype=torch.float64, device="cuda"), n, n, lam, None, Ab)
    x, lam, got = X.cpu().numpy(), lam.cpu().numpy(), Ab.cpu().numpy()
    # scales of row i of Z and of column j of W after the balancing of each k
    big = np.abs(x.real), np.abs(x.imag)
    big = np.maximum(*big) * np.sqrt(lam)[None, :]
    rmax = big.max(axis=1)
    rng = np.random.default_rng(N)
    for i, j in rng.integers(0, N, (150, 2)):
        re = im = Fraction(0)
        for k in range(n):
            a, b = x[i, k], x[j, k]
            ar, ai, br, bi = map(Fraction, (a.real, a.imag, b.real, b.imag))
            s = Fraction(lam[k])
            re += s * (ar * br + ai * bi)
            im += s * (ai * br - ar * bi)
        bound = np.sqrt(2 * n) * 2.0 ** -52 * rmax[i] * rmax[j] + 2.0 ** -52 * abs(complex(re, im))
        assert abs(complex(Fraction(got[i, j].real) - re, Fraction(got[i, j].imag) - im)) <= bound
