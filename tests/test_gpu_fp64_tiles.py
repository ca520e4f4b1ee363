"""CUDA-core FP64 products at the edges of their 16 x 16 tiles (64 x 16 for the
residual epilogue), 8-deep K slabs and split-K Grams, against numpy.

A dot product of N complex terms summed in FP64 in any order is off by at most
4 N 2^-53 of sum |a||b| (each real sum has 2 N products; twice that for the
reference's own rounding), and sum |a||b| <= N max|a| max|b|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rand(rng, m, n):
    return np.asfortranarray((rng.uniform(-1, 1, (m, n)) + 1j * rng.uniform(-1, 1, (m, n))))


def hermitian(rng, N):
    A = rand(rng, N, N)
    return np.asfortranarray((A + A.conj().T) / 2)


def dev(x, lib):
    return lib.colmajor(torch.from_numpy(np.asfortranarray(x)).cuda())


@pytest.mark.parametrize("N,n", [(2, 1), (15, 3), (16, 16), (17, 17), (63, 15), (65, 33),
                                 (130, 64), (257, 31)])
def test_filter_and_residuals(lib, N, n):
    rng = np.random.default_rng(100 * N + n)
    A, V = hermitian(rng, N), rand(rng, N, n)
    theta = rng.uniform(-1, 1, n)
    u = 4 * N * 2.0 ** -53
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=0, lanczos_steps=min(N, 2))) as ctx:
        Vd, Ad = dev(V, lib), dev(A, lib)
        resid = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.chase_residuals(Ad, Vd, torch.from_numpy(theta).cuda(), n, resid)
        c, e, mu1 = 0.25, 1.0, -2.0
        ctx.chase_filter(Ad, Vd, n, np.full(n, 2, dtype=np.int32), c, e, mu1)
        got = Vd.cpu().numpy()
    size = np.abs(A).max() * np.abs(V).max() * N  # of an entry of A V
    r = np.linalg.norm(A @ V - V * theta[None, :], axis=0)
    assert np.all(np.abs(resid.cpu().numpy() - r) <= u * 2 * size * np.sqrt(N))
    s1 = e / (mu1 - c)
    s2 = 1.0 / (2.0 / s1 - s1)
    Y1 = (s1 / e) * (A @ V - c * V)
    ref = (2 * s2 / e) * (A @ Y1 - c * Y1) - s1 * s2 * V
    assert np.abs(got - ref).max() <= 8 * u * size * N * np.abs(A).max()


@pytest.mark.parametrize("m,n", [(64, 5), (129, 17), (1025, 16), (4099, 5), (3001, 40)])
def test_gram_splits_through_qr(lib, m, n):
    # CholeskyQR2's orthogonality is the Gram's error: m 2^-53 of the unit columns
    rng = np.random.default_rng(m + n)
    X = rand(rng, m, n)
    with lib.Context(lib.default_params(m, n, 0, fp64_tensor=0)) as ctx:
        Xd = dev(X, lib)
        ctx.chase_qr(Xd, n, 1e3)
        Q = Xd.cpu().numpy()
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() <= 8 * m * 2.0 ** -53
    R = Q.conj().T @ X
    assert np.abs(np.tril(R, -1)).max() <= 1e-12 * np.abs(R).max()
