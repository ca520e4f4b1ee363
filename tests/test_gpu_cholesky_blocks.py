"""Cholesky factorisation and triangular inverse at the edges of the 64-wide
diagonal blocks and the 16-wide tiles of the trailing update, through one
CholeskyQR pass (condition estimate below 20) and through a failing pivot.

One pass on a block of condition kappa <= 4 leaves an orthogonality error of
kappa^2 times the relative errors of the Gram (m 2^-53) and of the
factorisation (n 2^-53 each for U and U^-1): 16 (m + 2 n) 2^-53 bounds it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def block(m, n, seed):
    rng = np.random.default_rng(seed)
    Z = rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))
    U, _, Wh = np.linalg.svd(Z, full_matrices=False)
    return np.asfortranarray((U * np.linspace(1.0, 0.25, n)[None, :]) @ Wh)


@pytest.mark.parametrize("tensor", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 16, 17, 63, 64, 65, 80, 128, 129, 200])
def test_one_pass(lib, n, tensor):
    m = 2 * n + 100
    X = block(m, n, n)
    with lib.Context(lib.default_params(m, n, 0, fp64_tensor=tensor)) as ctx:
        Xd = lib.colmajor(torch.from_numpy(X).cuda())
        assert ctx.chase_qr(Xd, n, 4.0) == 1
        Q = Xd.cpu().numpy()
    R = Q.conj().T @ X
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() <= 16 * (m + 2 * n) * 2.0 ** -53
    assert np.abs(np.tril(R, -1)).max() <= 16 * (m + 2 * n) * 2.0 ** -53
    assert np.all(np.diag(R).real > 0)


@pytest.mark.parametrize("n,bad", [(30, 0), (70, 64), (130, 100)])
def test_zero_column_fails_the_pivot(lib, n, bad):
    # a zero pivot in the first block, at the start of the second and inside it:
    # both Cholesky variants give up and the Householder factorisation answers
    m = 300
    X = block(m, n, 3 * n)
    X[:, bad] = 0.0
    with lib.Context(lib.default_params(m, n, 0, fp64_tensor=0)) as ctx:
        Xd = lib.colmajor(torch.from_numpy(X).cuda())
        v = ctx.chase_qr(Xd, n, 4.0)
        Q = Xd.cpu().numpy()
    assert v in (3, 4)
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() <= 1e-12
