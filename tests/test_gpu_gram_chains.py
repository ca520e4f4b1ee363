"""A Gram matrix on the CUDA cores is summed in parts of at most about 512 rows (eight
parts at the most): the rounding of a sum grows with the length of its chain. The
columns are those of a Hadamard matrix times a number whose square, added up N times,
is rounded the same way almost every time while a partial sum lies in [1/4, 1/2), as
half of the sum does: two parts of 1536 rows give -4.1e-14, six of 512 give 1e-16.
The bound is the largest error that any number could give in six parts: half a unit
in the last place of the partial sum for each of the 512 additions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def hadamard(N):  # order 12 (Paley), doubled
    q = np.arange(11)
    chi = np.where(q == 0, 0, np.where(np.isin(q, q[1:] ** 2 % 11), 1, -1))
    S = np.block([[np.zeros((1, 1)), np.ones((1, 11))],
                  [-np.ones((11, 1)), chi[(q[None, :] - q[:, None]) % 11]]])
    H = S + np.eye(12)
    while len(H) < N:
        H = np.block([[H, H], [H, -H]])
    return H


@pytest.mark.parametrize("n", [150, 400])
def test_rounding_of_a_gram(lib, n):
    N, parts = 3072, 6
    H = hadamard(N)
    assert np.array_equal(H @ H.T, N * np.eye(N))
    c = float.fromhex("0x1.28f5cb86b7df9p-6")
    Q = np.asfortranarray((c * H[:, :n]).astype(complex))
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=0)) as ctx:
        Vd = lib.colmajor(torch.from_numpy(Q).cuda())
        ritz = torch.zeros(n, dtype=torch.float64, device="cuda")
        A = lib.colmajor(torch.eye(N, dtype=torch.complex128, device="cuda"))
        ctx.chase_rayleigh_ritz(A, Vd, n, ritz)
    sums = c * c * np.arange(1, N // parts + 1)
    bound = parts * (np.spacing(sums) / 2).sum() + 2 * parts * 2.0 ** -53
    assert bound < 2.3e-14
    assert np.abs(ritz.cpu().numpy() - N * c * c).max() <= bound
