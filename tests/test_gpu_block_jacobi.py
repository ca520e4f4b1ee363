"""The blocked FP32 Jacobi stage at the edges of its 32-wide blocks (a last block
of 1, 31, 32 or 33 columns, an odd number of blocks), through Rayleigh-Ritz
against numpy. The FP64 refinement that follows has to reach FP64 accuracy: n
times 2^-48 of ||A|| for the values and the residuals (the tensor-core products'
digits; the CUDA-core ones are better)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def check(lib, n, tensor, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    N = n + 37
    Z = rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))
    A = np.asfortranarray((Z + Z.conj().T) / 2) * scale
    Q = np.asfortranarray(np.linalg.qr(Z[:, :n])[0])
    ref = np.linalg.eigvalsh(Q.conj().T @ A @ Q)
    nA = np.linalg.norm(A, 2)
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=tensor)) as ctx:
        Vd = lib.colmajor(torch.from_numpy(Q).cuda())
        ritz = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.chase_rayleigh_ritz(lib.colmajor(torch.from_numpy(A).cuda()), Vd, n, ritz)
        V, th = Vd.cpu().numpy(), ritz.cpu().numpy()
    bound = n * 2.0 ** -48
    assert np.abs(th - ref).max() <= bound * nA
    G = V.conj().T @ A @ V
    assert np.abs(V.conj().T @ V - np.eye(n)).max() <= 1e-12
    assert np.abs(G - np.diag(th)).max() <= bound * nA


@pytest.mark.parametrize("n", [65, 66, 95, 96, 97, 127, 129, 161])
@pytest.mark.parametrize("tensor", [0, 1])
def test_block_edges(lib, n, tensor):
    check(lib, n, tensor, n)
