"""CholeskyQR of blocks at the ends of FP64's range: the Gram matrix of a block
scaled by 2^-519 has subnormal pivots of 44 good bits, one scaled by 2^505 pivots
near the largest numbers. Neither is a breakdown: the variant is the one of the
unscaled block, and the factor is orthonormal (a second pass repairs the first's
2^-36 at the most) and spans the block."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-519, -505, 0, 505])
@pytest.mark.parametrize("tensor", [0, 1])
def test_scaled_block(lib, exponent, tensor):
    N, n = 300, 70
    rng = np.random.default_rng(4)
    X0 = rng.standard_normal((N, n)) + 1j * rng.standard_normal((N, n))
    X = np.asfortranarray(X0 * 2.0 ** exponent)
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=tensor)) as ctx:
        Vd = lib.colmajor(torch.from_numpy(X).cuda())
        variant = ctx.chase_qr(Vd, n, 1e4)
        Q = Vd.cpu().numpy()
    assert variant == lib.CHASE_QR_CHOLQR2
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() <= 1e-12
    assert np.abs(X0 - Q @ (Q.conj().T @ X0)).max() <= 1e-8 * np.abs(X0).max()
