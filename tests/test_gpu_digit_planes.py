"""Digit planes at odd sizes and over wide ranges of exponents, through the
residual norms with theta = 0: ||A v_j||, exact diagonal apart, is off in row i
by at most 2 N (2^-48 + 2^-49) rowmax_i colmax_j (rounding of both operands'
digits and the dropped pairs, all with one sign)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n", [(2, 1), (31, 5), (33, 32), (65, 33), (127, 7), (129, 64),
                                 (255, 40), (385, 3)])
@pytest.mark.parametrize("graded", [0, 1])
def test_digit_products(lib, N, n, graded):
    rng = np.random.default_rng(10 * N + graded)
    A = rng.uniform(-1, 1, (N, N)) + 1j * rng.uniform(-1, 1, (N, N))
    V = rng.uniform(-1, 1, (N, n)) + 1j * rng.uniform(-1, 1, (N, n))
    if graded:
        d = 2.0 ** rng.integers(-20, 20, N)
        A *= d[:, None] * d[None, :]
        V *= 2.0 ** rng.integers(-200, 200, n)[None, :]
        A[0, :] = A[:, 0] = 0.0      # a zero row: only the diagonal is left
        V[-1, :] = 0.0
        V[0, -1] = 5e-324            # subnormal beside normal entries
    A = np.asfortranarray((A + A.conj().T) / 2)
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=1, lanczos_steps=min(N, 2))) as ctx:
        resid = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.chase_residuals(lib.colmajor(torch.from_numpy(A).cuda()),
                            lib.colmajor(torch.from_numpy(np.asfortranarray(V)).cuda()),
                            torch.zeros(n, dtype=torch.float64, device="cuda"), n, resid)
        got = resid.cpu().numpy()
    ref = np.linalg.norm(A @ V, axis=0)
    off = A - np.diag(np.diag(A))
    row = np.linalg.norm(np.maximum(np.abs(off.real), np.abs(off.imag)).max(axis=1))
    col = np.maximum(np.abs(V.real), np.abs(V.imag)).max(axis=0)
    assert np.all(np.abs(got - ref) <= 2 * N * 2.0 ** -47 * row * col + 1e-14 * ref)
