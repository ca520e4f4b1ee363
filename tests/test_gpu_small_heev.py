"""Rayleigh-Ritz problems of order up to 64: in FP64 in one CTA up to order 24,
from FP32 sweeps in one CTA and FP64 refinement above. Both sides of the line
and the largest order, over scales that FP32 cannot hold, degenerate spectra,
diagonal input and a NaN."""
import numpy as np
import pytest

from test_gpu_block_jacobi import check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 23, 24, 25, 26, 31, 32, 33, 50, 63, 64])
@pytest.mark.parametrize("scale", [1.0, 1e-60, 1e60])
def test_orders_and_scales(lib, n, scale):
    check(lib, n, 0, n, scale)


@pytest.mark.parametrize("n", [24, 25, 60, 64])
@pytest.mark.parametrize("kind", ["degenerate", "diagonal", "zero", "close"])
def test_spectra(lib, n, kind):
    rng = np.random.default_rng(n)
    N = n + 11
    H = np.linalg.qr(rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N)))[0]
    lam = np.linspace(1.0, 2.0, N)
    if kind == "degenerate":
        lam[: n // 2] = 1.0
    if kind == "close":
        lam[: n // 2] = 1.0 + 1e-11 * np.arange(n // 2)
    if kind == "zero":
        lam[:] = 0.0
    A = (H * lam[None, :]) @ H.conj().T
    Q = np.asfortranarray(H[:, :n] @ np.linalg.qr(rng.standard_normal((n, n)))[0])
    if kind == "diagonal":
        A, Q = np.diag(lam).astype(complex), np.asfortranarray(np.eye(N, n, dtype=complex))
    A = np.asfortranarray((A + A.conj().T) / 2)
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=0)) as ctx:
        Vd = lib.colmajor(torch.from_numpy(Q).cuda())
        ritz = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.chase_rayleigh_ritz(lib.colmajor(torch.from_numpy(A).cuda()), Vd, n, ritz)
        V, th = Vd.cpu().numpy(), ritz.cpu().numpy()
    bound = n * 2.0 ** -48 * max(1.0, lam.max())
    assert np.abs(th - np.sort(lam[:n])).max() <= bound
    assert np.abs(V.conj().T @ V - np.eye(n)).max() <= 1e-12
    assert np.abs(V.conj().T @ A @ V - np.diag(th)).max() <= bound


@pytest.mark.parametrize("n", [20, 40])
def test_nan_is_an_error(lib, n):
    A = np.eye(n + 5, dtype=complex)
    A[1, 0] = A[0, 1] = np.nan
    with lib.Context(lib.default_params(n + 5, n, 0, fp64_tensor=0)) as ctx:
        Vd = lib.colmajor(torch.from_numpy(np.eye(n + 5, n, dtype=complex, order="F")).cuda())
        ritz = torch.zeros(n, dtype=torch.float64, device="cuda")
        with pytest.raises(Exception):
            ctx.chase_rayleigh_ritz(lib.colmajor(torch.from_numpy(A).cuda()), Vd, n, ritz)
