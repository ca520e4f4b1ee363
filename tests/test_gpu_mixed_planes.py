"""BF16 hi / lo planes at odd sizes (two entries a lane, the last one past the
end) and with entries that FP32 holds as subnormals or not at all, against the
FP64 recurrence: degree 2, at most degs[j] 2^-16 of the column's largest entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n", [(3, 1), (63, 5), (65, 2), (129, 129), (191, 7)])
@pytest.mark.parametrize("tiny", [0, 1])
def test_planes(lib, N, n, tiny):
    rng = np.random.default_rng(N + tiny)
    A = rng.uniform(0.1, 1, (N, N)) + 1j * rng.uniform(-1, 1, (N, N))
    A = np.asfortranarray((A + A.conj().T) / 2)
    V = np.asfortranarray(rng.uniform(0.1, 1, (N, n)) + 1j * rng.uniform(-1, 1, (N, n)))
    if tiny:
        A[0, -1] = A[-1, 0] = 1e-310
        A[1, 0] = A[0, 1] = 3e-41
        V[0, :] = 1e-42
        V[-1, 0] = -0.0
    c, e, mu1 = 0.5, 1.0, -2.0
    prm = lib.default_params(N, n, 0, precision=lib.CHASE_MIXED_BF16X3, lanczos_steps=min(N, 2))
    with lib.Context(prm) as ctx:
        Vd = lib.colmajor(torch.from_numpy(V).cuda())
        ctx.chase_filter(lib.colmajor(torch.from_numpy(A).cuda()), Vd, n,
                         np.full(n, 2, dtype=np.int32), c, e, mu1,
                         precision=lib.CHASE_MIXED_BF16X3)
        got = Vd.cpu().numpy()
    s1 = e / (mu1 - c)
    s2 = 1.0 / (2.0 / s1 - s1)
    Y1 = (s1 / e) * (A @ V - c * V)
    ref = (2 * s2 / e) * (A @ Y1 - c * Y1) - s1 * s2 * V
    assert np.all(np.isfinite(got))
    rel = np.abs(got - ref).max(axis=0) / np.abs(ref).max(axis=0)
    assert np.all(rel <= 2 * 2.0 ** -16)
