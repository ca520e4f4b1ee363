"""Every tile width of the reduced-precision filter (32, 64, 128 complex columns,
chosen by the number of rows and columns), with a ragged last tile and with
degrees that leave some of its columns, against the FP64 recurrence: at most
degs[j] 2^-16 of the column's largest entry, as the other tests of this filter."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n", [(300, 1), (300, 33), (520, 97), (2600, 195), (2600, 500),
                                 (2600, 600), (2600, 700), (2700, 129)])
def test_widths(lib, N, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(N + n)
    Z = torch.randn(N, N, dtype=torch.complex128, device="cuda", generator=g)
    A = lib.colmajor((Z + Z.mH) / (4 * N ** 0.5))
    V = lib.colmajor(torch.randn(n, N, dtype=torch.complex128, device="cuda", generator=g).mT)
    degs = np.full(n, 4, dtype=np.int32)
    degs[: n // 3] = 2
    c, e, mu = 0.3, 0.9, -1.2
    s1 = e / (mu - c)
    al, be, s = [0.0, s1 / e], [0.0, 0.0], s1
    for _ in range(2, 5):
        nx = 1.0 / (2.0 / s1 - s)
        al.append(2.0 * nx / e)
        be.append(-s * nx)
        s = nx
    Y = [V]
    for i in range(1, 5):
        y = al[i] * (A @ Y[-1] - c * Y[-1])
        Y.append(y + be[i] * Y[-2] if i > 1 else y)
    ref = Y[4].clone()
    ref[:, : n // 3] = Y[2][:, : n // 3]
    prm = lib.default_params(N, n, 0, precision=lib.CHASE_MIXED_BF16X3)
    with lib.Context(prm) as ctx:
        got = lib.colmajor(V.clone())
        ctx.chase_filter(A, got, n, degs, c, e, mu, precision=lib.CHASE_MIXED_BF16X3)
    rel = ((got - ref).abs().amax(0) / ref.abs().amax(0)).cpu().numpy()
    assert np.all(rel <= degs * 2.0 ** -16)
