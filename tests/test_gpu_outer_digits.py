"""The filter adjoint's outer product on the tensor cores (from 2e8 FP64 operations
on): column blocks with a ragged last one, several parts of K, orders around the
line between the CUDA-core and the tensor-core product, against torch in FP64.

Z and Y come from digit-sliced products here and FP64 ones in the reference: each
of the `deg` steps of both recurrences carries at most 2^-42 of the column's largest
entry (the bound of the filter's own tests), so the adjoint, a sum of deg products
of the two, carries at most 2 deg 2^-42 of sum_i |Z_i| |Y_i|, entry by entry of the
maxima's product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n,deg", [(500, 40, 6), (700, 33, 4), (1031, 130, 6), (1300, 17, 10)])
def test_filter_adjoint(lib, N, n, deg):
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    Z = torch.randn(N, N, dtype=torch.complex128, device="cuda", generator=g)
    A = lib.colmajor((Z + Z.mH) / (4 * N ** 0.5))
    V = lib.colmajor(torch.randn(n, N, dtype=torch.complex128, device="cuda", generator=g).mT)
    Yb = lib.colmajor(torch.randn(n, N, dtype=torch.complex128, device="cuda", generator=g).mT)
    c, e, mu = 0.3, 0.9, -1.2
    s1 = e / (mu - c)
    al, be, s = [0.0, s1 / e], [0.0, 0.0], s1
    for _ in range(2, deg + 1):
        nx = 1.0 / (2.0 / s1 - s)
        al.append(2.0 * nx / e)
        be.append(-s * nx)
        s = nx
    be.append(0.0)
    Y = [V]
    for i in range(1, deg + 1):
        y = al[i] * (A @ Y[-1] - c * Y[-1])
        Y.append(y + be[i] * Y[-2] if i > 1 else y)
    z1, z = torch.zeros_like(V), Yb
    G, size = torch.zeros_like(A), 0.0
    for i in range(deg, 0, -1):
        G += al[i] * (z @ Y[i - 1].mH)
        size += abs(al[i]) * float(z.abs().max()) * float(Y[i - 1].abs().max()) * n
        z, z1 = al[i] * (A @ z - c * z) + be[i + 1] * z1, z
    G = (G + G.mH) / 2
    Ab, Vb = torch.empty_like(A), torch.empty_like(V)
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=1)) as ctx:
        ctx.chase_filter_vjp(A, V, n, deg, c, e, mu, Yb, lib.colmajor(Ab), lib.colmajor(Vb))
    assert float((lib.colmajor(Ab) - G).abs().max()) <= 2 * deg * 2.0 ** -42 * size
    assert float((Vb - z).abs().max()) <= deg * 2.0 ** -42 * float(z.abs().max())
