"""The digit-sliced FP64 product over 1 to 9 exact chunks of 256 K values: levels
2 and 3 are drained every four and every two chunks and at the end, so every
remainder of the chunk count occurs, with operands whose digits all lie near
+-127 and add up with one sign (the largest sums the accumulators can hold).

One filter step pair (degree 2) against numpy in FP64. Error bound per column:
each product of K = 2N terms is off by at most K 2^-48 of max|a| max|y|
(rounding of the operands' digits and dropped pairs, all with one sign), and
the columns here have the size N max|a| max|y|, so 2^-47 of it per degree; the
bound is 16 times that. One lost or doubled chunk of any level from 2 to 5
exceeds it (level 5 weighs 2^-24 of the result and is 1/9 of it at least)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# all digits 127 but the last: 0.5 (1 - 2^-7) in base 256
ONE_SIGN = sum(127 / 256.0 ** s for s in range(1, 7))


@pytest.mark.parametrize("N", [100, 200, 384, 400, 513, 700, 800, 1000, 1100])
def test_chunk_remainders(lib, N):
    n = 33
    A = np.full((N, N), ONE_SIGN, dtype=np.complex128)
    A += np.triu(np.full((N, N), 1j * ONE_SIGN), 1) + np.tril(np.full((N, N), -1j * ONE_SIGN), -1)
    V = np.full((N, n), ONE_SIGN * (1 + 1j)) * (1.0 + np.arange(n))[None, :]
    c, e, mu1 = 0.0, 1.0, -2.0
    s1 = e / (mu1 - c)
    s2 = 1.0 / (2.0 / s1 - s1)
    Y1 = (s1 / e) * (A @ V)
    ref = (2 * s2 / e) * (A @ Y1) - s1 * s2 * V
    with lib.Context(lib.default_params(N, n, 0, fp64_tensor=1)) as ctx:
        Vd = lib.colmajor(torch.from_numpy(np.asfortranarray(V)).cuda())
        Ad = lib.colmajor(torch.from_numpy(np.asfortranarray(A)).cuda())
        ctx.chase_filter(Ad, Vd, n, np.full(n, 2, dtype=np.int32), c, e, mu1)
        got = Vd.cpu().numpy()
    rel = np.abs(got - ref).max(axis=0) / np.abs(ref).max(axis=0)
    assert np.all(rel <= 2 * 16 * 2.0 ** -47)
