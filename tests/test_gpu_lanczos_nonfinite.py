"""Lanczos bounds with a NaN or infinity in the start vectors or the matrix: the pooled
Ritz values are sorted by rank before the eigensolver's failure is known, and NaN take
ranks of their own, so that every slot of the order holds an index. A NaN in a
recurrence of several steps is an error; the device goes on working."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,steps,nvec", [(31, 25, 4), (31, 2, 1), (300, 25, 8), (300, 64, 6), (5, 1, 2)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["one", "all", "matrix"])
@pytest.mark.parametrize("tensor", [0, 1])
def test_bounds(lib, N, steps, nvec, bad, where, tensor):
    rng = np.random.default_rng(N)
    Z = rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))
    A = Z + Z.conj().T
    Q0 = rng.standard_normal((N, nvec)) + 1j * rng.standard_normal((N, nvec))
    if where == "matrix":
        A[2, 2] = bad
    else:
        Q0[1, 0 if where == "one" else slice(None)] = bad
    dev = lambda x: lib.colmajor(torch.from_numpy(np.asfortranarray(x)).cuda())
    prm = lib.default_params(N, 1, 0, fp64_tensor=tensor, lanczos_steps=steps, lanczos_vecs=nvec)
    with lib.Context(prm) as ctx:
        if steps > 1 and np.isnan(bad):
            with pytest.raises(Exception, match="HEEV_NOCONV"):
                ctx.chase_lanczos(dev(A), dev(Q0))
        else:
            try:
                ctx.chase_lanczos(dev(A), dev(Q0))
            except Exception as e:
                assert "HEEV_NOCONV" in str(e)
    torch.cuda.synchronize()
