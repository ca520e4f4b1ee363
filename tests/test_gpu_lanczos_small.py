"""The real eigensolver of the Lanczos tridiagonals and the chained reductions of the
Lanczos vectors: 1 to 64 steps (even and odd orders), 1 to 8 vectors, orders of A
around the reductions' blocks, against the CPU oracle; a spectrum scaled out of
FP32's range; the complex solver is covered by the small Rayleigh-Ritz tests.

Bound: 1e-11 of ||A||, as the other Lanczos tests (the recurrence loses at most
k 2^-53 of ||A|| a step on both sides, the eigensolver 1e-15 of the tridiagonal)."""
import numpy as np
import pytest

from oracle import chase_oracle as O
from synth import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,k,nvec", [(80, 1, 1), (80, 2, 4), (100, 24, 3), (129, 25, 4),
                                      (300, 37, 8), (257, 10, 6), (256, 64, 2)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 200])
def test_bounds(lib, N, k, nvec, scale):
    p = Problem(N=N, nev=8, nex=4, spectrum="uniform", lo=-1.0, hi=3.0, reflectors=4, seed=N)
    A = np.asfortranarray(p.matrix() * scale)
    Q0 = p.lanczos_start(nvec)
    ref = O.lanczos_bounds(A, Q0, k, p.ne)
    prm = lib.default_params(N, p.nev, p.nex, lanczos_steps=k, lanczos_vecs=nvec)
    with lib.Context(prm) as ctx:
        got = ctx.chase_lanczos(lib.colmajor(torch.from_numpy(A).cuda()),
                                lib.colmajor(torch.from_numpy(Q0).cuda()))
    # mu_ne picks one Ritz value by accumulated weights: not a continuous quantity
    err = np.abs([got[0] - ref.b_sup, got[1] - ref.mu_1, got[3] - ref.norm_est])
    assert err.max() <= 1e-11 * p.norm2() * scale
