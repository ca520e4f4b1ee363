"""heev_sweeps counts the FP32 sweeps whichever kernel runs them: a problem of 64
columns (one CTA) takes as many steps as one of 65 (blocked), give or take two."""
import pytest

from synth import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def sweeps(lib, nev, nex):
    p = Problem(N=512, nev=nev, nex=nex, spectrum="uniform", lo=0.0, hi=10.0, reflectors=8, seed=3)
    dev = lambda x: lib.colmajor(torch.from_numpy(x).cuda())
    ritz = torch.zeros(nev + nex, dtype=torch.float64, device="cuda")
    with lib.Context(lib.default_params(512, nev, nex, max_iter=1)) as ctx:
        st = ctx.chase_solve(dev(p.matrix()), dev(p.start_block()), ritz, torch.zeros_like(ritz),
                             lanczos_start=dev(p.lanczos_start()), allow_not_converged=True)
    return st["heev_sweeps"]


def test_sweeps_on_both_sides_of_64(lib):
    assert abs(sweeps(lib, 44, 20) - sweeps(lib, 45, 20)) <= 2
