"""A kernel launch that the runtime refuses ends the call with CHASE_ERR_CUDA: a
product must not go on with the digits of an earlier operand, a graph must not be
replayed without one of its steps. The library's objects are linked against a CUDA
runtime that runs no kernels (fake_cudart.cpp) and refuses one launch of a call
after the other. No GPU is used."""
import ctypes
import glob
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
OK, CUDA = 0, 2


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    import paper_2309_15595_gb300 as pkg

    objs = sorted(glob.glob(os.path.join(os.path.dirname(pkg._lib.LIB_PATH), "_build", "*.o")))
    gxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    if gxx is None or not objs or not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("needs g++, the CUDA headers and the library's object files")
    so = str(tmp_path_factory.mktemp("fake") / "libchase_fake.so")
    subprocess.run([gxx, "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include, "-o", so,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-lpthread"], check=True)
    lib = pkg._lib.load(so)
    lib.launches = ctypes.c_longlong.in_dll(lib, "fake_launches")
    lib.fail_at = ctypes.c_longlong.in_dll(lib, "fake_fail_at")
    return lib, pkg


def every_launch_counts(lib, call):
    lib.launches.value = lib.fail_at.value = 0
    assert call() == OK
    total = lib.launches.value
    assert total > 0
    lost = []
    for k in range(1, total + 1):
        lib.launches.value, lib.fail_at.value = 0, k
        if call() != CUDA:
            lost.append(k)
    lib.fail_at.value = 0
    assert not lost, f"of {total} launches"


class Problem:
    def __init__(self, fake, N, ne, tensor, mixed=0):
        self.lib, pkg = fake
        prm = pkg.default_params(N, ne, 0, fp64_tensor=tensor, precision=mixed, max_iter=1,
                                 lanczos_steps=4)
        self.ctx = ctypes.c_void_p()
        assert self.lib.chase_create(ctypes.byref(prm), None, ctypes.byref(self.ctx)) == OK
        self.N, self.ne, self.keep = N, ne, []
        self.A, self.V, self.B = self.array(N * N), self.array(N * ne), self.array(N * ne)
        self.d = self.array(ne)

    def array(self, n):  # "device" memory
        self.keep.append(np.zeros(2 * n))
        return self.keep[-1].ctypes.data

    def close(self):
        self.lib.chase_destroy(self.ctx)


# 60 columns of 700 (digits of a column by one CTA) and of 1100 rows (two passes); in
# both, the adjoints' N x N product runs on the tensor cores
@pytest.mark.parametrize("N,ne", [(700, 60), (1100, 60)])
@pytest.mark.parametrize("op", ["filter", "mixed", "residuals", "rr", "qr1", "qr2", "filter_vjp",
                                "eig_vjp"])
def test_refused_launch(fake, op, N, ne):
    p = Problem(fake, N, ne, 1, int(op == "mixed"))
    L, c, A, V, B, d = p.lib, p.ctx, p.A, p.V, p.B, p.d
    degs = (ctypes.c_int32 * ne)(*([2] * (ne // 2) + [4] * (ne - ne // 2)))
    call = {
        "filter": lambda: L.chase_filter(c, A, N, V, N, ne, degs, 0.5, 1.0, -1.0, 0),
        "mixed": lambda: L.chase_filter(c, A, N, V, N, ne, degs, 0.5, 1.0, -1.0, 1),
        "residuals": lambda: L.chase_residuals(c, A, N, V, N, d, ne, d),
        "rr": lambda: L.chase_rayleigh_ritz(c, A, N, V, N, ne, d),
        "qr1": lambda: L.chase_qr(c, V, N, ne, 10.0, None),
        "qr2": lambda: L.chase_qr(c, V, N, ne, 1e4, None),
        "filter_vjp": lambda: L.chase_filter_vjp(c, A, N, V, N, ne, 4, 0.5, 1.0, -1.0, B, N,
                                                 p.array(N * N), N, p.array(N * ne), N, 0),
        "eig_vjp": lambda: L.chase_eig_vjp(c, A, N, V, N, d, ne, ne, d, B, N, p.array(N * N), N,
                                           1e-10, 8, None),
    }[op]
    every_launch_counts(L, call)
    p.close()


@pytest.mark.parametrize("mixed", [0, 1])
def test_refused_launch_in_a_batch(fake, mixed):
    # two worker threads: an error left behind by the grouped filter's thread is not theirs
    probs = [Problem(fake, N, ne, 1, mixed) for N, ne in ((300, 20), (200, 12))]
    L, n = probs[0].lib, len(probs)
    ptrs = lambda xs: (ctypes.c_void_p * n)(*xs)
    ld = (ctypes.c_int64 * n)(*(p.N for p in probs))
    status = (ctypes.c_int32 * n)()
    args = (ptrs(p.ctx.value for p in probs), ptrs(p.A for p in probs), ld,
            ptrs(p.V for p in probs), ld, None, None, ptrs(p.d for p in probs),
            ptrs(p.array(p.ne) for p in probs), None, status, 2)
    every_launch_counts(L, lambda: L.chase_solve_batch(n, *args))
    for p in probs:
        p.close()
