"""The FP32 Jacobi stage, in one CTA and blocked, on matrices whose entries, or whose
entries' squares, FP32 does not hold: it works on a copy scaled by a power of two. The
bounds are those of the block-edge tests."""
import pytest

from test_gpu_block_jacobi import check

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 64, 65, 97])
@pytest.mark.parametrize("scale", [2.0 ** -60, 2.0 ** 40, 1e25, 1e-60, 1e60])
def test_scales(lib, n, scale):
    check(lib, n, 0, n, scale)
