"""The FP32 Jacobi stage, in one CTA and blocked, on matrices whose entries FP32 holds
but whose squares, at 2^-60, it does not (its rotations are formed from 2^50 times the
block there). The bounds are those of the block-edge tests."""
import pytest

from test_gpu_block_jacobi import check

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 64, 65, 97])
@pytest.mark.parametrize("scale", [2.0 ** -60, 2.0 ** 40])
def test_scales(lib, n, scale):
    check(lib, n, 0, n, scale)
