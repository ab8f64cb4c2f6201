"""GPU test of the refinement residual on zeros and numbers near float32's
smallest, whose exponents lie far below that of c b for b = 1."""
import numpy as np
import pytest

from test_gpu_residual_norm import L, first_residual  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stretch", [1.0, 0.75])
def test_zero_and_tiny_values(L, stretch):  # noqa: F811
    """A guess that is zero on most of the grid, b zero on another part, and
    numbers near float32's smallest beside zeros of b."""
    rng = np.random.default_rng(9)
    shape, bc, h = (48, 72), (0, 1, 0, 0), (0.125, 0.125 * stretch)
    b = rng.standard_normal(shape).astype(np.float32)
    b[:, 40:] = 0.0
    x0 = np.zeros(shape, np.float32)
    x0[20:30, 10:30] = rng.standard_normal((10, 20)).astype(np.float32)
    x0[:, 56:60] = 1e-44
    got, ref = first_residual(L, shape, h, bc, None, b, x0)
    assert abs(got - ref) <= 1e-12 * ref, (got / ref - 1.0)
    # b = 0 beside tiny x: only the tiny cells count
    b[:] = 0.0
    b[3, 5] = 1e-15
    x0[:] = 0.0
    x0[30, 61] = 3e-39
    got, ref = first_residual(L, shape, h, bc, None, b, x0)
    assert abs(got - ref) <= 1e-6 * ref, (got / ref - 1.0)
