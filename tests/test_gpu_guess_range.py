"""GPU test of a guess far from the solution: the inner solve then works on
numbers far above those of the right-hand side."""
import numpy as np
import pytest

from test_gpu_rhs_range import L, poisson, unit_rhs  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(320, 448), (32, 48, 64), (64, 64, 72)])
def test_guess_of_a_large_residual_is_solved(L, shape):  # noqa: F811
    """||b - A x0|| / ||b|| about 1e18: r' squared fits float32 in a thread's
    cells but not over the grid.  The solution is that from a zero guess to
    the two solves' residuals (1e-6 of b; ||A^-1|| ||b|| / ||x|| is at most
    about 30 for these blobs)."""
    b = unit_rhs(shape)
    x0 = torch.from_numpy(np.random.default_rng(4).uniform(-1.0, 1.0, shape).astype(np.float32)).cuda()
    x0 *= 2.0 ** 56 * torch.linalg.norm(b).item() / b.numel() ** 0.5
    status, st, ref = poisson(L, b)
    assert status == L.MG_OK
    status, st, x = poisson(L, b, x0=x0)
    assert status == L.MG_OK and st["relres0"] > 1e16 and st["relres"] <= 1e-6, st
    assert torch.linalg.norm(x - ref) <= 1e-4 * torch.linalg.norm(ref)
