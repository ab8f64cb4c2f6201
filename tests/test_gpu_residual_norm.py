"""GPU tests of the refinement residual's norm."""
import numpy as np
import pytest

from oracle import poisson as P
from paper_2402_17913_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2402_17913_gb300 import build, lib
    build.build()
    lib.load()
    return lib


def first_residual(L, shape, h, bc, solid, b, x0):
    """||b - A x0|| as the solve reports it, and in float64."""
    st = None if solid is None else torch.from_numpy(solid.astype(np.uint8)).cuda()
    hdl = L.mg_create(len(shape), tuple(reversed(shape)), h, bc, st)
    try:
        x = torch.from_numpy(x0).cuda()
        _, s = L.mg_solve(hdl, torch.from_numpy(b).cuda(), x, 1e-6)
    finally:
        L.mg_destroy(hdl)
    lv = P.Level(shape, h, bc, solid)
    x64 = x0.astype(np.float64) * lv.fluid
    return s["relres0"] * s["bnorm"], np.linalg.norm((b.astype(np.float64) - P.apply_A(lv, x64)) * lv.fluid)


NORM = [((40, 64), (0, 0, 0, 0), 0.0), ((36, 50), (1, 0, 1, 1), 0.06), ((16, 24, 40), (1, 0, 1, 1, 0, 1), 0.06),
        ((12, 14, 18), (0,) * 6, 0.0)]


@pytest.mark.parametrize("shape,bc,frac", NORM)
@pytest.mark.parametrize("stretch", [1.0, 0.75])
def test_norm_of_the_float64_residual(L, shape, bc, frac, stretch):
    """The norm is that of the float64 residual: r has no cancellation here
    (a random guess), so each cell's float64 residual is good to a few 2^-53
    and the norm's sums to 2^-48; 1e-12 is well above both.  Squares of r
    rounded to float32 would miss it by 2^-25 / sqrt(cells), 1e-10 and more."""
    rng = np.random.default_rng(8)
    solid = I.flood_fill_unreachable(rng.random(shape) < frac, bc) if frac > 0 else None
    h = (0.125,) * (len(shape) - 1) + (0.125 * stretch,)
    b = rng.standard_normal(shape).astype(np.float32)
    x0 = rng.standard_normal(shape).astype(np.float32)
    got, ref = first_residual(L, shape, h, bc, solid, b, x0)
    assert abs(got - ref) <= 1e-12 * ref, (got / ref - 1.0)
