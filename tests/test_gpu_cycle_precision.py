"""GPU test of how far one cycle is from the float64 oracle's: no further than
float32 legs around an exact coarse cycle are.  The legs of the levels above
2048 cells are emulated in numpy float32, the cycle of the others in float64,
rounded once.  The GPU's float32 product with the coarse matrix, whose lanes
add up to sixteen terms, may add half as much again (in squares: 1.12), and
the order of a stencil's sums differs: 1.3."""
import numpy as np
import pytest

from oracle import poisson as P
from paper_2402_17913_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

F = np.float32
OMEGA = 2.0 / 3.0


@pytest.fixture(scope="module")
def L():
    from paper_2402_17913_gb300 import build, lib
    build.build()
    lib.load()
    return lib


def neighbours(x):
    """Sum of the neighbours along each axis, 0 beyond the grid."""
    total = F(0)
    for ax in range(x.ndim):
        lo, hi = np.zeros_like(x), np.zeros_like(x)
        n = x.shape[ax]
        at = lambda a, b: tuple(slice(a, b) if k == ax else slice(None) for k in range(x.ndim))  # noqa: E731
        lo[at(1, n)] = x[at(0, n - 1)]
        hi[at(0, n - 1)] = x[at(1, n)]
        total = total + (lo + hi)
    return total


def cycle32(hier, b, c):
    """V(2,2) on A' = c A_h with float32 legs; b, result in float32.  The
    level's axis weight c / h_k^2 is a power of four."""
    lv = hier[0]
    if b.size <= 2048:
        return (P.Multigrid(hier, s=1.0).precondition(b.astype(np.float64)) / c).astype(F)
    wt = F(c / lv.h[0] ** 2)
    d = (c * lv.diag).astype(F)
    w, keep = F(OMEGA) / d, F(1) - F(OMEGA)
    sweep = lambda x: keep * x + w * (b + wt * neighbours(x))  # noqa: E731
    x = sweep(w * b)
    r = b - (d * x - wt * neighbours(x))
    x = x + P.prolong(cycle32(hier[1:], P.restrict(r).astype(F), c).astype(np.float64), lv).astype(F)
    return sweep(sweep(x))


CASES = [((64, 64), (0, 0, 0, 0)), ((40, 96), (0, 0, 0, 0)), ((136, 144), (0, 0, 0, 0))]


@pytest.mark.parametrize("shape,bc", CASES)
def test_cycle_is_as_close_as_float32_legs(L, shape, bc):
    h = (1.0 / 64,) * len(shape)
    got, want = [], []
    hdl = L.mg_create(len(shape), tuple(reversed(shape)), h, bc)
    try:
        hier = P.build_hierarchy(shape, h, bc, None, levels=L.mg_num_levels(hdl))
        for seed in range(3):
            r = I.blob_rhs(shape, seed).astype(F)
            ref = P.Multigrid(hier, s=1.0).precondition(r.astype(np.float64)) / h[0] ** 2
            z = torch.empty(shape, device="cuda")
            L.mg_precondition(hdl, torch.from_numpy(r).cuda(), z)
            for out, v in ((got, z.cpu().numpy()), (want, cycle32(hier, r, h[0] ** 2))):
                out.append(np.linalg.norm(v - ref) / np.linalg.norm(ref))
    finally:
        L.mg_destroy(hdl)
    assert max(want) <= 2e-7 and np.mean(got) <= 1.3 * np.mean(want), (got, want)
