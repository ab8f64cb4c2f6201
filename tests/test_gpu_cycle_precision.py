"""GPU test of how far one cycle is from the float64 oracle's: no further than
float32 legs around a coarse matrix that is exact up to its float32 rounding.
The legs of the levels above 2048 cells and the product are emulated in numpy
float32 (128 partial sums a row; where b changes sign the product rounds as
much as the legs do).  The order and fusing of a stencil's sums differ: 1.3."""
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


def product32(hier, b, c, kept):
    """M b (M kept for the next b) with the columns of M rounded to float32 and the products added in
    float32: lane l takes columns 4 (l + 32 k) .. + 3 into sum k mod 4."""
    mg, n = P.Multigrid(hier, s=1.0), b.size
    if "m" not in kept:
        m = kept["m"] = np.zeros((n, 2048), F)
        for j in range(n):
            e = np.zeros(n)
            e[j] = 1.0
            m[:, j] = (mg.precondition(e.reshape(b.shape)) / c).ravel()
    v = np.zeros(2048, F)
    v[:n] = b.ravel()
    m, v = kept["m"].reshape(n, 16, 32, 4), v.reshape(16, 32, 4)
    acc = np.zeros((n, 32, 4), F)
    for k in range(16):
        for q in range(4):
            acc[:, :, k & 3] = (m[:, k, :, q].astype(np.float64) * v[k, :, q] + acc[:, :, k & 3]).astype(F)
    t = (acc[:, :, 0] + acc[:, :, 1]) + (acc[:, :, 2] + acc[:, :, 3])
    for o in (16, 8, 4, 2, 1):
        t = t + t[:, np.arange(32) ^ o]
    return t[:, 0].reshape(b.shape)


def cycle32(hier, b, c, kept):
    """V(2,2) on A' = c A_h with float32 legs; b, result in float32.  The
    level's axis weight c / h_k^2 is a power of four."""
    lv = hier[0]
    if b.size <= 2048:
        return product32(hier, b, c, kept)
    wt = F(c / lv.h[0] ** 2)
    d = (c * lv.diag).astype(F)
    w, keep = F(OMEGA) / d, F(1) - F(OMEGA)
    sweep = lambda x: keep * x + w * (b + wt * neighbours(x))  # noqa: E731
    x = sweep(w * b)
    r = b - (d * x - wt * neighbours(x))
    x = x + P.prolong(cycle32(hier[1:], P.restrict(r).astype(F), c, kept).astype(np.float64), lv).astype(F)
    return sweep(sweep(x))


# three sides of the coarse matrix, then levels on the 256-cell tiles with
# diagonals that are no powers of two
CASES = [((64, 64), (0, 0, 0, 0)), ((40, 96), (0, 0, 0, 0)), ((136, 144), (0, 0, 0, 0)), ((72, 104), (1, 0, 1, 1)),
         ((40, 32, 32), (0,) * 6), ((56, 64, 48), (0, 0, 1, 1, 0, 1)), ((64, 80, 96), (1, 0, 0, 1, 1, 1))]


@pytest.mark.parametrize("shape,bc", CASES)
def test_cycle_is_as_close_as_float32_legs(L, shape, bc):
    h = (1.0 / 64,) * len(shape)
    got, want, kept = [], [], {}
    hdl = L.mg_create(len(shape), tuple(reversed(shape)), h, bc)
    try:
        hier = P.build_hierarchy(shape, h, bc, None, levels=L.mg_num_levels(hdl))
        for seed in range(3):
            r = I.blob_rhs(shape, seed).astype(F)
            ref = P.Multigrid(hier, s=1.0).precondition(r.astype(np.float64)) / h[0] ** 2
            z = torch.empty(shape, device="cuda")
            L.mg_precondition(hdl, torch.from_numpy(r).cuda(), z)
            for out, v in ((got, z.cpu().numpy()), (want, cycle32(hier, r, h[0] ** 2, kept))):
                out.append(np.linalg.norm(v - ref) / np.linalg.norm(ref))
    finally:
        L.mg_destroy(hdl)
    assert max(want) <= 2e-7 and np.mean(got) <= 1.3 * np.mean(want), (got, want)
