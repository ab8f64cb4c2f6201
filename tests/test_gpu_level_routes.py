"""GPU parity of the level kernels that the tiles of small levels stand in
front of, on grids small enough for the FP64 oracle: the TMA-fed and the
plain 2D tiles, the z-streaming 3D kernels and the 3D tiles, masked and not,
in every level storage.  Bounds as in the other one-cycle and solve tests
(2e-5 of a float32 cycle's norm; relres 1e-6 and 1e-5 of the solution)."""
import numpy as np
import pytest

from oracle import poisson as P
from paper_2402_17913_gb300 import inputs as I
from test_gpu_small_levels import L, check_cycle, setup  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROUTES = {
    "tma2d": dict(NPMG_SMALL2D_MAX="0"),
    "tiles2d": dict(NPMG_SMALL2D_MAX="0", NPMG_NO_TMA="1"),
    "stream3d": dict(NPMG_SMALL3D_MAX="0", NPMG_NO_TMA3D="1", NPMG_NO_ROWS3D="1"),
    "tiles3d": dict(NPMG_SMALL3D_MAX="0", NPMG_NO_TMA3D="1", NPMG_NO_ROWS3D="1", NPMG_NO_STREAM3D="1"),
}
# two levels or more above the coarse matrix; widths of whole 16-cell chunks
# (TMA) and others, ragged tiles and runs
GRIDS = {
    "2d": [((96, 192), (0, 0, 0, 0), 0.0), ((80, 160), (1, 0, 1, 1), 0.08), ((88, 120), (0, 1, 0, 0), 0.06)],
    "3d": [((32, 32, 32), (0,) * 6, 0.0), ((40, 24, 56), (1, 0, 1, 1, 0, 1), 0.06),
           ((40, 40, 136), (0, 1, 0, 0, 1, 0), 0.05)],
}
CASES = [(r, g) for r in ROUTES for g in GRIDS[r[-2:]]]


@pytest.mark.parametrize("route,grid", CASES)
def test_cycle_matches_oracle(L, monkeypatch, route, grid):  # noqa: F811
    for k, v in ROUTES[route].items():
        monkeypatch.setenv(k, v)
    check_cycle(L, *grid)
    check_cycle(L, *grid, cycle="sawtooth")


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("route,grid", CASES)
def test_solve_in_every_storage(L, monkeypatch, route, grid, prec):  # noqa: F811
    for k, v in ROUTES[route].items():
        monkeypatch.setenv(k, v)
    shape, bc, frac = grid
    hdl, solid, h = setup(L, shape, bc, frac, prec=prec)
    try:
        b = I.blob_rhs(shape, 0, solid=solid).astype(np.float32)
        x = torch.zeros(shape, device="cuda")
        status, st = L.mg_solve(hdl, torch.from_numpy(b).cuda(), x, 1e-6)
    finally:
        L.mg_destroy(hdl)
    assert status == L.MG_OK and st["relres"] <= 1e-6, st
    xs = P.solve_reference(shape, h, bc, b.astype(np.float64), solid, tol=1e-12, s=1.0)
    assert np.linalg.norm(x.cpu().numpy() - xs) / np.linalg.norm(xs) <= 1e-5
