"""GPU parity of the level kernels and of the coarse cycle of small grids
against the FP64 oracle: the 256-cell tiles of small levels at their
edges (one tile, whole tiles, remainders along each axis, a finest level, all
storage types), and the coarse cycle as a dense matrix.  One cycle is compared to 2e-5 of its norm: each of its
some thirty float32 steps rounds to 2^-24 of the field's scale and the
smoothers do not amplify (eight levels of a V(2,2) cycle: below 1e-5)."""
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


def setup(L, shape, bc, frac, levels=0, **opt):
    rng = np.random.default_rng(17)
    solid = I.flood_fill_unreachable(rng.random(shape) < frac, bc) if frac > 0 else None
    h = tuple(1.0 / (s + 1) for s in reversed(shape))
    st = None if solid is None else torch.from_numpy(solid.astype(np.uint8)).cuda()
    hdl = L.mg_create(len(shape), tuple(reversed(shape)), h, bc, st, L.default_options(levels=levels, **opt))
    return hdl, solid, h


def check_cycle(L, shape, bc, frac, levels=0, cycle="V", **opt):
    kw = dict(cycle=L.MG_CYCLE_SAWTOOTH, coarse_scale=0.5) if cycle == "sawtooth" else {}
    hdl, solid, h = setup(L, shape, bc, frac, levels, **kw, **opt)
    try:
        hier = P.build_hierarchy(shape, h, bc, solid, levels=L.mg_num_levels(hdl))
        mg = (P.Multigrid(hier, post=2, s=0.5, cycle="sawtooth") if cycle == "sawtooth"
              else P.Multigrid(hier, pre=opt.get("pre", 2), post=opt.get("post", 2), s=1.0))
        r = I.blob_rhs(shape, 3, solid=solid).astype(np.float32)
        z = torch.full(shape, float("nan"), device="cuda")
        L.mg_precondition(hdl, torch.from_numpy(r).cuda(), z)
        ref = mg.precondition(r.astype(np.float64)) / h[0] ** 2
        err = np.linalg.norm(z.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= 2e-5, err
    finally:
        L.mg_destroy(hdl)


SMALL3D = [
    # (z, y, x), faces x- x+ y- y+ z- z+ (0 = Dirichlet), solid fraction
    ((16, 32, 32), (0,) * 6, 0.0),              # whole tiles
    ((20, 24, 40), (1, 0, 1, 1, 0, 1), 0.06),   # a remainder in x (40 = 2.5 tiles)
    ((20, 28, 44), (0, 1, 0, 0, 1, 0), 0.0),    # level 1 (10, 14, 22): remainders along every axis
    ((56, 40, 88), (1, 0, 1, 1, 1, 1), 0.05),   # close to the largest level (197,120 cells)
]


SMALL2D = [
    ((64, 64), (0, 0, 0, 0), 0.0),            # whole tiles
    ((72, 104), (1, 0, 1, 1), 0.06),          # a remainder in x (3.25 tiles), level 1 (36, 52) in both
    ((400, 480), (0, 0, 1, 0), 0.05),         # close to the largest level (192,000 cells)
    ((512, 416), (0, 1, 0, 0), 0.0),          # just above it: the TMA-fed tiles, then the small ones
]


@pytest.mark.parametrize("shape,bc,frac", SMALL2D)
def test_small_2d_tiles_match_oracle(L, shape, bc, frac):
    check_cycle(L, shape, bc, frac)
    check_cycle(L, shape, bc, frac, cycle="sawtooth")


@pytest.mark.parametrize("shape,bc,frac", SMALL3D)
def test_small_3d_tiles_match_oracle(L, shape, bc, frac):
    check_cycle(L, shape, bc, frac)
    check_cycle(L, shape, bc, frac, cycle="sawtooth")


@pytest.mark.parametrize("shape,bc,prec", [((20, 24, 40), (1, 0, 1, 1, 0, 1), 0), ((20, 24, 40), (1, 0, 1, 1, 0, 1), 1),
                                           ((20, 24, 40), (1, 0, 1, 1, 0, 1), 2), ((72, 104), (1, 0, 1, 1), 0),
                                           ((72, 104), (1, 0, 1, 1), 1)])
def test_small_tiles_solve_in_every_storage(L, shape, bc, prec):
    """The finest level on the tiles (its up leg reduces (r, z)), in every
    level storage: relres 1e-6 and the oracle's solution."""
    hdl, solid, h = setup(L, shape, bc, 0.06, prec=prec)
    try:
        b = I.blob_rhs(shape, 0, solid=solid).astype(np.float32)
        x = torch.zeros(shape, device="cuda")
        status, st = L.mg_solve(hdl, torch.from_numpy(b).cuda(), x, 1e-6)
    finally:
        L.mg_destroy(hdl)
    assert status == L.MG_OK, st
    xs = P.solve_reference(shape, h, bc, b.astype(np.float64), solid, tol=1e-12, s=1.0)
    assert np.linalg.norm(x.cpu().numpy() - xs) / np.linalg.norm(xs) <= 1e-5


DENSE = [
    # shape, faces, solid fraction, levels (0: until a side is odd or 4)
    ((64, 128), (0, 0, 0, 0), 0.0, 0),               # level 1 has 2048 cells, the most the matrix takes
    ((60, 100), (1, 0, 1, 1), 0.05, 0),              # 1500 rows, coarsest 15 x 25
    ((46, 46), (0, 0, 0, 0), 0.0, 2),                # 529 rows (no multiple of four), the matrix is the inverse
    ((52, 92), (1, 0, 0, 1), 0.08, 0),               # 1196 rows over 299
    ((24, 36, 20), (1, 0, 1, 1, 1, 1), 0.05, 0),     # 3D: 2160 cells on the tiles, 270 rows
    ((18, 18, 24), (0,) * 6, 0.0, 2),                # 3D: 972 rows, the inverse
    ((32, 96), (0, 0, 0, 1), 0.0, 5),                # the smallest matrices: 192, coarsest 2 x 6
]


@pytest.mark.parametrize("shape,bc,frac,levels", DENSE)
def test_dense_coarse_cycle_matches_oracle(L, shape, bc, frac, levels):
    check_cycle(L, shape, bc, frac, levels)
    check_cycle(L, shape, bc, frac, levels, cycle="sawtooth")
    check_cycle(L, shape, bc, frac, levels, pre=1, post=3)  # not symmetric
