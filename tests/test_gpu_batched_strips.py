"""GPU tests of the batched solver's work lists: strips at the edges of their
range (one warp's width of 128 cells, one group more, halos on one and both
sides, runs of rows with remainders) against the FP64 oracle, and a tile
choice left and taken up again between solves (the lists a captured launch
reads are rebuilt)."""
import numpy as np
import pytest

from oracle import poisson as P
from paper_2402_17913_gb300 import inputs as I
from test_gpu_batched import L, make_batch  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BC = (0, 0, 0, 0)


def test_a_choice_taken_up_again_gives_the_same_bits(L):  # noqa: F811
    shapes, spacings, solids, rhs = make_batch([(64, 64), (128, 64), (96, 96)], seed=5)
    masks = [None if s is None else torch.from_numpy(s.astype(np.uint8)).cuda() for s in solids]
    b = L.mg_create_batched(shapes, spacings, BC, masks)
    try:
        bt = [torch.from_numpy(r).cuda() for r in rhs]
        out = []
        for tile in ((64, 16), (32, 16), (64, 16)):
            L.mg_batched_config(b, tile[0], tile[1], 2)
            xt = [torch.zeros_like(t) for t in bt]
            status, _ = L.mg_solve_batched(b, bt, xt, 1e-6)
            assert status == L.MG_OK
            out.append(xt)
        for p, q in zip(out[0], out[2]):
            assert torch.equal(p, q)
    finally:
        L.mg_destroy_batched(b)


# a warp's whole width, one group more (two strips), three strips, five; 132, 500
# and 40 halve to a width off the strips; heights that no long run divides
SIDES = [(128, 32), (132, 28), (248, 16), (256, 16), (500, 8), (64, 60), (40, 28)]


def test_more_partials_than_a_warp_sums(L):  # noqa: F811
    """An instance of more than 128 strips (its sums have phases of their own)
    beside small ones; relative residual as asked for."""
    shapes, spacings, solids, rhs = make_batch([(512, 512), (64, 64), (160, 96)], seed=9)
    masks = [None if s is None else torch.from_numpy(s.astype(np.uint8)).cuda() for s in solids]
    b = L.mg_create_batched(shapes, spacings, BC, masks)
    try:
        bt = [torch.from_numpy(r).cuda() for r in rhs]
        xt = [torch.zeros_like(t) for t in bt]
        status, stats = L.mg_solve_batched(b, bt, xt, 1e-6)
    finally:
        L.mg_destroy_batched(b)
    assert status == L.MG_OK and all(s["relres"] <= 1e-6 for s in stats)
    for (nx, ny), h, solid, r, x in zip(shapes, spacings, solids, rhs, xt):
        lv = P.Level((ny, nx), h, BC, solid)
        b64, x64 = r.astype(np.float64) * lv.fluid, x.cpu().numpy().astype(np.float64)
        # float32 rounding of x passes through the operator: 6e-8 ||A|| ||x|| / ||b||
        bound = 1e-6 + 6e-8 * 8 * (max(nx, ny) + 1) ** 2 * np.linalg.norm(x64) / np.linalg.norm(b64)
        assert np.linalg.norm(b64 - P.apply_A(lv, x64)) / np.linalg.norm(b64) <= bound


@pytest.mark.parametrize("sweeps", [1, 2, 3])
@pytest.mark.parametrize("bc,with_masks", [((0, 0, 0, 0), True), ((1, 0, 1, 1), False), ((0, 1, 1, 0), True)])
def test_strips_match_oracle(L, sweeps, bc, with_masks):  # noqa: F811
    """Solved to a relative residual of 1e-8.  ||b|| / (lambda_min ||x||) is
    at most about 50 for these problems (25 to 35 for the ducts closed on
    three sides), so the error stays below 5e-7, and float32 rounding adds
    6e-8: 1e-6 of the solution's norm."""
    rng = np.random.default_rng(17)
    shapes = SIDES
    spacings = [(1.0 / (nx + 1), 1.0 / (nx + 1)) for nx, _ in shapes]
    solids = [I.random_solid_mask((ny, nx), rng, 0.08, bc) if with_masks and k % 2 == 0 else None
              for k, (nx, ny) in enumerate(shapes)]
    rhs = [I.blob_rhs((ny, nx), 100 + k, solid=solids[k]).astype(np.float32) for k, (nx, ny) in enumerate(shapes)]
    masks = [None if s is None else torch.from_numpy(s.astype(np.uint8)).cuda() for s in solids]
    b = L.mg_create_batched(shapes, spacings, bc, masks)
    try:
        L.mg_batched_config(b, 64, 32, sweeps)
        bt = [torch.from_numpy(r).cuda() for r in rhs]
        xt = [torch.zeros_like(t) for t in bt]
        status, stats = L.mg_solve_batched(b, bt, xt, 1e-8)
    finally:
        L.mg_destroy_batched(b)
    assert status == L.MG_OK, [s["status_name"] for s in stats]
    for (nx, ny), h, solid, r, x in zip(shapes, spacings, solids, rhs, xt):
        ref = P.solve_reference((ny, nx), h, bc, r.astype(np.float64), solid, tol=1e-12, s=1.0)
        assert np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref) <= 1e-6
