"""GPU tests of the batched solver's work lists: a tile choice left and taken
up again between solves (the lists a captured launch reads are rebuilt)."""
import numpy as np
import pytest

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
