"""GPU test of the tuner's cache: a stored choice is taken up again by the
same batch alone, not by one of equal totals and other faces, sides or solids,
nor from a line without the kernels' generation."""
import numpy as np
import pytest

from test_gpu_batched import L, make_batch  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def iterations(L, sides, bc, with_masks, tune=False):  # noqa: F811
    """CG iterations with the choice that the batch's creation took."""
    shapes, spacings, solids, rhs = make_batch(sides, seed=3, with_masks=with_masks)
    masks = [None if s is None else torch.from_numpy(s.astype(np.uint8)).cuda() for s in solids]
    b = L.mg_create_batched(shapes, spacings, bc, masks)
    try:
        bt = [torch.from_numpy(r).cuda() for r in rhs]
        xt = [torch.zeros_like(t) for t in bt]
        if tune:
            L.mg_tune_batched(b, bt, xt, 1e-6)
            return None
        status, st = L.mg_solve_batched(b, bt, xt, 1e-6)
        assert status == L.MG_OK
        return [s["iters"] for s in st]
    finally:
        L.mg_destroy_batched(b)


def test_choice_belongs_to_its_batch(L, tmp_path, monkeypatch):  # noqa: F811
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("NPMG_TUNE_CACHE", str(cache))
    D = (0, 0, 0, 0)
    base = ([(64, 128), (128, 64)], D, False)
    others = [([(64, 128), (128, 64)], (0, 1, 0, 0), False), ([(64, 128), (128, 64)], D, True),
              ([(128, 64), (64, 128)], (0, 0, 1, 0), False), ([(128, 96), (32, 128)], D, False)]
    plain = [iterations(L, *c) for c in [base] + others]
    iterations(L, *base, tune=True)
    key = cache.read_text().split()[0]
    cache.write_text("%s 0 1 1.0\n" % key)  # one sweep: more iterations
    assert sum(iterations(L, *base)) > sum(plain[0])
    assert [iterations(L, *c) for c in others] == plain[1:]
    cache.write_text("%s 0 1 1.0\n" % key[:key.index("|g")])
    assert iterations(L, *base) == plain[0]
