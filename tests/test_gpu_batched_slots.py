"""GPU test of the batched solver's partial-sum slots: right-hand sides off
16-byte alignment sum their residual by tiles, the aligned ones by strips, at
the same time and each in slots of its own."""
import numpy as np
import pytest

from oracle import poisson as P
from test_gpu_batched import BC, L, make_batch  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# grids of 8, 32 and 64 columns: 128 x 8 tiles are the most there (32 x 64:
# eight, where 32 x 16 tiles are four), 32 x 16 on the wider ones
@pytest.mark.parametrize("sides", [[(32, 64)] * 4, [(32, 256), (8, 256), (64, 64), (32, 64)]])
@pytest.mark.parametrize("tile", [(128, 8), (32, 16)])
def test_tiles_and_strips_sum_apart(L, sides, tile):  # noqa: F811
    """Each reported residual is the oracle's of the returned solution, up to
    float32 rounding of that solution through the operator."""
    shapes, spacings, _, rhs = make_batch(sides, seed=3, with_masks=False)
    b = L.mg_create_batched(shapes, spacings, BC, None)
    try:
        L.mg_batched_config(b, tile[0], tile[1], 2)
        bt, xt = [], []
        for k, r in enumerate(rhs):
            buf = torch.zeros(r.size + 1, device="cuda")
            t = buf[k % 2:][:r.size].view(r.shape)
            t.copy_(torch.from_numpy(r))
            bt.append(t)
            xt.append(torch.zeros(r.shape, device="cuda"))
        status, stats = L.mg_solve_batched(b, bt, xt, 1e-6)
    finally:
        L.mg_destroy_batched(b)
    assert status == L.MG_OK, [s["status_name"] for s in stats]
    for (nx, ny), h, r, x, st in zip(shapes, spacings, rhs, xt, stats):
        lv = P.Level((ny, nx), h, BC, None)
        b64, x64 = r.astype(np.float64), x.cpu().numpy().astype(np.float64)
        ref = P.solve_reference((ny, nx), h, BC, b64, None, tol=1e-12, s=1.0)
        assert st["relres0"] == pytest.approx(1.0, abs=1e-6) and 0 < st["relres"] <= 1e-6
        assert np.linalg.norm(x64 - ref) <= 1e-5 * np.linalg.norm(ref)
