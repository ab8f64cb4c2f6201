"""GPU parity of the convolution and the weight gradient where a block takes
several z-runs one after another (more columns than resident blocks) and
where a run is cut inside the grid, with ragged tiles in x and y.  Inputs and
weights are exact in BF16, so outputs differ from the float64 oracle by
float32 accumulation only: within n 2^-24 of the sum of absolute terms, n
terms summed."""
import numpy as np
import pytest

from oracle import convnet as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def L():
    from paper_2402_17913_gb300 import build, lib
    build.build()
    lib.load()
    return lib


def draw(shape, scale=1.0, seed=0):
    a = np.random.default_rng(seed).standard_normal(shape).astype(np.float32) * scale
    return torch.from_numpy(a).bfloat16()


# (n, x, y, z): 800 columns of 8 x 16 voxels (several items per block), and a
# long column cut into runs of a few planes
@pytest.mark.parametrize("n,nx,ny,nz", [(1, 315, 310, 3), (2, 9, 17, 70)])
def test_conv_over_several_runs(L, n, nx, ny, nz):
    x, w = draw((n, nz, ny, nx, 16), seed=1), draw((27, 16, 16), 0.2, seed=2)
    y = torch.empty((n, nz, ny, nx, 16), dtype=torch.float32, device="cuda")
    L.gn_conv3d(x.cuda(), w.float().cuda(), y, (nx, ny, nz), n=n, mode=L.GN_CONV_F32)
    got, xd, wd = y.cpu().double().numpy(), x.double().numpy(), w.double().numpy()
    for s in range(n):
        xs = np.moveaxis(xd[s], -1, 0)
        ref = np.moveaxis(C.conv3d(xs, wd), 0, -1)
        bound = 432 * U32 * np.moveaxis(C.conv3d(np.abs(xs), np.abs(wd)), 0, -1) + 1e-30
        assert np.all(np.abs(got[s] - ref) <= bound), (s, np.max(np.abs(got[s] - ref) / bound))


def test_wgrad_over_many_tiles(L):
    """More tiles than blocks, ragged along every axis (19 = 4 tiles of 4 and 3)."""
    n, nx, ny, nz = 2, 150, 60, 19
    x, g = draw((n, nz, ny, nx, 16), seed=3), draw((n, nz, ny, nx, 16), seed=4)
    dw = torch.empty((27, 16, 16), dtype=torch.float32, device="cuda")
    L.gn_conv3d_wgrad(x.cuda(), g.cuda(), dw, (nx, ny, nz), n=n)
    xd, gd = (np.moveaxis(t.double().numpy(), -1, 1) for t in (x, g))
    ref = sum(C.conv3d_wgrad(xd[s], gd[s]) for s in range(n))
    bound = n * nx * ny * nz * U32 * sum(C.conv3d_wgrad(np.abs(xd[s]), np.abs(gd[s])) for s in range(n))
    got = dw.cpu().double().numpy()
    assert np.all(np.abs(got - ref) <= bound)
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
