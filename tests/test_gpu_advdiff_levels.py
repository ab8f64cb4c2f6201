"""GPU parity of the advection-diffusion level kernels at their edges: one
cycle from a random guess against the FP64 oracle's correction (2e-5 of its
norm, the bound of the other one-cycle tests: some thirty float32 steps on a
float-float residual), on levels of the 32 x 8 tiles with remainders, on both
sides of the largest such level, with a coarse matrix whose rows are no
multiple of four, rows that are not whole float4, and outputs off 16-byte
alignment; and the device-side loop against the host-driven one."""
import numpy as np
import pytest

from oracle import advdiff as A
from paper_2402_17913_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P = dict(h=1.0, dt=50.0, nu=2.0, u=1.0, v=-0.5)


@pytest.fixture(scope="module")
def L():
    from paper_2402_17913_gb300 import build, lib
    build.build()
    lib.load()
    return lib


def make(L, shape, cycle="V", pre=2, post=2, omega=2 / 3, s=1.0, max_cycles=1000):
    opt = L.ad_default_options(cycle=L.MG_CYCLE_SAWTOOTH if cycle == "sawtooth" else L.MG_CYCLE_V, pre=pre,
                               post=post, omega=omega, coarse_scale=s, max_cycles=max_cycles)
    hd = L.ad_create((shape[1], shape[0]), P["h"], P["dt"], P["nu"], P["u"], P["v"], L.AD_UPWIND, opt)
    hier = A.build_hierarchy(shape, P["h"], P["dt"], P["nu"], P["u"], P["v"], "upwind", "rediscretise",
                             levels=L.ad_num_levels(hd))
    return hd, A.ADMultigrid(hier, cycle, pre if cycle == "V" else 0, post, omega, s)


@pytest.mark.parametrize("shape,cycle,pre,post", [
    ((48, 208), "V", 2, 2),         # remainders in x on three levels
    ((18, 22), "V", 2, 2),          # rows of 22 nodes; 99 rows in the matrix
    ((16, 8), "V", 2, 2),           # one tile; 4 x 8 coarsest
    ((448, 640), "V", 2, 2),        # level 0 (286,720 nodes) just on the small tiles
    ((448, 704), "V", 2, 2),        # and just above them
    ((96, 160), "V", 1, 2),         # other sweep counts: the 64 x 16 tiles
    ((36, 52), "sawtooth", 0, 1),   # coarse matrix of the sawtooth
])
def test_one_cycle(L, shape, cycle, pre, post):
    omega, s = (1.0, 0.5) if cycle == "sawtooth" else (2 / 3, 1.0)
    hd, mg = make(L, shape, cycle, pre, post, omega, s, max_cycles=1)
    try:
        rng = np.random.default_rng(3)
        b = I.advdiff_gaussian(shape, gamma=shape[1] / 12.0).astype(np.float32)
        x0 = (0.3 * rng.standard_normal(shape)).astype(np.float32)
        z = mg.precondition(A.residual(mg.hier[0], b.astype(np.float64), x0.astype(np.float64)))
        for off in (0, 1):  # the output 4 bytes off 16-byte alignment
            buf = torch.zeros(b.size + 4, device="cuda")
            x = buf[off:off + b.size].view(shape)
            status, st = L.ad_solve(hd, torch.from_numpy(b).cuda(), x, rel_tol=0.0, l1_tol=0.0,
                                    x0=torch.from_numpy(x0).cuda())
            assert status == L.MG_NOT_CONVERGED and st["cycles"] == 1, st
            got = x.cpu().numpy().astype(np.float64) - x0
            assert np.linalg.norm(got - z) <= 2e-5 * np.linalg.norm(z)
    finally:
        L.ad_destroy(hd)


@pytest.mark.parametrize("max_cycles", [1000, 3])
def test_device_loop_equals_host_loop(L, monkeypatch, max_cycles):
    b = torch.from_numpy(I.advdiff_gaussian((96, 160)).astype(np.float32)).cuda()
    out = []
    for host in (False, True):
        if host:
            monkeypatch.setenv("NPMG_NO_DEVICE_LOOP", "1")
        hd, _ = make(L, (96, 160), max_cycles=max_cycles)
        try:
            x = torch.zeros_like(b)
            for _ in range(2):
                status, st = L.ad_solve(hd, b, x)
            out.append((status, st["cycles"], st["relres"], x))
        finally:
            L.ad_destroy(hd)
    assert out[0][:3] == out[1][:3] and torch.equal(out[0][3], out[1][3]), (out[0][:3], out[1][:3])
