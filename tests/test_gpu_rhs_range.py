"""GPU tests of right-hand sides over float32's range.  ||b||^2 and the first
residual are sums in the caller's units: b times a power of two takes the
same iterations to the same solution times that power (every operation of a
solve scales exactly), and a right-hand side whose norm is not a finite
number ends as MG_DIVERGED instead of being returned unsolved."""
import numpy as np
import pytest

from paper_2402_17913_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2402_17913_gb300 import build, lib
    build.build()
    lib.load()
    return lib


def unit_rhs(shape):
    b = I.blob_rhs(shape, 0)
    return torch.from_numpy((b / np.abs(b).max()).astype(np.float32)).cuda()


def poisson(L, b, tol=1e-6, x0=None, **opt):
    shape = tuple(b.shape)
    hdl = L.mg_create(len(shape), tuple(reversed(shape)), (1.0,) * len(shape), (0,) * (2 * len(shape)), None,
                      L.default_options(**opt))
    try:
        x = torch.zeros_like(b) if x0 is None else x0.clone()
        status, st = L.mg_solve(hdl, b, x, tol)
    finally:
        L.mg_destroy(hdl)
    return status, st, x


def advdiff(L, b, cycle):
    opt = (L.ad_default_options(cycle=L.MG_CYCLE_SAWTOOTH, coarse_scale=0.5) if cycle == "sawtooth"
           else L.ad_default_options())
    hd = L.ad_create(tuple(reversed(b.shape)), 1.0, 0.5, 1.0, 0.5, -0.25, L.AD_UPWIND, opt)
    try:
        x = torch.zeros_like(b)
        status, st = L.ad_solve(hd, b, x, 1e-6)
    finally:
        L.ad_destroy(hd)
    return status, st, x


# 2^60: the squares of a thread's few cells stay below float32's largest
# number, those of the grid do not; 2^-40: far inside the range
@pytest.mark.parametrize("power", [60, -40])
@pytest.mark.parametrize("shape", [(256, 256), (320, 448), (64, 64, 96)])
@pytest.mark.parametrize("refine", [0, 1])
def test_scaled_rhs_gives_the_scaled_solution(L, shape, refine, power):
    b = unit_rhs(shape)
    opt = dict(refine=(L.MG_REFINE_FP64, L.MG_REFINE_FF)[refine])
    s0, st0, x0 = poisson(L, b, **opt)
    s1, st1, x1 = poisson(L, b * 2.0 ** power, **opt)
    assert s0 == L.MG_OK and s1 == L.MG_OK and st1["iters"] == st0["iters"] and st1["outer"] == st0["outer"]
    assert st1["relres"] <= 1e-6 and st1["relres0"] == pytest.approx(1.0, abs=1e-5)
    # the same roundings; 1e-6 leaves room for low words that underflow
    assert torch.linalg.norm(x1 * 2.0 ** -power - x0) <= 1e-6 * torch.linalg.norm(x0)


@pytest.mark.parametrize("power", [60, -40])
@pytest.mark.parametrize("cycle", ["V", "sawtooth"])
def test_scaled_advection_diffusion_step(L, cycle, power):
    b = torch.from_numpy(np.random.default_rng(3).uniform(-1.0, 1.0, (320, 384)).astype(np.float32)).cuda()
    s0, st0, x0 = advdiff(L, b, cycle)
    s1, st1, x1 = advdiff(L, b * 2.0 ** power, cycle)
    assert s0 == L.MG_OK and s1 == L.MG_OK and st1["cycles"] == st0["cycles"] and 0 < st1["relres"] <= 1e-6
    assert torch.linalg.norm(x1 * 2.0 ** -power - x0) <= 1e-6 * torch.linalg.norm(x0)


BAD = [float("inf"), float("-inf"), float("nan"), 1e30]  # 1e30: its square is not a float32 number


@pytest.mark.parametrize("bad", BAD)
def test_norm_not_finite_is_reported(L, bad):
    for shape in ((256, 256), (320, 448), (32, 32, 48)):
        b = unit_rhs(shape)
        b.view(-1)[b.numel() // 3] = bad
        for refine in (L.MG_REFINE_FP64, L.MG_REFINE_FF):
            status, st, _ = poisson(L, b, refine=refine)
            assert status == L.MG_DIVERGED and not st["relres"] <= 1e-6, (shape, st)
    b = torch.ones((96, 160), device="cuda")
    b[7, 9] = bad
    for cycle in ("V", "sawtooth"):
        status, st, _ = advdiff(L, b, cycle)
        assert status == L.MG_DIVERGED and not st["relres"] <= 1e-6, st


@pytest.mark.parametrize("bad", BAD)
def test_norm_not_finite_in_a_batch(L, bad):
    """The instance that holds it diverges, the other one is solved."""
    shapes = [(64, 64), (96, 64)]
    rhs = [unit_rhs((ny, nx)) for nx, ny in shapes]
    rhs[0][5, 6] = bad
    b = L.mg_create_batched(shapes, [(1.0, 1.0)] * 2, (0, 0, 0, 0))
    try:
        x = [torch.zeros_like(t) for t in rhs]
        _, st = L.mg_solve_batched(b, rhs, x, 1e-6)
    finally:
        L.mg_destroy_batched(b)
    assert st[0]["status"] == L.MG_DIVERGED and st[1]["status"] == L.MG_OK and st[1]["relres"] <= 1e-6, st
