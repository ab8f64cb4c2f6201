"""The calls whose speed is measured: what users of this framework have it do.

Twelve listed cases and a generator of further ones over the same ranges, all
through the public binding (``paper_2402_17913_gb300.lib``):

* ``cycle``    one preconditioner cycle, for programs with a Krylov loop of
               their own (``mg_precondition``);
* ``poisson``  one pressure-Poisson solve to a relative residual of 1e-6
               (``mg_solve``), in each level storage (float32, FP16, BF16);
* ``flow``     one projection step of the flow past a block (``ns_step``),
               with the 5/7-point or the finite-element momentum filters;
* ``batched``  one solve of a batch of uneven 2D problems with solids
               (``mg_solve_batched``);
* ``advdiff``  one implicit advection-diffusion step (``ad_solve``);
* ``guess``    the learned initial guess: the network's inference on a whole
               grid (``gn_forward``) and one training step's loss and
               gradient on a minibatch (``gn_gradients``).

Sizes are those of the benchmark's configurations and tests, and odd ones of
the same range.  Grids whose sides are not powers of two have cells of equal
sides, as flow domains do.
"""
import itertools
import math

import numpy as np
import torch

from paper_2402_17913_gb300 import lib

TOL = 1e-6
PREC = {"fp32": lib.MG_FP32, "fp16": lib.MG_MIXED_FP16, "bf16": lib.MG_MIXED_BF16}
F64 = torch.float64


# ---------------------------------------------------------------------------
# the cases
def listed():
    return [
        # the smallest call: one cycle inside somebody else's iteration on a
        # small 2D grid, where the launch and the chain of levels are all
        {"name": "cycle2d_64", "kind": "cycle", "nx": 64, "ny": 64, "nz": 1, "faces": "DDDD", "solids": False},
        # the same on a ragged 3D grid with solid bodies and open, closed faces
        {"name": "cycle3d_96x80x64_solids", "kind": "cycle", "nx": 96, "ny": 80, "nz": 64, "faces": "NDNNNN",
         "solids": True},
        # the paper's 2D pressure problem at the size of its examples
        {"name": "poisson2d_256", "kind": "poisson", "nx": 256, "ny": 256, "nz": 1, "faces": "DDDD", "prec": "fp32"},
        # a large ragged 2D duct with closed walls
        {"name": "poisson2d_1600x960", "kind": "poisson", "nx": 1600, "ny": 960, "nz": 1, "faces": "NDNN",
         "prec": "fp32"},
        # a mid-size ragged 3D duct, levels stored in FP16
        {"name": "poisson3d_160x96x80_fp16", "kind": "poisson", "nx": 160, "ny": 96, "nz": 80, "faces": "NDNNNN",
         "prec": "fp16"},
        # the headline solve: larger than the caches, bound by memory
        {"name": "poisson3d_256", "kind": "poisson", "nx": 256, "ny": 256, "nz": 256, "faces": "DDDDDD",
         "prec": "fp32"},
        # one time step of the 2D flow past a square block
        {"name": "flow2d_2048x1024", "kind": "flow", "nx": 2048, "ny": 1024, "nz": 1, "block": 64, "fe": False},
        # one time step of the 3D flow past a cube with the finite-element filters
        {"name": "flow3d_256x128x128_fe", "kind": "flow", "nx": 256, "ny": 128, "nz": 128, "block": 32, "fe": True},
        # a batch of uneven problems with solids, as a quarter of the benchmark's batch
        {"name": "batched_256", "kind": "batched", "count": 256, "sides": "64,128,256,512"},
        # one implicit step of the advection-diffusion equation at C = 50
        {"name": "advdiff_1024", "kind": "advdiff", "nx": 1024, "ny": 1024, "u": 1.0, "v": 1.0},
        # the learned guess of a whole 3D step
        {"name": "guess_forward_256x128x128", "kind": "guess", "mode": "forward", "n": 1, "nx": 256, "ny": 128,
         "nz": 128},
        # its training: a minibatch of 64^3 crops, forward and backward
        {"name": "guess_train_8x64", "kind": "guess", "mode": "train", "n": 8, "nx": 64, "ny": 64, "nz": 64},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sides(rng, cells, dim, stretch, most=1000):
    """Sides of about `cells` cells, the longest at most `stretch` times the
    shortest, that halve until at most `most` cells are left (at least four
    along each side)."""
    f = [_log(rng, 1.0, stretch) for _ in range(dim)]
    base = (cells / math.prod(f)) ** (1.0 / dim)
    k = 0
    while math.prod(max(4, round(base * a / 2 ** k)) for a in f) > most:
        k += 1
    return [max(4, round(base * a / 2 ** k)) << k for a in f]


def draw(rng):
    kind = rng.choice(["cycle", "poisson", "poisson", "poisson", "flow", "batched", "advdiff", "guess"])
    if kind in ("cycle", "poisson"):
        dim = rng.choice([2, 3])
        top = (2e6, 6e5) if kind == "cycle" else (2.1e6, 1.2e7)
        n = _sides(rng, _log(rng, 64 * 64 if dim == 2 else 32 ** 3, top[dim - 2]), dim, 2.0)
        c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2] if dim == 3 else 1,
             "faces": rng.choice(["DDDDDD", "NDNNNN", "DDNNDN"])[:2 * dim]}
        if kind == "cycle":
            c["solids"] = rng.random() < 0.5
        else:
            # the 16-bit level storage is for 3D solves bound by memory
            c["prec"] = rng.choice(["fp32", "fp32", "fp16", "bf16"]) if dim == 3 else "fp32"
        return c
    if kind == "flow":
        dim = rng.choice([2, 3])
        n = _sides(rng, _log(rng, 1e5, 2e6 if dim == 2 else 4e6), dim, 1.5)
        nx, rest = max(n), sorted(n)[:-1]
        return {"kind": kind, "nx": nx, "ny": rest[0], "nz": rest[1] if dim == 3 else 1,
                "block": 2 * max(2, round(rest[0] / rng.uniform(10, 24))), "fe": rng.random() < 0.5}
    if kind == "batched":
        sides = rng.choice(["64,128,256,512", "64,96,128,192", "96,100,160,320", "256,384,512"])
        most = 256 * 87040 / max(int(s) ** 2 for s in sides.split(","))
        return {"kind": kind, "count": max(4, round(_log(rng, 4, min(256, most)))), "sides": sides}
    if kind == "advdiff":
        n = _sides(rng, _log(rng, 128 * 128, 1024 * 1024), 2, 2.0, 250)
        return {"kind": kind, "nx": n[0], "ny": n[1], "u": rng.choice([1.0, 0.5, -1.0]), "v": rng.choice([1.0, -0.5])}
    if rng.random() < 0.5:
        n = [4 * round(_log(rng, 8, hi)) for hi in (60, 31, 31)]
        return {"kind": kind, "mode": "forward", "n": 1, "nx": n[0], "ny": n[1], "nz": n[2]}
    n = [4 * round(_log(rng, 6, 15)) for _ in range(3)]
    return {"kind": kind, "mode": "train", "n": rng.randint(1, 8), "nx": n[0], "ny": n[1], "nz": n[2]}


# ---------------------------------------------------------------------------
# inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _shape(c):
    return (c["nz"], c["ny"], c["nx"]) if c["nz"] > 1 else (c["ny"], c["nx"])


def _spacing(c):
    """Cells of equal sides, 1 / (n + 1) along the longest side."""
    return [1.0 / (max(_shape(c)) + 1)] * len(_shape(c))


def _blobs(shape, gen, solid=None):
    """Eight Gaussian blobs of random amplitude, width and centre, with zero
    mean over the cells that are not solid (float32)."""
    dim, k = len(shape), 8
    r = torch.rand(k, 2 + dim, generator=gen, device="cuda", dtype=F64)
    amp, width = 2 * r[:, 0] - 1, 0.02 + 0.08 * r[:, 1]
    prof = []
    for a, n in enumerate(shape):
        x = (torch.arange(n, device="cuda", dtype=F64) + 1) / (n + 1)
        prof.append(torch.exp(-((x[None] - (0.1 + 0.8 * r[:, 2 + a, None])) ** 2) / (2 * width[:, None] ** 2)))
    f = (torch.einsum("k,ky,kx->yx", amp, *prof) if dim == 2 else
         torch.einsum("kzy,kx->zyx", torch.einsum("k,kz,ky->kzy", amp, prof[0], prof[1]), prof[2]))
    fluid = torch.ones_like(f) if solid is None else (solid == 0).to(F64)
    f = f * fluid
    return (f - fluid * (f.sum() / fluid.sum())).float().contiguous()


def _solids(shape, gen, frac):
    """Solid boxes covering about `frac` of the grid (uint8): one random box
    inside every tile of a lattice, none touching another, so that the
    fluid stays in one piece."""
    solid = torch.ones(shape, dtype=torch.bool, device="cuda")
    tiles = [max(1, n // 16) for n in shape]
    share = (4 * frac) ** (1.0 / len(shape))  # a box has about a quarter of its largest size
    for a, (n, t) in enumerate(zip(shape, tiles)):
        size = n // t
        g = torch.rand(2, *tiles, generator=gen, device="cuda")
        w = (1 + g[0] * (share * (size - 3) * 1.4)).floor().clamp(max=size - 2)
        lo = (1 + g[1] * (size - 1 - w)).floor()
        i = torch.arange(n, device="cuda")
        at, off = (i // size).clamp(max=t - 1), i % size
        off = torch.where(i // size >= t, torch.full_like(off, size), off)
        view = [1] * len(shape)
        view[a] = n

        def spread(v, a=a, at=at):
            v = v.index_select(a, at)
            for d, (m, s) in enumerate(zip(shape, tiles)):
                if d != a:
                    j = (torch.arange(m, device="cuda") // (m // s)).clamp(max=s - 1)
                    v = v.index_select(d, j)
            return v

        o = off.view(view)
        lo, w = spread(lo), spread(w)
        solid &= (o >= lo) & (o < lo + w)
    return solid.to(torch.uint8).contiguous()


def _block(c):
    """The solid block of a flow, a quarter of the way down the channel."""
    shape = _shape(c)
    solid = torch.ones(shape, dtype=torch.bool, device="cuda")
    for a, n in enumerate(shape):
        mid = n // 4 if a == len(shape) - 1 else n // 2
        i = torch.arange(n, device="cuda")
        view = [1] * len(shape)
        view[a] = n
        solid &= ((i >= mid - c["block"] // 2) & (i < mid + c["block"] // 2)).view(view)
    return solid.to(torch.uint8).contiguous()


def _flow_fields(c, seed):
    """Velocity on the faces and pressure in the cells: a uniform stream, a
    row of alternating vortices behind the block and 1% noise."""
    shape, gen = _shape(c), _gen(seed)
    dim, s = len(shape), 0.6 * c["block"]
    jit = torch.rand(6, dim, generator=gen, device="cuda")
    cen = [[(c["nx"] // 4 + c["block"] * (1.2 + 1.6 * k + 0.5 * j[0])),
            c["ny"] / 2 + 0.5 * c["block"] * ((-1) ** k + j[1] - 0.5)] + ([c["nz"] / 2 + c["block"] * (j[2] - 0.5)]
                                                                          if dim == 3 else [])
           for k, j in enumerate(jit.tolist())]

    def profiles(k, face):
        out = []
        for a in range(dim):
            n = shape[dim - 1 - a] + (1 if a == face else 0)
            x = torch.arange(n, device="cuda", dtype=torch.float32) + (0.0 if a == face else 0.5) - cen[k][a]
            out.append((x / s, torch.exp(-(x / s) ** 2 / (2 if a < 2 else 8))))
        return out

    fields = []
    for comp in range(dim):
        sh = list(shape)
        sh[dim - 1 - comp] += 1
        q = 0.01 * torch.randn(sh, generator=gen, device="cuda")
        if comp == 0:
            q += 1.0
        for k in range(6 if comp < 2 else 0):
            pr = profiles(k, comp)
            gx, gy = pr[0][1], pr[1][1]
            if comp == 0:
                gy = -pr[1][0] * gy
            else:
                gx = pr[0][0] * gx
            v = 0.3 * (-1) ** k * gy[:, None] * gx[None]
            q += v if dim == 2 else pr[2][1][:, None, None] * v[None]
        fields.append(q.contiguous())
    p = torch.zeros(shape, device="cuda")
    for k in range(6):
        pr = profiles(k, -1)
        v = -0.1 * pr[1][1][:, None] * pr[0][1][None]
        p += v if dim == 2 else pr[2][1][:, None, None] * v[None]
    return fields, p


def _batch_inputs(c, seed):
    # the sizes belong to the case (the benchmark's generator seed), the solids
    # and right-hand sides to the seed
    rng, gen = np.random.Generator(np.random.PCG64(1234)), _gen(seed)
    sides = [int(v) for v in rng.choice([int(s) for s in c["sides"].split(",")], size=c["count"])]
    fracs = rng.uniform(0.0, 0.1, size=c["count"])
    masks = [_solids((n, n), gen, f) for n, f in zip(sides, fracs)]
    return sides, masks, [_blobs((n, n), gen, m) for n, m in zip(sides, masks)]


def _adv_rhs(c, seed):
    """A Gaussian of a twelfth of the domain's width, a little off the centre."""
    r = torch.rand(3, generator=_gen(seed), device="cuda").tolist()
    nx, ny = c["nx"], c["ny"]
    g = 10.0 * min(nx, ny) / 128 * (0.8 + 0.4 * r[0])
    x = torch.arange(nx, device="cuda", dtype=torch.float32) - (nx - 1) / 2 - (r[1] - 0.5) * 0.2 * nx
    y = torch.arange(ny, device="cuda", dtype=torch.float32) - (ny - 1) / 2 - (r[2] - 0.5) * 0.2 * ny
    return (torch.exp(-y ** 2 / (2 * g * g))[:, None] * torch.exp(-x ** 2 / (2 * g * g))[None]).contiguous()


GN_IO = [(2, 16)] + [(16, 16)] * 7 + [(16, 1)]


def _guess_inputs(c, seed):
    """Weights of a freshly initialised network, and (b, p) fields with the
    fluid flags of a box in each sample."""
    gen, shape = _gen(seed), (c["nz"], c["ny"], c["nx"])
    w = [(torch.randn(27, ci, co, generator=gen, device="cuda") * math.sqrt(2.0 / (27 * ci))).cpu().numpy()
         for ci, co in GN_IO]
    b, p, fluid = [], [], []
    for _ in range(c["n"]):
        solid = torch.zeros(shape, device="cuda")
        solid[tuple(slice(n // 4, n // 2) for n in shape)] = 1.0
        noise = torch.randn(shape, generator=gen, device="cuda")
        b.append((_blobs(shape, gen) + 0.05 * noise) * (1 - solid))
        p.append(_blobs(shape, gen))
        fluid.append(1 - solid)
    return w, torch.stack(b).contiguous(), torch.stack(p).contiguous(), torch.stack(fluid).contiguous()


class State:
    """A handle with the arrays it works on; gives the handle back when dropped."""

    def __init__(self, case, handle, destroy, **arrays):
        self.case, self.handle, self._destroy = case, handle, destroy
        self.__dict__.update(arrays)

    def __del__(self):
        self._destroy(self.handle)


def _faces(text):
    return [lib.MG_BC_DIRICHLET if t == "D" else lib.MG_BC_NEUMANN for t in text]


def _grid_inputs(c, seed):
    """(solids or None, right-hand side) of a cycle or a Poisson solve."""
    gen, shape = _gen(seed), _shape(c)
    solid = _solids(shape, gen, 0.06) if c.get("solids") else None
    return solid, _blobs(shape, gen, solid)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("cycle", "poisson"):
        solid, b = _grid_inputs(c, seed)
        shape = _shape(c)
        opt = lib.default_options(prec=PREC[c.get("prec", "fp32")])
        h = lib.mg_create(len(shape), shape[::-1], _spacing(c), _faces(c["faces"]), solid, opt)
        return State(c, h, lib.mg_destroy, b=b, x=torch.zeros_like(b))
    if kind == "flow":
        q, p = _flow_fields(c, seed)
        cells = _shape(c)[::-1]
        h = lib.ns_create(len(cells), cells, 1.0, _block(c))
        if c["fe"]:
            lib.ns_set_stencils(h, lib.NS_STENCIL_FE)
        return State(c, h, lib.ns_destroy, old=q + [p], new=[torch.empty_like(t) for t in q + [p]])
    if kind == "batched":
        sides, masks, b = _batch_inputs(c, seed)
        h = lib.mg_create_batched([(n, n) for n in sides], [(1.0 / (n + 1),) * 2 for n in sides], _faces("DDDD"), masks)
        lib.mg_batched_config(h, 64, 32, 3)  # the autotuner's choice for such batches, kept by the program
        return State(c, h, lib.mg_destroy_batched, b=b, x=[torch.zeros_like(t) for t in b])
    if kind == "advdiff":
        b = _adv_rhs(c, seed)
        h = lib.ad_create((c["nx"], c["ny"]), 1.0, 50.0, 2.0, c["u"], c["v"], lib.AD_UPWIND)
        return State(c, h, lib.ad_destroy, b=b, x=torch.empty_like(b))
    w, b, p, fluid = _guess_inputs(c, seed)
    return State(c, lib.gn_create(w), lib.gn_destroy, b=b, p=p, fluid=fluid, x=torch.empty_like(b))


def run(state):
    s, c, kind = state, state.case, state.case["kind"]
    if kind == "cycle":
        lib.mg_precondition(s.handle, s.b, s.x)
        return s.x
    if kind == "poisson":
        s.x.zero_()
        lib.mg_solve(s.handle, s.b, s.x, TOL)
        return s.x
    if kind == "flow":
        # the last accepted time level is kept, as a program that controls its step does
        for new, old in zip(s.new, s.old):
            new.copy_(old)
        q, p = s.new[:-1], s.new[-1]
        lib.ns_step(s.handle, q[0], q[1], q[2] if len(q) == 3 else None, p, 0.1, 0.01 * c["block"], 1.0, TOL)
        return s.new
    if kind == "batched":
        torch._foreach_zero_(s.x)
        lib.mg_solve_batched(s.handle, s.b, s.x, TOL)
        return torch.cat([t.view(-1) for t in s.x])
    if kind == "advdiff":
        lib.ad_solve(s.handle, s.b, s.x, TOL)
        return s.x
    cells = (c["nx"], c["ny"], c["nz"])
    if c["mode"] == "forward":
        lib.gn_forward(s.handle, cells, s.b, s.p, s.x, n=c["n"])
        return s.x
    loss, grad = lib.gn_gradients(s.handle, cells, s.b, s.p, n=c["n"], fluid=s.fluid,
                                  loss_mode=lib.GN_LOSS_RESIDUAL, h=1.0)
    return {"loss": loss, "grad": grad}


def work(case):
    """Inputs read and outputs written once, and the arithmetic of the method:
    per cell and V(2,2) cycle four sweeps, one residual and the transfers on
    all levels; a solve takes about 20 (2D) or 25 (3D) of them, each with the
    two vector updates of the conjugate gradients."""
    c, kind = case, case["kind"]
    if kind == "batched":
        cells = c["count"] * sum(int(s) ** 2 for s in c["sides"].split(",")) / len(c["sides"].split(","))
        return {"bytes": 9 * cells, "flops": 25 * 95 * cells}
    cells, dim = c["nx"] * c["ny"] * c.get("nz", 1), 3 if c.get("nz", 1) > 1 else 2
    sweep = 2 * (2 * dim + 1) + 2
    cycle = (5 * sweep + 4) * 2 ** dim / (2 ** dim - 1)
    if kind == "cycle":
        return {"bytes": (8 + c["solids"]) * cells, "flops": cycle * cells}
    if kind == "poisson":
        return {"bytes": 8 * cells, "flops": (20 if dim == 2 else 25) * (cycle + sweep + 12) * cells}
    if kind == "flow":
        taps = 3 ** dim * (1 + dim) if c["fe"] else 3 * dim
        return {"bytes": (2 * dim + 2) * 4 * cells + cells,
                "flops": ((20 if dim == 2 else 25) * (cycle + sweep + 12) + 4 * dim * taps) * cells}
    if kind == "advdiff":
        return {"bytes": 8 * cells, "flops": 15 * cycle * cells}
    # the network per voxel: three 16-channel layers and the first and last
    # ones at full resolution, three at half and two at a quarter
    conv = 2 * 27 * (16 * 16 * (2 + 3 / 8 + 2 / 64) + 2 * 16 + 16)
    n = c["n"] * cells
    if c["mode"] == "forward":
        return {"bytes": 12 * n, "flops": conv * n}
    return {"bytes": 12 * n + 4 * lib.GN_NUM_WEIGHTS, "flops": 3 * conv * n}


# ---------------------------------------------------------------------------
# the same in 64 bits, from the definitions
def _slice(f, ax, lo, hi):
    return f.narrow(ax, lo, hi - lo)


def _pad(f, ax, lo, hi):
    """One layer on both sides of `ax`: 'z' zeros, 'c' the adjacent value."""
    n = f.shape[ax]
    first, last = _slice(f, ax, 0, 1), _slice(f, ax, n - 1, n)
    return torch.cat([first if lo == "c" else torch.zeros_like(first), f,
                      last if hi == "c" else torch.zeros_like(last)], ax)


class Grid:
    """The operator sum_a w_a (x_c - x_n) over fluid neighbours and open faces."""

    def __init__(self, shape, w, faces, solid=None):
        self.shape, self.w, self.faces = tuple(shape), w, faces
        self.fluid = torch.ones(shape, dtype=F64, device="cuda") if solid is None else (solid == 0).to(F64)
        self.solid = solid
        self.diag = torch.zeros(shape, dtype=F64, device="cuda")
        dim = len(shape)
        for a in range(dim):
            ax, n = dim - 1 - a, shape[dim - 1 - a]
            f = _pad(self.fluid, ax, "z", "z")
            links = _slice(f, ax, 0, n) + _slice(f, ax, 2, n + 2)
            if faces[2 * a] == "D":
                _slice(links, ax, 0, 1).add_(1)
            if faces[2 * a + 1] == "D":
                _slice(links, ax, n - 1, n).add_(1)
            self.diag += w[a] * links
        self.diag *= self.fluid

    def apply(self, x):
        y, dim = self.diag * x, len(self.shape)
        for a in range(dim):
            ax, n = dim - 1 - a, self.shape[dim - 1 - a]
            p = _pad(x * self.fluid, ax, "z", "z")
            y = y - self.w[a] * (_slice(p, ax, 0, n) + _slice(p, ax, 2, n + 2))
        return y * self.fluid

    def coarse(self):
        solid = None
        if self.solid is not None:
            s = self.solid.to(F64)
            for ax in range(s.dim()):
                n = s.shape[ax]
                s = s.index_select(ax, torch.arange(0, n, 2, device="cuda")) * s.index_select(
                    ax, torch.arange(1, n, 2, device="cuda"))
            solid = s
        return Grid([n // 2 for n in self.shape], [w / 4 for w in self.w], self.faces, solid)


def _restrict(r):
    for ax in range(r.dim()):
        sh = list(r.shape)
        r = r.reshape(sh[:ax] + [sh[ax] // 2, 2] + sh[ax + 1:]).mean(ax + 1)
    return r


def _prolong(e):
    for ax in range(e.dim()):
        e = e.repeat_interleave(2, ax)
    return e


def _vcycle(g, b):
    """V(2,2): two Jacobi sweeps (2/3), the residual's average, the copied
    correction, two sweeps; the coarsest level solved."""
    inv = torch.where(g.diag > 0, (2.0 / 3.0) / g.diag.clamp(min=1e-300), torch.zeros_like(g.diag))
    if any(n % 2 or n // 2 < 4 for n in g.shape):
        n = g.diag.numel()
        keep = (g.diag.reshape(-1) > 0).nonzero().reshape(-1)
        a = torch.stack([g.apply(r.view(g.shape)).reshape(-1)
                         for r in torch.eye(n, dtype=F64, device="cuda")[keep]])[:, keep]
        x = torch.zeros(n, dtype=F64, device="cuda")
        x[keep] = torch.linalg.solve(a, b.reshape(-1)[keep])
        return x.view(g.shape)
    x = inv * b
    x = x + inv * (b - g.apply(x))
    x = (x + _prolong(_vcycle(g.coarse(), _restrict((b - g.apply(x)) * g.fluid)))) * g.fluid
    for _ in range(2):
        x = x + inv * (b - g.apply(x))
    return x


class Separable:
    """The inverse of a Grid's operator without solids, by its eigenvectors."""

    def __init__(self, shape, w, faces):
        self.v, lam = [], torch.zeros([1] * len(shape), dtype=F64, device="cuda")
        for ax, n in enumerate(shape):
            a = len(shape) - 1 - ax
            ends = faces[2 * a:2 * a + 2]
            i, k = torch.arange(n, device="cuda", dtype=F64)[:, None], torch.arange(n, device="cuda", dtype=F64)[None]
            if ends == "DD":
                v, t = torch.sin(math.pi * (k + 1) * (i + 1) / (n + 1)), math.pi * (k + 1) / (n + 1)
            elif ends == "NN":
                v, t = torch.cos(math.pi * k * (i + 0.5) / n), math.pi * k / n
            else:
                v, t = torch.cos(math.pi * (2 * k + 1) * (2 * i + 1) / (2 * (2 * n + 1))), math.pi * (2 * k + 1) / (2 * n + 1)
                v = v if ends == "ND" else v.flip(0)
            self.v.append(v / v.norm(dim=0, keepdim=True))
            view = [1] * len(shape)
            view[ax] = n
            lam = lam + (w[a] * 4 * torch.sin(t / 2) ** 2).view(view)
        self.lam = lam

    def __call__(self, b):
        for ax, v in enumerate(self.v):
            b = torch.movedim(torch.tensordot(v, b, ([0], [ax])), 0, ax)
        b = b / self.lam
        for ax, v in enumerate(self.v):
            b = torch.movedim(torch.tensordot(v, b, ([1], [ax])), 0, ax)
        return b


def _solve(g, b, tol=1e-12):
    """The solution on the fluid cells: directly without solids, else by
    conjugate gradients with the solid-free inverse."""
    m = Separable(g.shape, g.w, g.faces)
    if g.solid is None:
        x = m(b)
        return x + m(b - g.apply(x))
    b = b * g.fluid
    x, r = torch.zeros_like(b), b.clone()
    stop, rz, p = tol * float(b.norm()), None, None
    for _ in range(200):
        if float(r.norm()) <= stop:
            break
        z = m(r) * g.fluid
        new = (r * z).sum()
        p = z if p is None else z + (new / rz) * p
        ap, rz = g.apply(p), new
        alpha = rz / (p * ap).sum()
        x, r = x + alpha * p, r - alpha * ap
    return x


def _flow_step(c, q, p, solid):
    """One projection step: predictor, corrector, pressure increment, correction."""
    dim, dt, nu, uin = len(q), 0.1, 0.01 * c["block"], 1.0
    axis = [dim - 1 - a for a in range(dim)]
    n = [p.shape[axis[a]] for a in range(dim)]
    q = [t.clone() for t in q]

    def ghosts(comp, a):
        return ("z" if a == 0 and comp != 0 else "c"), "c"

    def pairs(f, a, lo, hi):
        f = _pad(f, axis[a], lo, hi)
        return _slice(f, axis[a], 0, n[a] + 1), _slice(f, axis[a], 1, n[a] + 2)

    fixed, denom, fix, grad = [], [], [], []
    for a in range(dim):
        m = torch.zeros_like(q[a], dtype=torch.bool)
        _slice(m, axis[a], 0, 1).fill_(True)
        if a:
            _slice(m, axis[a], n[a], n[a] + 1).fill_(True)
        q[a][m] = uin if a == 0 else 0.0
        fixed.append(m)
        lo, hi = pairs((solid != 0).to(F64), a, "c", "c")
        denom.append(1.0 + 1e8 * dt * ((lo + hi) > 0).to(F64))
        lo, hi = pairs((solid == 0).to(F64), a, "z", "c" if a == 0 else "z")
        fix.append(lo * hi)
        lo, hi = pairs(p, a, "c", "z" if a == 0 else "c")
        grad.append(hi - lo)

    def advecting(comp, b):
        if comp == b:
            return q[b]
        lo, hi = pairs(q[b], comp, *ghosts(b, comp))
        s = lo + hi
        return 0.25 * (_slice(s, axis[b], 0, n[b]) + _slice(s, axis[b], 1, n[b] + 1))

    vel = [[advecting(comp, b) for b in range(dim)] for comp in range(dim)]

    def rate(comp, f):
        out = grad[comp].clone()
        if not c["fe"]:
            for a in range(dim):
                e = _pad(f, axis[a], *ghosts(comp, a))
                m = f.shape[axis[a]]
                lo, hi = _slice(e, axis[a], 0, m), _slice(e, axis[a], 2, m + 2)
                out += vel[comp][a] * (hi - lo) / 2 + nu * (2 * f - lo - hi)
            return out
        e = f
        for a in range(dim):
            e = _pad(e, axis[a], *ghosts(comp, a))
        for off in itertools.product((-1, 0, 1), repeat=dim):
            v = e
            for a in range(dim):
                v = _slice(v, axis[a], 1 + off[a], 1 + off[a] + f.shape[axis[a]])
            far = sum(o != 0 for o in off)
            out += (nu / (4 if dim == 2 else 26) * ((12, -2, -1) if dim == 2 else (88, -6, -3, -2))[far]) * v
            for a in range(dim):
                if off[a]:
                    side = math.prod((1, 4, 1)[off[b] + 1] for b in range(dim) if b != a)
                    out += (off[a] * side / (12.0 if dim == 2 else 72.0)) * vel[comp][a] * v
        return out

    pred = [torch.where(fixed[a], q[a], (q[a] - dt * rate(a, q[a])) / denom[a]) for a in range(dim)]
    star = [torch.where(fixed[a], q[a], (q[a] - dt * rate(a, 0.5 * (pred[a] + q[a]))) / denom[a]) for a in range(dim)]
    b = torch.zeros_like(p)
    for a in range(dim):
        b -= (_slice(star[a], axis[a], 1, n[a] + 1) - _slice(star[a], axis[a], 0, n[a])) / dt
    g = Grid(p.shape, [1.0] * dim, "ND" + "NN" * (dim - 1), solid)
    dp = _solve(g, b)
    for a in range(dim):
        lo, hi = pairs(dp, a, "c", "z" if a == 0 else "c")
        g0 = (hi - lo) * fix[a]
        g0[fixed[a]] = 0.0
        star[a] = star[a] - dt * g0
    return star + [p + dp]


def _advdiff(c, b):
    """Float64 V(2,2) cycles down to rounding."""
    def weights(k):
        """(centre, x-, x+, y-, y+) of level k: upwind differences, nu dt = 100."""
        h = 2.0 ** k
        kd, a, b = 100.0 / h ** 2, 50.0 * c["u"] / h, 50.0 * c["v"] / h
        return (1 + 4 * kd + abs(a) + abs(b), -kd - max(a, 0.0), -kd + min(a, 0.0), -kd - max(b, 0.0),
                -kd + min(b, 0.0))

    def apply(k, x):
        w = weights(k)
        p = torch.nn.functional.pad(x, (1, 1, 1, 1))
        return w[0] * x + w[1] * p[1:-1, :-2] + w[2] * p[1:-1, 2:] + w[3] * p[:-2, 1:-1] + w[4] * p[2:, 1:-1]

    def cycle(k, r):
        om = (2.0 / 3.0) / weights(k)[0]
        if any(n % 2 or n // 2 < 4 for n in r.shape):
            n = r.numel()
            a = torch.stack([apply(k, e.view(r.shape)).reshape(-1) for e in torch.eye(n, dtype=F64, device="cuda")])
            return torch.linalg.solve(a.T, r.reshape(-1)).view(r.shape)
        x = om * r
        x = x + om * (r - apply(k, x))
        x = x + _prolong(cycle(k + 1, _restrict(r - apply(k, x))))
        for _ in range(2):
            x = x + om * (r - apply(k, x))
        return x

    x, stop = b.clone(), 1e-13 * float(b.norm())
    for _ in range(80):
        r = b - apply(0, x)
        if float(r.norm()) <= stop:
            break
        x = x + cycle(0, r)
    return x


def _net(c, seed):
    w, b, p, fluid = _guess_inputs(c, seed)
    w = [torch.from_numpy(t).to("cuda", F64).requires_grad_() for t in w]
    b, p, fluid = b.to(F64), p.to(F64), fluid.to(F64)
    rb, rp = (t.square().mean((1, 2, 3), keepdim=True).sqrt() for t in (b, p))

    def conv(x, k):
        ci, co = GN_IO[k]
        return torch.nn.functional.conv3d(x, w[k].permute(2, 1, 0).reshape(co, ci, 3, 3, 3), padding=1)

    def pool(x):
        return torch.nn.functional.avg_pool3d(x, 2)

    def up(x):
        return x.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)

    relu = torch.relu
    with torch.set_grad_enabled(c["mode"] == "train"):
        e1 = relu(conv(relu(conv(torch.stack([b / rb, p / rp], 1), 0)), 1))
        e2 = relu(conv(relu(conv(pool(e1), 2)), 3))
        e3 = relu(conv(relu(conv(pool(e2), 4)), 5))
        d1 = relu(conv(up(relu(conv(up(e3) + e2, 6))) + e1, 7))
        y = conv(d1, 8)[:, 0]
        if c["mode"] == "forward":
            return y * rb
        r = -b / rb
        for ax in (1, 2, 3):
            m = y.shape[ax]
            f, v = _pad(fluid, ax, "z", "z"), _pad(y, ax, "z", "z")
            for k in (0, 2):
                r = r + fluid * _slice(f, ax, k, k + m) * (y - _slice(v, ax, k, k + m))
        inside = torch.zeros_like(fluid)
        inside[:, 1:-1, 1:-1, 1:-1] = 1
        loss = 0.5 * (r * fluid * inside).square().sum() / y.numel()
        loss.backward()
    return {"loss": float(loss), "grad": torch.cat([t.grad.reshape(-1) for t in w])}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("cycle", "poisson"):
        solid, b = _grid_inputs(c, seed)
        shape, h = _shape(c), _spacing(c)
        if kind == "cycle":
            return _vcycle(Grid(shape, [1.0] * len(shape), c["faces"], solid), b.to(F64) * (1 if solid is None else solid == 0))
        return _solve(Grid(shape, [1 / v ** 2 for v in h], c["faces"]), b.to(F64))
    if kind == "flow":
        q, p = _flow_fields(c, seed)
        return _flow_step(c, [t.to(F64) for t in q], p.to(F64), _block(c))
    if kind == "batched":
        sides, masks, b = _batch_inputs(c, seed)
        return torch.cat([_solve(Grid((n, n), [float(n + 1) ** 2] * 2, "DDDD", m), r.to(F64), 1e-11).reshape(-1)
                          for n, m, r in zip(sides, masks, b)])
    if kind == "advdiff":
        return _advdiff(c, _adv_rhs(c, seed).to(F64))
    return _net(c, seed)
