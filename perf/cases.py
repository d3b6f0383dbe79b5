"""Timing cases of the octree multigrid: what a user's program calls, over the sizes it is used at.

A case is one pass of such a program on a mesh it keeps (a Tree or a Batch): a new right-hand
side goes in, the solve runs to its tolerance, the solution comes out; or the same with the
gradients of a loss; or one cleaning step of a vector field.  The mesh follows from the case
alone, the fields from the seed.  `kind` is one of

  uniform   constant coefficient on a uniform grid (2D or 3D), any boundary types, Helmholtz term
  gauss     3D octree refined in nested spheres around a Gaussian charge
  varcoef   3D uniform grid with a coefficient jump, forward solve
  train     3D uniform grid, solve and backward pass for the source and the coefficient (MGSolve)
  batch     many cylindrical trees of uneven size solved together
  clean     divergence cleaning of a 3D vector field on a refined periodic octree
  cleangrad divergence cleaning and its backward pass on a uniform periodic grid (CleanB)
"""
import functools
import math

import numpy as np
import torch

import paper_1901_11370_gb300 as mg

DIRICHLET, NEUMANN, PERIODIC, AXIS = 0, 1, 2, 3
BC = {"d": DIRICHLET, "n": NEUMANN, "p": PERIODIC}


def listed():
    return [
        # the smallest call: the paper's first 2D example, one small field per call, as in a coupled 2D code
        dict(name="uniform2d_64_fp64", kind="uniform", dim=2, N=8, bx=8, by=8, bz=1, bc="ddd", helm=0.0, prec="fp64",
             smoother="gs", tol=1e-10),
        # an implicit diffusion step: Helmholtz term, insulated in x and periodic in y, uneven block counts
        dict(name="helmholtz2d_1152x864", kind="uniform", dim=2, N=16, bx=72, by=54, bz=1, bc="npd", helm=1.0e3,
             prec="mixed", smoother="gs", tol=1e-10),
        # a box that is not a cube, its block counts odd after two halvings: an ordinary 3D Poisson solve per time step
        dict(name="uniform3d_160x96x48", kind="uniform", dim=3, N=8, bx=20, by=12, bz=6, bc="ddd", helm=0.0,
             prec="mixed", smoother="gs", tol=1e-10),
        # the paper's scaling problem: zero boundary values, 16^3 blocks, Jacobi 2 + 2, FP64 throughout
        dict(name="jacobi3d_128_fp64", kind="uniform", dim=3, N=16, bx=8, by=8, bz=8, bc="ddd", helm=0.0, prec="fp64",
             smoother="jacobi", tol=1e-10),
        # the benchmark tree: 128^3 base and three refined depths around a charge (19.8M unknowns), mixed precision
        dict(name="gauss3d_128_mixed", kind="gauss", base=128, N=8, levels=3, prec="mixed", tol=1e-10),
        # the same solve for a user who wants FP64 cycles
        dict(name="gauss3d_128_fp64", kind="gauss", base=128, N=8, levels=3, prec="fp64", tol=1e-10),
        # a dielectric body: coefficient contrast 100, insulated in x and periodic elsewhere, the coefficient kept
        dict(name="varcoef3d_256_mixed", kind="varcoef", n=256, N=16, contrast=100.0, prec="mixed", tol=1e-10),
        # one training step that learns the coefficient field: new coefficients each step, forward and backward
        dict(name="train3d_64", kind="train", n=64, N=8, tol=1e-11),
        # 512 axisymmetric discharges of 32^2 to 512^2 cells with up to two refined depths, solved as one batch
        dict(name="batch512_mixed", kind="batch", trees=512, kmin=2, kmax=32, prec="mixed", tol=1e-10),
        # a small ensemble of the same, FP64 throughout
        dict(name="batch24_fp64", kind="batch", trees=24, kmin=2, kmax=12, prec="fp64", tol=1e-10),
        # one cleaning step of a magnetic field on a periodic 128^3 grid of 16^3 blocks refined around a source
        dict(name="clean3d_128_mixed", kind="clean", n=128, N=16, levels=2, prec="mixed", order=4, tol=1e-10),
        # cleaning inside a training loop: the cleaned field and the gradient of a loss on it
        dict(name="cleangrad3d_64", kind="cleangrad", n=64, N=16, tol=1e-10),
    ]


def draw(rng):
    """One more case: a kind, then sizes over that kind's whole range."""
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def halvable(b):
        """Block counts near b whose common halvings leave at most 200 blocks (the coarsest level is solved directly)."""
        k = 1
        while True:
            q = [max(k, (v + k // 2) // k * k) for v in b]
            r = list(q)
            while all(v % 2 == 0 for v in r):
                r = [v // 2 for v in r]
            if math.prod(r) <= 200:
                return q
            k *= 2
    kind = rng.choice(["uniform2d", "uniform3d", "gauss", "varcoef", "train", "batch", "clean", "cleangrad"])
    if kind == "uniform2d":
        N = rng.choice([4, 8, 16])
        n = logint(64, 1100)
        bx, by = halvable([max(2, n // N), max(2, int(n * rng.uniform(0.5, 1.0)) // N)])
        bc = rng.choice(["ddd", "npd", "ppd", "dnd"])
        return dict(kind="uniform", dim=2, N=N, bx=bx, by=by, bz=1, bc=bc, helm=rng.choice([0.0, 10.0, 1.0e3]) if bc in ("ddd", "dnd") else 1.0e3,
                    prec=rng.choice(["fp64", "mixed"]), smoother=rng.choice(["gs", "gs", "jacobi"]), tol=1e-10)
    if kind == "uniform3d":
        N = rng.choice([4, 8, 8, 16])
        n = logint(32, 176)
        b = halvable([max(2, int(n * s) // N) for s in (1.0, rng.uniform(0.4, 1.0), rng.uniform(0.4, 1.0))])
        bc = rng.choice(["ddd", "ddn", "dpp"])
        return dict(kind="uniform", dim=3, N=N, bx=b[0], by=b[1], bz=b[2], bc=bc, helm=rng.choice([0.0, 0.0, 30.0]),
                    prec=rng.choice(["fp64", "mixed"]), smoother=rng.choice(["gs", "gs", "jacobi"]), tol=1e-10)
    if kind == "gauss":
        N = rng.choice([8, 8, 16])
        return dict(kind="gauss", base=16 * rng.choice([2, 3, 4, 5, 6, 8] if N == 8 else [2, 3, 4, 5, 6]), N=N, levels=rng.choice([1, 2, 3]),
                    prec=rng.choice(["fp64", "mixed", "mixed"]), tol=1e-10)
    if kind == "varcoef":
        N = rng.choice([8, 16])
        prec = rng.choice(["fp64", "mixed", "mixed"])
        return dict(kind="varcoef", n=N * 2 * logint(32 // N, (128 if prec == "fp64" else 224) // (2 * N)), N=N,
                    contrast=math.exp(rng.uniform(math.log(3.0), math.log(100.0))), prec=prec, tol=1e-10)
    if kind == "train":
        N = rng.choice([8, 16])
        return dict(kind="train", n=N * logint(2, 80 // N), N=N, tol=1e-11)
    if kind == "batch":
        kmax = logint(3, 24)
        return dict(kind="batch", trees=logint(2, 128), kmin=2, kmax=kmax, prec=rng.choice(["fp64", "mixed", "mixed"]), tol=1e-10)
    if kind == "clean":
        N = rng.choice([8, 16])
        return dict(kind="clean", n=N * 2 * logint(2, 128 // (2 * N)), N=N, levels=rng.choice([1, 2]), prec=rng.choice(["fp64", "mixed", "mixed"]),
                    order=rng.choice([2, 4]), tol=1e-10)
    N = rng.choice([8, 16])
    return dict(kind="cleangrad", n=N * 2 * logint(1, 96 // (2 * N)), N=N, tol=1e-10)


# ------------------------------------------------------------------ meshes --

def _refine(dim, nblk, lengths, centre, radii, periodic):
    """Blocks to refine, int32 [k, 4] (depth, i, j, k): depth r where a block's centre lies within
    radii[r] of the centre, closed under 2:1 balance across faces."""
    nblk = [nblk[d] if d < dim else 1 for d in range(3)]
    cur = np.stack(np.meshgrid(*[np.arange(q) for q in nblk], indexing="ij"), -1).reshape(-1, 3)
    kids = np.stack(np.meshgrid(*[np.arange(2 if d < dim else 1) for d in range(3)], indexing="ij"), -1).reshape(-1, 3)
    twice = np.array([2 if d < dim else 1 for d in range(3)])
    sets = []
    for r, rad in enumerate(radii):
        size = np.array([lengths[d] / (nblk[d] << r) for d in range(dim)])
        far = (((cur[:, :dim] + 0.5) * size - np.asarray(centre[:dim])) ** 2).sum(1)
        sets.append(cur[far <= rad * rad])
        cur = (sets[-1][:, None, :] * twice + kids[None]).reshape(-1, 3)
    for r in range(len(sets) - 1, 0, -1):
        ext = np.array([nblk[d] << r if d < dim else 1 for d in range(3)])
        need = [sets[r - 1]]
        for d in range(dim):
            for s in (-1, 1):
                q = sets[r].copy()
                q[:, d] += s
                if periodic[d]:
                    q[:, d] %= ext[d]
                else:
                    q = q[(q[:, d] >= 0) & (q[:, d] < ext[d])]
                need.append(q // twice)
        sets[r - 1] = np.unique(np.concatenate(need), axis=0)
    rows = [np.concatenate([np.full((len(s), 1), r), s], 1) for r, s in enumerate(sets) if len(s)]
    return np.concatenate(rows).astype(np.int32) if rows else np.zeros((0, 4), np.int32)


RADII3 = (0.30, 0.22, 0.14)
CENTRE3 = (0.55, 0.45, 0.52)


@functools.lru_cache(maxsize=64)
def _mesh(kind, **kw):
    if kind == "gauss":
        nb = kw["base"] // kw["N"]
        return _refine(3, (nb,) * 3, (1.0,) * 3, CENTRE3, RADII3[:kw["levels"]], (False,) * 3)
    nb = kw["n"] // kw["N"]
    return _refine(3, (nb,) * 3, (1.0,) * 3, CENTRE3, (0.28, 0.12)[:kw["levels"]], (True,) * 3)


def _case_mesh(c):
    if c["kind"] == "gauss":
        return _mesh("gauss", base=c["base"], N=c["N"], levels=c["levels"])
    return _mesh("clean", n=c["n"], N=c["N"], levels=c["levels"])


@functools.lru_cache(maxsize=16)
def _rings(trees, kmin, kmax):
    """The batch's meshes: (blocks per side, ring point, refine records) per tree."""
    rng = np.random.default_rng(1901)
    out = []
    for _ in range(trees):
        k, lev = int(rng.integers(kmin, kmax + 1)), int(rng.integers(0, 3))
        at = tuple(rng.uniform(0.2, 0.8, 2))
        out.append((k, at, _refine(2, (k, k), (1.0, 1.0), at, (0.1, 0.05)[:lev], (False, False))))
    return out


def _cells(c):
    """Leaf cells of the case's mesh."""
    k = c["kind"]
    if k == "uniform":
        return c["bx"] * c["by"] * c["bz"] * c["N"] ** c["dim"]
    if k == "gauss":
        return ((c["base"] // c["N"]) ** 3 + 7 * len(_case_mesh(c))) * c["N"] ** 3
    if k == "clean":
        return ((c["n"] // c["N"]) ** 3 + 7 * len(_case_mesh(c))) * c["N"] ** 3
    if k == "batch":
        return sum((b * b + 3 * len(r)) * 256 for b, _, r in _rings(c["trees"], c["kmin"], c["kmax"]))
    return c["n"] ** 3


def work(case):
    """What one pass cannot do without: its fields read and written once; the operator applied to every
    cell once per field solved for."""
    n, k = _cells(case), case["kind"]
    fields, solves = {"uniform": (2, 1), "gauss": (2, 1), "varcoef": (2, 1), "batch": (2, 1), "train": (6, 2),
                      "clean": (7, 1), "cleangrad": (12, 2)}[k]
    return {"bytes": 8.0 * n * fields, "flops": (17.0 if k in ("varcoef", "train", "batch") else 8.0) * n * solves}


# ------------------------------------------------------------------ fields --

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, n, a, b):
    return (a + (b - a) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)).tolist()


def _leaf_index(leaf_blocks, dim, N):
    """Global cell index (I, J, K) on its own depth's grid and the depth of every leaf cell, leaf order."""
    lb = torch.from_numpy(leaf_blocks).cuda().long()
    a = torch.arange(N, device="cuda")
    if dim == 2:
        lk, lj, li = torch.meshgrid(torch.zeros(1, device="cuda", dtype=torch.long), a, a, indexing="ij")
    else:
        lk, lj, li = torch.meshgrid(a, a, a, indexing="ij")
    idx = [(lb[:, d + 1:d + 2] * (N if d < dim else 1) + v.reshape(1, -1)).reshape(-1) for d, v in enumerate((li, lj, lk))]
    return idx, lb[:, :1].expand(-1, N ** dim).reshape(-1)


def _field(shape, corr, g):
    """Zero-mean Gaussian random field of unit variance on a periodic grid, correlation length `corr` of its longest side."""
    w = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    top = max(shape)
    k2 = sum((2 * math.pi * torch.fft.fftfreq(s, 1.0 / top, device="cuda", dtype=torch.float64).reshape([-1 if e == d else 1 for e in range(len(shape))])) ** 2
             for d, s in enumerate(shape))
    f = torch.fft.ifftn(torch.fft.fftn(w) * torch.exp(-0.5 * k2 * corr ** 2)).real
    f -= f.mean()
    return f / f.std()


def _uniform_geom(c):
    """(cells per dimension, cell size): the longest side is 1 and cells are cubes."""
    n = [c["N"] * b for b in (c["bx"], c["by"], c["bz"])[:c["dim"]]]
    return n, 1.0 / max(n)


def _uniform_fields(c, seed):
    n, _ = _uniform_geom(c)
    f = _field(tuple(n), 0.04, _gen(seed))
    return f + (0.3 if "d" in c["bc"][:c["dim"]] or c["helm"] > 0 else 0.0)


def _varcoef_fields(c, seed):
    """eps (a sphere of the given contrast) and a right-hand side of zero mean, [x, y, z]."""
    g = _gen(seed)
    ctr = _rand(g, 3, 0.35, 0.65)
    x = (torch.arange(c["n"], device="cuda", dtype=torch.float64) + 0.5) / c["n"]
    r2 = (x[:, None, None] - ctr[0]) ** 2 + (x[None, :, None] - ctr[1]) ** 2 + (x[None, None, :] - ctr[2]) ** 2
    return 1.0 + (c["contrast"] - 1.0) * (r2 < 0.0625).double(), _field((c["n"],) * 3, 0.05, g)


def _train_fields(c, seed):
    """Log-normal eps, source and target, [x, y, z]."""
    g = _gen(seed)
    n = (c["n"],) * 3
    return torch.exp(0.7 * _field(n, 0.08, g)), _field(n, 0.05, g) + 0.5, 0.02 * _field(n, 0.1, g)


def _turbulence(n, g):
    """Vector field on a periodic n^3 grid, component spectra k^(-11/3) for 1 <= k <= n/2, mean square 1."""
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    kk = torch.sqrt(k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2)
    amp = torch.where((kk >= 1) & (kk <= n / 2), kk.clamp(min=1.0) ** (-11.0 / 6.0), 0.0)
    b = torch.stack([torch.fft.ifftn(torch.fft.fftn(torch.randn((n,) * 3, generator=g, device="cuda", dtype=torch.float64)) * amp).real for _ in range(3)])
    return b / torch.sqrt((b * b).sum(0).mean())


def _params(c):
    jac = c.get("smoother") == "jacobi"
    return dict(rel_tol=c["tol"], max_cycles=150, precision=mg.MG_FP64 if c["prec"] == "fp64" else mg.MG_FP32_DC,
                inner_cycles=1 if c["prec"] == "fp64" else 3 if c["kind"] == "varcoef" or jac else 2,
                smoother=mg.MG_SMOOTH_JACOBI if jac else mg.MG_SMOOTH_RBGS)


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _faces(bc, dim):
    t = [BC[bc[d]] for d in range(dim) for _ in (0, 1)]
    return t + [PERIODIC] * (6 - len(t))


def _solve_state(tree, c, f, **more):
    return dict(tree=tree, f=f, zero=torch.zeros_like(f), args=_params(c), **more)


def _prepare_uniform(c, seed):
    n, h = _uniform_geom(c)
    t = mg.Tree(c["dim"], c["N"], mg.MG_CART, _faces(c["bc"], c["dim"]), [0.0] * 6, n, [0.0] * c["dim"], [h * q for q in n], helm=c["helm"])
    idx, _ = _leaf_index(t.leaf_blocks(), c["dim"], c["N"])
    return _solve_state(t, c, _uniform_fields(c, seed)[tuple(idx[:c["dim"]])].contiguous())


def _prepare_gauss(c, seed):
    g = _gen(seed)
    ctr = [q + d for q, d in zip(CENTRE3, _rand(g, 3, -0.01, 0.01))]
    sg, q = _rand(g, 1, 0.018, 0.024)[0], _rand(g, 1, 0.5, 2.0)[0]
    t = mg.Tree(3, c["N"], mg.MG_CART, [DIRICHLET] * 6, [0.0] * 6, (c["base"],) * 3, (0.0,) * 3, (1.0,) * 3, _case_mesh(c), finalize=False)

    def potential(x, y, z):
        r = torch.sqrt((x - ctr[0]) ** 2 + (y - ctr[1]) ** 2 + (z - ctr[2]) ** 2)
        return q * torch.erf(r / sg) / (4 * math.pi * r)
    for lev, info in enumerate(t.levels()):
        a = [(torch.arange(info["ncell"][d], device="cuda", dtype=torch.float64) + 0.5) * info["h"][d] for d in range(3)]
        for face in range(6):
            d, at = face // 2, torch.tensor(float(face % 2), device="cuda", dtype=torch.float64)
            xyz = [at if e == d else None for e in range(3)]
            t1, t2 = [e for e in range(3) if e != d]
            xyz[t1], xyz[t2] = a[t1][None, :], a[t2][:, None]
            t.set_bc_plane(face, lev, potential(*xyz).cpu().numpy())
    t.finalize()
    idx, dep = _leaf_index(t.leaf_blocks(), 3, c["N"])
    h = 1.0 / (c["base"] * torch.pow(2.0, dep.double()))
    r2 = sum(((i + 0.5) * h - o) ** 2 for i, o in zip(idx, ctr))
    return _solve_state(t, c, (-q / (sg ** 3 * math.pi ** 1.5) * torch.exp(-r2 / sg ** 2)).contiguous())


def _cube(c, faces):
    return mg.Tree(3, c["N"], mg.MG_CART, faces, [0.0] * 6, (c["n"],) * 3, (0.0,) * 3, (1.0,) * 3)


VAR_FACES = [NEUMANN, NEUMANN, PERIODIC, PERIODIC, PERIODIC, PERIODIC]
TRAIN_FACES = [DIRICHLET, DIRICHLET, NEUMANN, NEUMANN, PERIODIC, PERIODIC]


def _prepare_varcoef(c, seed):
    t = _cube(c, VAR_FACES)
    at = tuple(_leaf_index(t.leaf_blocks(), 3, c["N"])[0])
    eps, f = _varcoef_fields(c, seed)
    t.set_eps(eps[at].contiguous())
    return _solve_state(t, c, f[at].contiguous())


def _prepare_train(c, seed):
    t = _cube(c, TRAIN_FACES)
    at = tuple(_leaf_index(t.leaf_blocks(), 3, c["N"])[0])
    eps, f, target = (v[at].contiguous() for v in _train_fields(c, seed))
    return dict(tree=t, f=f.requires_grad_(), eps=eps.requires_grad_(), target=target, vol=1.0 / c["n"] ** 3, tol=c["tol"])


def _prepare_batch(c, seed):
    g = _gen(seed)
    faces = [AXIS, DIRICHLET, DIRICHLET, DIRICHLET, PERIODIC, PERIODIC]
    trees, fs, es = [], [], []
    rings = _rings(c["trees"], c["kmin"], c["kmax"])
    rnd = np.array(_rand(g, 3 * len(rings), 0.0, 1.0)).reshape(-1, 3)
    for (k, at, ref), u in zip(rings, rnd):
        t = mg.Tree(2, 16, mg.MG_CYL, faces, [0.0] * 6, (16 * k, 16 * k), (0.0, 0.0), (1.0, 1.0), ref, coarse_max=1024, finalize=False)
        (i, j, _), dep = _leaf_index(t.leaf_blocks(), 2, 16)
        h = 1.0 / (16 * k * torch.pow(2.0, dep.double()))
        r, z = (i + 0.5) * h, (j + 0.5) * h
        w = 0.025 + 0.01 * u[0]
        fs.append(-torch.exp(-((r - at[0]) ** 2 + (z - at[1]) ** 2) / w ** 2) / (math.pi * w * w))
        es.append(1.0 + 0.5 * torch.sin(2 * math.pi * (z + u[1])))
        trees.append(t)
    b = mg.Batch(trees)
    b.set_eps(torch.cat(es))
    return _solve_state(b, c, torch.cat(fs))


def _prepare_clean(c, seed):
    g = _gen(seed)
    t = mg.Tree(3, c["N"], mg.MG_CART, [PERIODIC] * 6, [0.0] * 6, (c["n"],) * 3, (0.0,) * 3, (1.0,) * 3, _case_mesh(c))
    (i, j, k), dep = _leaf_index(t.leaf_blocks(), 3, c["N"])
    b = _turbulence(c["n"], g)[:, i >> dep, j >> dep, k >> dep]
    h = 1.0 / (c["n"] * torch.pow(2.0, dep.double()))
    dx = torch.stack([(q + 0.5) * h - o for q, o in zip((i, j, k), CENTRE3)])
    b -= 60.0 * dx * torch.exp(-(dx * dx).sum(0) / 0.0025)
    return dict(tree=t, B=b.contiguous(), args=dict(rel_tol=c["tol"], max_cycles=80, order=c["order"],
                                                   precision=mg.MG_FP64 if c["prec"] == "fp64" else mg.MG_FP32_DC))


def _prepare_cleangrad(c, seed):
    g = _gen(seed)
    t = _cube(c, [PERIODIC] * 6)
    at = tuple(_leaf_index(t.leaf_blocks(), 3, c["N"])[0])
    B, target = (_turbulence(c["n"], g)[(slice(None),) + at].contiguous() for _ in range(2))
    return dict(tree=t, B=B.requires_grad_(), target=target, tol=c["tol"])


# -------------------------------------------------------------------- runs --

def run(state):
    t = state["tree"]
    if "eps" in state:
        phi = mg.MGSolve.apply(t, state["f"], state["eps"], state["tol"], 100, state["tol"])
        loss = 0.5 * state["vol"] * ((phi - state["target"]) ** 2).sum()
        df, de = torch.autograd.grad(loss, (state["f"], state["eps"]))
        return phi.detach(), df, de
    if "B" in state and "target" in state:
        Bn = mg.CleanB.apply(t, state["B"], state["tol"], 100)
        loss = 0.5 * ((Bn - state["target"]) ** 2).mean()
        return Bn.detach(), torch.autograd.grad(loss, state["B"])[0]
    if "B" in state:
        Bn, div, _, _ = t.clean(state["B"], **state["args"])
        return Bn, div
    t.set_rhs(state["f"])
    t.set_phi(state["zero"])
    t.solve(**state["args"])
    return t.get_phi()


# ------------------------------------------------------------- exact values --

def _line(n, h, bc):
    """Second difference of cell-centred values along one dimension (Dirichlet ghost -x, Neumann ghost x)."""
    m = torch.diag(torch.full((n,), -2.0, device="cuda", dtype=torch.float64))
    m += torch.diag(torch.ones(n - 1, device="cuda", dtype=torch.float64), 1) + torch.diag(torch.ones(n - 1, device="cuda", dtype=torch.float64), -1)
    if bc == PERIODIC:
        m[0, -1] += 1.0
        m[-1, 0] += 1.0
    else:
        s = -1.0 if bc == DIRICHLET else 1.0
        m[0, 0] += s
        m[-1, -1] += s
    return m / h ** 2


class _Separable:
    """The constant-coefficient operator minus `helm`, diagonalised one dimension at a time."""

    def __init__(self, n, h, bc, helm=0.0):
        ev = [torch.linalg.eigh(_line(q, h, b)) for q, b in zip(n, bc)]
        self.q = [e.eigenvectors for e in ev]
        lam = sum(e.eigenvalues.reshape([-1 if a == d else 1 for a in range(len(n))]) for d, e in enumerate(ev)) - helm
        self.inv = torch.where(lam.abs() < 1e-6 * lam.abs().max() / max(n) ** 2, 0.0, 1.0 / lam)  # the constants: zero mean

    def solve(self, f):
        for d, q in enumerate(self.q):
            f = torch.movedim(torch.tensordot(q, f, dims=([0], [d])), 0, d)
        f = f * self.inv
        for d, q in enumerate(self.q):
            f = torch.movedim(torch.tensordot(q, f, dims=([1], [d])), 0, d)
        return f


def _shift(x, d, s, bc, coef=False):
    """The neighbour on side s (+1, -1) of dimension d, with the ghost rules of the boundary."""
    if bc == PERIODIC:
        return torch.roll(x, -s, d)
    inner = x.narrow(d, 1, x.shape[d] - 1) if s > 0 else x.narrow(d, 0, x.shape[d] - 1)
    edge = x.narrow(d, x.shape[d] - 1, 1) if s > 0 else x.narrow(d, 0, 1)
    if bc == DIRICHLET and not coef:
        edge = -edge
    return torch.cat([inner, edge] if s > 0 else [edge, inner], d)


def _apply(x, eps, h, bc):
    """div(eps grad x), eps at a face the harmonic mean of its two cells."""
    out = torch.zeros_like(x)
    for d, b in enumerate(bc):
        for s in (1, -1):
            e2 = _shift(eps, d, s, b, True)
            out = out + 2 * eps * e2 / (eps + e2) * (_shift(x, d, s, b) - x)
    return out / h ** 2


def _pcg(f, eps, h, bc):
    """Solution of div(eps grad x) = f by conjugate gradients in 64 bits, preconditioned by the
    constant-coefficient operator; zero mean where no face is Dirichlet."""
    sep = _Separable(f.shape, h, bc)
    free = DIRICHLET not in bc

    def proj(v):
        return v - v.mean() if free else v

    def prec(r):
        return proj(sep.solve(r))
    x, r = torch.zeros_like(f), proj(f)
    best, since, z = (float("inf"), x), 0, prec(r)
    p, rz, r0 = z, (r * z).sum(), r.norm()
    for it in range(400):
        ap = proj(_apply(p, eps, h, bc))
        a = rz / (p * ap).sum()
        x, r = x + a * p, r - a * ap
        if it % 25 == 24:  # the true residual now and then, so that it does not drift
            r = proj(f - _apply(x, eps, h, bc))
        rel = float(r.norm() / r0)
        if rel < best[0]:
            best, since = (rel, x), 0
        else:
            since += 1
        if rel < 1e-14 or since > 40:
            break
        z = prec(r)
        new = (r * z).sum()
        p, rz = z + new / rz * p, new
    return proj(best[1])


def _morton_blocks(nb):
    """The leaf blocks (depth, i, j, k) of a uniform mesh of nb blocks, in Morton order."""
    ijk = np.stack(np.meshgrid(*[np.arange(q) for q in nb], indexing="ij"), -1).reshape(-1, 3).astype(np.int64)
    code = sum(((ijk[:, d] >> b) & 1) << (3 * b + d) for b in range(20) for d in range(3))
    return np.concatenate([np.zeros((len(ijk), 1), np.int64), ijk], 1)[np.argsort(code)].astype(np.int32)


def exact(case, seed):
    """The discrete solution in 64 bits, by eigenvectors or conjugate gradients, on the uniform grids.  The refined
    meshes give None: without a multigrid method of its own, a Krylov solve of their composite operator takes far
    longer than 20 seconds."""
    c, kind = case, case["kind"]
    if kind in ("gauss", "clean", "batch"):
        return None

    dim = c.get("dim", 3)
    nb = [c["bx"], c["by"], c["bz"]] if kind == "uniform" else [c["n"] // c["N"]] * 3
    at = tuple(_leaf_index(_morton_blocks(nb), dim, c["N"])[0][:dim])
    if kind == "uniform":
        n, h = _uniform_geom(c)
        return _Separable(n, h, [BC[b] for b in c["bc"]][:c["dim"]], c["helm"]).solve(_uniform_fields(c, seed))[at]
    h = 1.0 / c["n"]
    if kind == "varcoef":
        eps, f = _varcoef_fields(c, seed)
        return _pcg(f, eps, h, VAR_FACES[::2])[at]
    if kind == "train":
        eps, f, target = _train_fields(c, seed)
        bc = TRAIN_FACES[::2]
        phi = _pcg(f, eps, h, bc)
        lam = _pcg(h ** 3 * (phi - target), eps, h, bc)
        e = eps.clone().requires_grad_()
        de = torch.autograd.grad(-(lam * _apply(phi, e, h, bc)).sum(), e)[0]
        return phi[at], lam[at], de[at]
    g = _gen(seed)
    sep = _Separable((c["n"],) * 3, h, [PERIODIC] * 3)

    def diff(x, d):
        return (torch.roll(x, -1, d) - torch.roll(x, 1, d)) / (2 * h)

    def clean(b):
        phi = sep.solve(sum(diff(b[d], d) for d in range(3)))
        return torch.stack([b[d] - diff(phi, d) for d in range(3)])
    B, target = _turbulence(c["n"], g), _turbulence(c["n"], g)
    Bn = clean(B)
    gB = clean((Bn - target) / B.numel())  # the map is symmetric on a uniform periodic grid
    return tuple(v[(slice(None),) + at] for v in (Bn, gB))
