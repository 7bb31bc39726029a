"""Performance cases of the patch-smoother library, through its public entry points.

A case is one call (or one solve) of a user's program on a problem that was set up before: patch sweeps and local
V-cycles on structured and unstructured meshes, the Lanczos estimate of the Chebyshev intervals, preconditioned CG
solves (alone and in a batch), and the training of the interval network.  Meshes, coefficients and vectors are
seeded; kappa is 10^U(-d, d) per cell (d = "decades", 0: constant).

Mixed-precision sweeps and local solves return their result as float32: the library computes it in FP32 and widens
it to the caller's FP64 vector, so the conversion is exact.
"""
import math

import numpy as np
import torch

from paper_2510_17785_gb300 import inputs, pmg

MAX_COARSE = 2600            # free DoFs of the coarsest level (dense coarse solve) of a drawn hierarchy


# ------------------------------------------------------------------ the cases
def _smooth(name, dim, p, n, precision, decades, smoother="chebyshev"):
    return {"name": name, "kind": "smooth", "dim": dim, "p": p, "n": n, "precision": precision, "decades": decades,
            "smoother": smoother}


def listed():
    return [
        # one small 2D sweep: launches and the latency of a patch are all there is (the benchmark's first workload)
        _smooth("smooth_2d_q4_n16_fp64", 2, 4, 16, "fp64", 0.0),
        # a large 2D sweep at high degree with jumping coefficients
        _smooth("smooth_2d_q7_n160_mixed", 2, 7, 160, "mixed", 2.0),
        # low degree in 3D: many small patches, little arithmetic per byte
        _smooth("smooth_3d_q2_n40_mixed", 3, 2, 40, "mixed", 1.0),
        # the finest-level sweep of the headline workload (3D Q4, 32^3 perturbed cells)
        _smooth("smooth_3d_q4_n32_mixed", 3, 4, 32, "mixed", 0.0),
        # degree 7 with coefficients over six decades (the variable-coefficient workload on a smaller mesh)
        _smooth("smooth_3d_q7_n24_mixed", 3, 7, 24, "mixed", 3.0),
        # the plain FP64 method
        _smooth("smooth_3d_q4_n16_fp64", 3, 4, 16, "fp64", 0.0),
        # local solves of some patches, two V-cycles each (a caller that drives the local solver itself)
        {"name": "local_3d_q6_n12_mixed", "kind": "local", "dim": 3, "p": 6, "n": 12, "precision": "mixed",
         "decades": 1.0, "smoother": "chebyshev", "count": 777, "cycles": 2},
        # a sweep on an unstructured hexahedral mesh (split tetrahedra, valences 4 to 24)
        {"name": "usmooth_tetsplit_q6_mixed", "kind": "usmooth", "mesh": "tetsplit", "size": 4, "p": 6,
         "precision": "mixed", "decades": 2.0, "smoother": "chebyshev"},
        # the headline: one GMG-preconditioned CG solve to 1e-8
        {"name": "solve_3d_q4_n32_mixed", "kind": "solve", "dim": 3, "p": 4, "n": 32, "precision": "mixed",
         "decades": 0.0, "rtol": 1e-8},
        # independent problems of mixed degree and mesh kind solved together
        {"name": "batch_4_unstructured_mixed", "kind": "batch", "count": 4, "size": 4, "precision": "mixed",
         "decades": 2.0, "rtol": 1e-8},
        # the Chebyshev intervals of every patch, mesh level and p-level (16 Lanczos steps each)
        {"name": "lanczos_3d_q4_n16", "kind": "lanczos", "dim": 3, "p": 4, "n": 16, "decades": 2.0},
        # training of the interval network on the estimates of a few problems (three epochs of the usual run)
        {"name": "train_n1750_b256", "kind": "train", "n": 1750, "batch": 256, "epochs": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _coarsest(n):
    while n % 2 == 0 and n // 2 >= 2:
        n //= 2
    return n


def _cells_per_side(rng, dim, p, cells):
    """Cells per direction, spread over [3, cells], whose coarsest level the dense coarse solve takes quickly."""
    while True:
        n = max(3, _log_int(rng, 3, cells))
        if (p * _coarsest(n) - 1) ** dim <= MAX_COARSE:
            return n


def draw(rng):
    kind = rng.choice(["smooth"] * 5 + ["usmooth"] * 2 + ["local", "solve", "batch", "lanczos", "train"])
    decades = rng.choice([0.0, round(rng.uniform(0.2, 3.0), 2)])
    smoother = rng.choice(["chebyshev", "chebyshev", "chebyshev", "jacobi"])
    if kind in ("smooth", "local"):
        dim = rng.choice([2, 3, 3])
        precision = rng.choice(["mixed", "mixed", "fp64"])
        p = rng.randint(2, 8 if dim == 2 or precision == "mixed" else 6)
        if dim == 2:
            n = _cells_per_side(rng, 2, p, 1100 // p if precision == "mixed" else 500 // p)
        else:
            n = _cells_per_side(rng, 3, p, 160 // p if precision == "mixed" else 56 // p)
        case = {"kind": kind, "dim": dim, "p": p, "n": n, "precision": precision, "decades": decades,
                "smoother": smoother}
        if kind == "local":
            patches = (n - 1) ** dim
            case["count"] = rng.randint(1, min(patches, 1500 if dim == 3 else 8000))
            case["cycles"] = rng.randint(1, 3)
        return case
    if kind == "usmooth":
        mesh = rng.choice(["tetsplit", "extruded", "trisplit2d"])
        size = rng.randint(4 if mesh == "extruded" else 2, {"tetsplit": 5, "extruded": 9, "trisplit2d": 30}[mesh])
        p = rng.randint(2, 8)
        precision = rng.choice(["mixed", "mixed", "fp64"]) if p <= 6 else "mixed"
        if precision == "fp64" and mesh != "trisplit2d":
            size = min(size, {"tetsplit": 3, "extruded": 6}[mesh])
        return {"kind": "usmooth", "mesh": mesh, "size": size, "p": p, "precision": precision, "decades": decades,
                "smoother": smoother}
    if kind == "solve":
        dim = rng.choice([2, 3])
        p = rng.randint(2, 6)
        n = 2 ** rng.randint(2, 6 if dim == 2 else (4 if p <= 4 else 3))
        return {"kind": "solve", "dim": dim, "p": p, "n": n, "precision": rng.choice(["mixed", "mixed", "fp64"]),
                "decades": min(decades, 1.0), "rtol": 10.0 ** rng.randint(-9, -7)}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(2, 4), "size": rng.randint(2, 4), "precision": "mixed",
                "decades": min(decades, 2.0), "rtol": 1e-8}
    if kind == "lanczos":
        dim = rng.choice([2, 3])
        p = rng.randint(2, 8 if dim == 2 else 5)
        n = _cells_per_side(rng, dim, p, 300 // p if dim == 2 else 64 // p)
        return {"kind": "lanczos", "dim": dim, "p": p, "n": n, "decades": decades}
    n = _log_int(rng, 150, 6000)
    batch = _log_int(rng, 64, min(1024, n))
    return {"kind": "train", "n": n, "batch": batch, "epochs": max(1, min(3, (18 * batch) // n))}


# ------------------------------------------------------------------ inputs
def _levels(n):
    levels = 1
    while n % 2 == 0 and n // 2 >= 2:
        n //= 2
        levels += 1
    return levels


def _kappa(rng, cells, decades):
    return 10.0 ** rng.uniform(-decades, decades, cells)


def _structured_inputs(case, seed):
    """(coords, kappa, b, u, ids, r) of a structured case, host arrays."""
    dim, p, n = case["dim"], case["p"], case["n"]
    rng = np.random.default_rng(seed)
    coords = inputs.valid_perturbation(rng, dim, n, 0.25 if dim == 3 else 0.2, "uniform", seed)
    kappa = _kappa(rng, n ** dim, case["decades"])
    free = inputs.free_dof_mask(dim, p, n)
    b = np.where(free, rng.uniform(-1.0, 1.0, free.size), 0.0)
    u = np.where(free, rng.uniform(-1.0, 1.0, free.size), 0.0)
    ids = r = None
    if case["kind"] == "local":
        ids = rng.permutation((n - 1) ** dim)[: case["count"]].astype(np.int64)
        r = rng.uniform(-1.0, 1.0, (ids.size, (2 * p - 1) ** dim))
    return coords, kappa, b, u, ids, r


def _options(case):
    return {"precision": pmg.PREC_MIXED if case.get("precision", "mixed") == "mixed" else pmg.PREC_FP64,
            "smoother": pmg.SMOOTHER_JACOBI if case.get("smoother") == "jacobi" else pmg.SMOOTHER_CHEBYSHEV}


def _unstructured_inputs(mesh, size, p, decades, seed):
    coords, cells, bnd = inputs.unstructured_mesh(mesh, size, seed)
    rng = np.random.default_rng([seed, 17])
    return coords, cells, bnd.astype(np.uint8), _kappa(rng, len(cells), decades)


def _batch_specs(case, seed):
    """(mesh kind, size, degree, seed) of every problem: degrees 2, 4, 6, 8 in turn, alternating mesh kinds."""
    kinds = [("tetsplit", 0), ("extruded", 2), ("tetsplit", -1), ("trisplit2d", 8)]
    return [(kinds[i][0], max(2, case["size"] + kinds[i][1]), (2, 4, 6, 8)[i], seed * 8 + i)
            for i in range(case["count"])]


def _vectors(total, seed):
    """b and u of an unstructured mesh (the library ignores their Dirichlet entries)."""
    rng = np.random.default_rng([seed, 23])
    return rng.uniform(-1.0, 1.0, total), rng.uniform(-1.0, 1.0, total)


def _unstructured_context(coords, cells, bnd, kappa, p, **options):
    dim = coords.shape[1]
    ctx = pmg.Context(0, bounds=pmg.BOUNDS_LANCZOS, **options)
    ctx.mesh_upload(dim, coords, cells, p, bnd, kappa)
    ctx.setup()
    return ctx


def _train_inputs(case, seed):
    """Features, targets (FP32), their normalisation and the start parameters, host arrays."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    x = rng.normal(size=(n, 16)) * np.linspace(0.1, 2.0, 16) + np.linspace(-1.0, 1.0, 16)
    w = rng.normal(size=(16, 2)) / 4.0
    t = np.tanh(x @ w) + 0.1 * rng.normal(size=(n, 2)) + np.array([0.8, -1.5])
    return x.astype(np.float32), t.astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    cuda = lambda a: torch.tensor(a, device="cuda")
    if kind in ("smooth", "local", "solve", "lanczos"):
        coords, kappa, b, u, ids, r = _structured_inputs(case, seed)
        ctx = pmg.Context(0, **_options(case))
        ctx.mesh_structured(case["dim"], case["n"], case["p"], _levels(case["n"]), coords, kappa)
        ctx.setup()
        state = {"case": dict(case), "ctx": ctx, "level": ctx.n_levels - 1}
        if kind in ("smooth", "solve"):
            state.update(b=cuda(b), u=cuda(u))
        if kind == "local":
            state.update(ids=cuda(ids), r=cuda(r), d=torch.empty(r.shape, dtype=torch.float64, device="cuda"))
        return state
    if kind == "usmooth":
        mesh = _unstructured_inputs(case["mesh"], case["size"], case["p"], case["decades"], seed)
        ctx = _unstructured_context(*mesh, case["p"], **_options(case))
        b, u = _vectors(ctx.num_dofs(0)[0], seed)
        return {"case": dict(case), "ctx": ctx, "level": 0, "b": cuda(b), "u": cuda(u)}
    if kind == "batch":
        ctxs, bs = [], []
        for mesh, size, p, s in _batch_specs(case, seed):
            ctx = _unstructured_context(*_unstructured_inputs(mesh, size, p, case["decades"], s), p, autotune=2,
                                        **_options(case))
            ctxs.append(ctx)
            bs.append(cuda(_vectors(ctx.num_dofs(0)[0], s)[0]))
        return {"case": dict(case), "ctxs": ctxs, "bs": bs, "us": [torch.zeros_like(b) for b in bs]}
    x, t = _train_inputs(case, seed)
    x, t = cuda(x), cuda(t)
    return {"case": dict(case), "x": x, "t": t, "norm": cuda(pmg.mlp_norm(x, t)), "theta": cuda(pmg.mlp_init(seed))}


# ------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    narrow = (lambda v: v.float()) if case.get("precision") == "mixed" else (lambda v: v)
    if kind in ("smooth", "usmooth"):
        state["ctx"].patch_smooth(state["level"], state["b"], state["u"], 1, False)
        return narrow(state["u"])
    if kind == "local":
        state["ctx"].local_vcycle(state["level"], state["ids"], state["r"], state["d"], case["cycles"])
        return narrow(state["d"])
    if kind == "solve":
        state["ctx"].solve_cg(state["b"], state["u"], case["rtol"], 300)
        return state["u"]
    if kind == "batch":
        pmg.batch_solve_cg(state["ctxs"], state["bs"], state["us"], case["rtol"], 300)
        return state["us"]
    if kind == "lanczos":
        ctx = state["ctx"]
        ctx.compute_bounds(pmg.BOUNDS_LANCZOS)
        return [ctx.get_ritz(level) for level in range(ctx.n_levels)]
    theta = state["theta"].clone()
    losses = pmg.mlp_train(theta, state["norm"], state["x"], state["t"], epochs=case["epochs"], batch=case["batch"],
                           lr=2e-3, asym=4.0)
    return theta, losses


# ------------------------------------------------------------------ work
def _cell_flops(dim, q):
    """One sum-factorised cell apply: 4 d one-dimensional sweeps and the point products."""
    n = q + 1
    return 8 * dim * n ** (dim + 1) + (2 * dim * dim - dim) * n ** dim


def _patch_flops(dim, p, cells, smoother, cycles, evaluate):
    """Flops of `cycles` local V-cycles (the first from zero) on a patch of `cells` cells, and of Evaluate."""
    flops = cells * _cell_flops(dim, p) * (1 if evaluate else 0)
    q, first = p, True
    while q > 1:
        # zero start: deg - 1 applies, the residual, deg applies after the coarse correction (Jacobi: 0, 1, 1)
        applies = (1 + 1 if smoother == "jacobi" else 2 + 1 + 3) * cycles + (cycles - 1 if first else 0)
        flops += cells * _cell_flops(dim, q) * applies
        if q // 2 >= 1:
            flops += cycles * 2 * cells * 2 * dim * (q + 1) ** dim * (q // 2 + 1)
        q, first = q // 2, False
    return flops


def _unstructured_counts(mesh, size):
    if mesh == "trisplit2d":
        return 2, 6 * size * size
    if mesh == "extruded":
        return 3, 6 * size * size * max(1, size // 2)
    return 3, 24 * size ** 3


def work(case):
    kind = case["kind"]
    if kind == "train":
        steps = case["epochs"] * (case["n"] // case["batch"])
        mults = 16 * 64 + 64 * 64 + 64 * 2
        return {"bytes": 4.0 * (18 * case["n"] + 4 * pmg.MLP_NPARAM), "flops": 6.0 * mults * case["batch"] * steps}
    if kind in ("usmooth", "batch"):
        specs = _batch_specs(case, 0) if kind == "batch" else [(case["mesh"], case["size"], case["p"], 0)]
        flops = bytes_ = 0.0
        for mesh, size, p, _ in specs:
            dim, cells = _unstructured_counts(mesh, size)
            # every cell belongs to at most 2^d patches; a fifth fewer next to the boundary of these small meshes
            visits = 0.8 * cells * 2 ** dim
            one = _patch_flops(dim, p, 1, case.get("smoother"), 1, True) * visits
            dofs = cells * p ** dim
            iterations = 12 if kind == "batch" else 0.5
            flops += 2 * iterations * one
            bytes_ += 24.0 * dofs + 8.0 * cells * (2 ** dim + 1)
        return {"bytes": bytes_, "flops": flops}
    dim, p, n = case["dim"], case["p"], case["n"]
    dofs, patches, cells = (p * n + 1) ** dim, (n - 1) ** dim, 2 ** dim
    mesh_bytes = 8.0 * (dim * (n + 1) ** dim + n ** dim)
    if kind == "local":
        ni = (2 * p - 1) ** dim
        return {"bytes": 16.0 * case["count"] * ni + mesh_bytes * min(1.0, case["count"] / patches),
                "flops": float(case["count"] * _patch_flops(dim, p, cells, case["smoother"], case["cycles"], False))}
    if kind == "smooth":
        return {"bytes": 24.0 * dofs + mesh_bytes,
                "flops": float(patches * _patch_flops(dim, p, cells, case["smoother"], 1, True))}
    if kind == "solve":
        iterations, sweep = 8, _patch_flops(dim, p, cells, "chebyshev", 1, True)
        coarse = 1.0 / (1.0 - 0.5 ** dim)
        return {"bytes": 16.0 * dofs + mesh_bytes,
                "flops": iterations * (2.0 * patches * sweep * coarse + 2.0 * n ** dim * _cell_flops(dim, p))}
    flops, q, total = 0.0, p, 0
    while q > 1:
        ni = (2 * q - 1) ** dim
        k = min(16, ni)
        flops += patches * (k * cells * _cell_flops(dim, q) + 4.0 * k * k * ni)
        total += 2 * patches
        q //= 2
    return {"bytes": mesh_bytes + 8.0 * total, "flops": flops / (1.0 - 0.5 ** dim)}


# ------------------------------------------------------------------ what the passes compute, in 64 bits
def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return (x + 1.0) / 2.0, w / 2.0


def _lobatto(q):
    inner = np.polynomial.legendre.Legendre.basis(q).deriv().roots() if q > 1 else np.zeros(0)
    return (np.concatenate([[-1.0], np.sort(inner.real), [1.0]]) + 1.0) / 2.0


def _lagrange(nodes, x):
    """Values and derivatives of the Lagrange basis on `nodes` at the points x: two [len(x)][len(nodes)] arrays."""
    m = len(nodes)
    val, der = np.ones((len(x), m)), np.zeros((len(x), m))
    for a in range(m):
        others = [b for b in range(m) if b != a]
        scale = np.prod([nodes[a] - nodes[b] for b in others])
        val[:, a] = np.prod([x - nodes[b] for b in others], axis=0) / scale
        for s in others:
            rest = [x - nodes[b] for b in others if b != s]
            der[:, a] += (np.prod(rest, axis=0) if rest else 1.0) / scale
    return val, der


def _splitmix(z):
    mask = (1 << 64) - 1
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
    return z ^ (z >> 31)


def _start_values(counters):
    """u of the Lanczos start vectors 1 + (u - 1/2) for an array of counters (seed 0)."""
    with np.errstate(over="ignore"):
        z = (counters.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


class _Mesh:
    """A conforming mesh with the Q_q spaces on it: plain dense tables and index arrays in 64 bits."""

    def __init__(self, coords, cells, kappa, dofs, patches, patch_ids, colours):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.dim = coords.shape[1]
        self.coords, self.cells, self.kappa = coords, cells, kappa
        self.dofs = dofs                      # q -> (cell DoFs [nc][(q+1)^d], number of DoFs, Dirichlet mask)
        self.patches = patches                # [np][valence], -1 padded
        self.patch_ids = patch_ids            # ids of the Lanczos counters
        self.colours = colours
        self.cache = {}

    def t(self, a):
        return torch.as_tensor(a, device=self.dev)

    def space(self, q):
        if q in self.cache:
            return self.cache[q]
        d, n = self.dim, q + 1
        gx, gw = _gauss(n)
        val, der = _lagrange(_lobatto(q), gx)
        s = {"B": self.t(val), "Bd": self.t(der)}
        grid = np.stack(np.meshgrid(*([np.arange(n)] * d), indexing="ij"), -1).reshape(-1, d)[:, ::-1]   # x fastest
        xi, w = gx[grid], gw[grid].prod(1)
        dn = np.ones((len(grid), 2 ** d, d))
        for v in range(2 ** d):
            for a in range(d):
                for k in range(d):
                    bit = (v >> k) & 1
                    dn[:, v, a] *= (1.0 if bit else -1.0) if k == a else (xi[:, k] if bit else 1.0 - xi[:, k])
        x = self.t(self.coords)[self.t(self.cells)]
        jac = torch.einsum("cvi,gva->cgia", x, self.t(dn))
        inv = torch.linalg.inv(jac)
        scale = self.t(w)[None, :] * self.t(self.kappa)[:, None] * torch.linalg.det(jac)
        s["G"] = torch.einsum("cgai,cgbi,cg->cgab", inv, inv, scale)
        cd, total, bnd = self.dofs(q)
        s["cd"], s["total"], s["bnd"] = self.t(cd), total, self.t(bnd)
        s["count"] = torch.bincount(s["cd"].reshape(-1), minlength=total)
        diag = torch.zeros(len(cd), n ** d, dtype=torch.float64, device=self.dev)
        for a in range(d):
            for b in range(d):
                y = s["G"][:, :, a, b].reshape(-1, *([n] * d))
                for ax in range(d):
                    m = s["Bd"] * s["Bd"] if a == b == ax else (s["B"] * s["Bd"] if ax in (a, b) else s["B"] * s["B"])
                    y = self.along(y, m.T, ax)
                diag += y.reshape(len(cd), -1)
        full = torch.zeros(total, dtype=torch.float64, device=self.dev).index_add_(0, s["cd"].reshape(-1), diag.reshape(-1))
        s["dinv"] = torch.where(s["bnd"], torch.zeros_like(full), 1.0 / full)
        if q > 1:
            s["E"] = self.t(_lagrange(_lobatto(q // 2), _lobatto(q))[0])
        self.cache[q] = s
        return s

    def along(self, y, m, axis):
        """m applied along reference axis `axis` (0 = x, the last array axis) of [cells][..z, y, x]."""
        k = y.dim() - 1 - axis
        return (y.movedim(k, -1) @ m.T).movedim(-1, k)

    def cell_apply(self, s, sel, v):
        d, n = self.dim, s["B"].shape[0]
        out = torch.empty_like(v)
        step = max(1, (1 << 24) // n ** d)
        for k in range(0, len(v), step):
            y = v[k:k + step].reshape(-1, *([n] * d))
            grad = []
            for a in range(d):
                g = y
                for ax in range(d):
                    g = self.along(g, s["Bd"] if ax == a else s["B"], ax)
                grad.append(g.reshape(len(g), -1))
            flux = torch.einsum("cgab,cgb->cga", s["G"][sel[k:k + step]], torch.stack(grad, -1))
            res = 0.0
            for a in range(d):
                f = flux[..., a].reshape(y.shape)
                for ax in range(d):
                    f = self.along(f, (s["Bd"] if ax == a else s["B"]).T, ax)
                res = res + f.reshape(len(f), -1)
            out[k:k + step] = res
        return out

    def view(self, q, chosen):
        """The interiors of the patches `chosen` (which share no cell) at degree q."""
        s = self.space(q)
        pc = self.patches[chosen]
        where, slot = np.nonzero(pc >= 0)
        cells, owner = self.t(pc[where, slot].astype(np.int64)), self.t(where.astype(np.int64))
        cd = s["cd"][cells]
        flat, own = cd.reshape(-1), owner[:, None].expand_as(cd).reshape(-1)
        count = torch.bincount(flat, minlength=s["total"])
        low = torch.full((s["total"],), 1 << 40, device=self.dev, dtype=torch.int64).scatter_reduce_(0, flat, own, "amin")
        high = torch.full((s["total"],), -1, device=self.dev, dtype=torch.int64).scatter_reduce_(0, flat, own, "amax")
        inside = (count == s["count"]) & (count > 0) & (low == high) & ~s["bnd"]
        return {"s": s, "q": q, "cells": cells, "cd": cd, "inside": inside.double(), "mask": inside, "count": count,
                "owner": torch.where(inside, low, torch.zeros_like(low)), "n": len(chosen), "chosen": chosen}

    def apply(self, w, v):
        y = self.cell_apply(w["s"], w["cells"], v[w["cd"]])
        out = torch.zeros_like(v).index_add_(0, w["cd"].reshape(-1), y.reshape(-1))
        return out * w["inside"]

    def ritz(self, w, steps=16):
        """(theta_min, theta_max) of every patch of the view after `steps` Lanczos steps."""
        ids = torch.nonzero(w["mask"]).reshape(-1)
        own = w["owner"][ids]
        order = torch.argsort(own, stable=True)
        ids, own = ids[order], own[order]
        size = torch.bincount(own, minlength=w["n"])
        rank = torch.arange(len(ids), device=self.dev) - (torch.cumsum(size, 0) - size)[own]
        pid = self.patch_ids[w["chosen"]][own.cpu().numpy()].astype(np.uint64)
        ctr = (pid << np.uint64(20)) | np.uint64(w["q"] << 16) | rank.cpu().numpy().astype(np.uint64)
        v = 1.0 + (self.t(_start_values(ctr)) - 0.5)
        root = torch.sqrt(w["s"]["dinv"][ids])
        dot = lambda a, b: torch.zeros(w["n"], dtype=torch.float64, device=self.dev).index_add_(0, own, a * b)
        v = v / torch.sqrt(dot(v, v))[own]
        basis, al, be = [], [], []
        for _ in range(steps):
            basis.append(v)
            x = torch.zeros(w["s"]["total"], dtype=torch.float64, device=self.dev)
            x[ids] = root * v
            y = root * self.apply(w, x)[ids]
            al.append(dot(v, y))
            for _ in range(2):
                coef = [dot(z, y) for z in basis]
                for c, z in zip(coef, basis):
                    y = y - c[own] * z
            b = torch.sqrt(dot(y, y))
            be.append(b)
            v = y / torch.clamp(b, min=1e-300)[own]
        k = torch.clamp(size, max=steps)[:, None]
        al, be = torch.stack(al, 1), torch.stack(be, 1)[:, :-1]
        at = torch.arange(steps, device=self.dev)[None]
        al = torch.where(at < k, al, al[:, :1])
        be = torch.where(at[:, 1:] < k, be, torch.zeros_like(be))
        ev = torch.linalg.eigvalsh(torch.diag_embed(al) + torch.diag_embed(be, 1) + torch.diag_embed(be, -1))
        return ev[:, 0], ev[:, -1]

    def smooth(self, w, d, r, smoother, degree=3):
        dinv = w["s"]["dinv"] * w["inside"]
        if smoother == "jacobi":
            return 0.5 * dinv * r if d is None else d + 0.5 * dinv * (r - self.apply(w, d))
        if "theta" not in w:
            lo, hi = self.ritz(w)
            hi = 1.1 * hi
            lo = torch.maximum(lo, hi / 10.0)
            w["theta"], w["delta"] = ((hi + lo) / 2)[w["owner"]], ((hi - lo) / 2)[w["owner"]]
        theta, delta = w["theta"], w["delta"]
        res = dinv * (r if d is None else r - self.apply(w, d))
        step = res / theta
        d = step if d is None else d + step
        sigma = theta / delta
        rho = 1.0 / sigma
        for _ in range(1, degree):
            nxt = 1.0 / (2.0 * sigma - rho)
            res = res - dinv * self.apply(w, step)
            step = nxt * rho * step + 2.0 * nxt / delta * res
            d = d + step
            rho = nxt
        return d

    def transfer(self, w, wc, v, up):
        """The embedding of the next coarser p-level (up) or its transpose, per cell."""
        e = w["s"]["E"]
        if up:
            y = (v * wc["inside"])[wc["cd"]].reshape(-1, *([e.shape[1]] * self.dim))
            for ax in range(self.dim):
                y = self.along(y, e, ax)
            out = torch.zeros(w["s"]["total"], dtype=torch.float64, device=self.dev)
            out[w["cd"].reshape(-1)] = y.reshape(-1)
            return out * w["inside"]
        share = v * w["inside"] / torch.clamp(w["count"], min=1)
        y = share[w["cd"]].reshape(-1, *([e.shape[0]] * self.dim))
        for ax in range(self.dim):
            y = self.along(y, e.T, ax)
        out = torch.zeros(wc["s"]["total"], dtype=torch.float64, device=self.dev)
        return out.index_add_(0, wc["cd"].reshape(-1), y.reshape(-1)) * wc["inside"]

    def vcycle(self, views, k, d, r, smoother):
        w = views[k]
        if w["q"] == 1:
            return r * w["s"]["dinv"] * w["inside"]
        d = self.smooth(w, d, r, smoother)
        rc = self.transfer(w, views[k + 1], r - self.apply(w, d), False)
        d = d + self.transfer(w, views[k + 1], self.vcycle(views, k + 1, None, rc, smoother), True)
        return self.smooth(w, d, r, smoother)

    def views(self, p, chosen):
        out = []
        while p >= 1:
            out.append(self.view(p, chosen))
            p //= 2
        return out

    def sweep(self, p, b, u, smoother):
        b, u = self.t(b), self.t(u)
        u = torch.where(self.space(p)["bnd"], torch.zeros_like(u), u)
        for c in range(int(self.colours.max()) + 1):
            views = self.views(p, np.nonzero(self.colours == c)[0])
            r = (b - self.apply(views[0], u)) * views[0]["inside"]
            u = u + self.vcycle(views, 0, None, r, smoother)
        return u

    def local(self, p, ids, r, smoother, cycles):
        r = self.t(r)
        out = torch.zeros_like(r)
        for c in range(int(self.colours.max()) + 1):
            rows = np.nonzero(self.colours[ids] == c)[0]
            if not len(rows):
                continue
            views = self.views(p, ids[rows])
            w = views[0]
            at = torch.nonzero(w["mask"]).reshape(-1)
            at = at[torch.argsort(w["owner"][at], stable=True)].reshape(len(rows), -1)
            rhs = torch.zeros(w["s"]["total"], dtype=torch.float64, device=self.dev)
            rows = self.t(rows)
            rhs[at.reshape(-1)] = r[rows].reshape(-1)
            d = None
            for _ in range(cycles):
                d = self.vcycle(views, 0, d, rhs, smoother)
            out[rows] = d[at]
        return out

    def solve(self, p, b, tol=1e-13):
        """Diagonally preconditioned CG on the whole mesh."""
        s = self.space(p)
        every = torch.arange(len(self.cells), device=self.dev)
        free = (~s["bnd"]).double()

        def a(v):
            y = self.cell_apply(s, every, v[s["cd"]])
            return torch.zeros_like(v).index_add_(0, s["cd"].reshape(-1), y.reshape(-1)) * free

        r = self.t(b) * free
        x, z = torch.zeros_like(r), r * s["dinv"]
        d, rz, stop = z, torch.dot(r, z), tol * float(torch.linalg.norm(r))
        for it in range(4000):
            q = a(d)
            alpha = rz / torch.dot(d, q)
            x, r = x + alpha * d, r - alpha * q
            if it % 20 == 0 and float(torch.linalg.norm(r)) <= stop:
                break
            z = r * s["dinv"]
            rz, old = torch.dot(r, z), rz
            d = z + (rz / old) * d
        return x


def _structured_mesh(dim, n, coords, kappa):
    grid = lambda m: np.stack(np.meshgrid(*([np.arange(m)] * dim), indexing="ij"), -1).reshape(-1, dim)[:, ::-1]
    index = lambda g, m: (g * m ** np.arange(dim)).sum(-1)
    corners = np.array([[(v >> a) & 1 for a in range(dim)] for v in range(2 ** dim)])
    cell = grid(n)

    def dofs(q):
        m = q * n + 1
        every = grid(m)
        return (index(q * cell[:, None] + grid(q + 1)[None], m), m ** dim,
                ((every == 0) | (every == m - 1)).any(1))

    vertex = grid(n - 1) + 1
    return _Mesh(coords, index(cell[:, None] + corners[None], n + 1), kappa, dofs,
                 index(vertex[:, None] - 1 + corners[None], n), np.arange(len(vertex)),
                 ((vertex & 1) << np.arange(dim)).sum(1))


def _unstructured_mesh(coords, cells, bnd, kappa):
    """The library's documented numbering: vertices, edges, faces, cell interiors; greedy colours."""
    dim, nc, nv = coords.shape[1], len(cells), len(coords)
    bit = lambda c, a: (c >> a) & 1
    edges = [(c, c | 1 << a, a) for a in range(dim) for c in range(2 ** dim) if not bit(c, a)]
    faces = [(c, a, b) for a in range(dim) for b in range(a + 1, dim) for c in range(2 ** dim)
             if not bit(c, a) and not bit(c, b)] if dim == 3 else []
    ekey = np.concatenate([np.sort(cells[:, [i, j]], 1) for i, j, _ in edges])
    eu, eid = np.unique(ekey, axis=0, return_inverse=True)
    eid = eid.reshape(len(edges), nc)
    fcorner = lambda c, a, b: [c, c | 1 << a, c | 1 << b, c | 1 << a | 1 << b]
    fu, fid = np.zeros((0, 4)), np.zeros((0, nc), dtype=np.int64)
    if faces:
        fu, fid, times = np.unique(np.concatenate([np.sort(cells[:, fcorner(*f)], 1) for f in faces]), axis=0,
                                   return_inverse=True, return_counts=True)
        fid = fid.reshape(len(faces), nc)
        fbnd = times == 1
        ebnd = np.zeros(len(eu), dtype=bool)
        number = {(i, j): k for k, (i, j, _) in enumerate(edges)}
        for k, f in enumerate(faces):
            on = fbnd[fid[k]]
            i, j, l, m = fcorner(*f)
            for pair in ((i, j), (l, m), (i, l), (j, m)):
                ebnd[eid[number[pair]][on]] = True
    else:
        fbnd, ebnd = np.zeros(0, dtype=bool), np.bincount(eid.reshape(-1), minlength=len(eu)) == 1

    def dofs(q):
        m, n = q - 1, q + 1
        e0 = nv
        f0 = e0 + len(eu) * m
        c0 = f0 + len(fu) * m * m
        node = np.stack(np.meshgrid(*([np.arange(n)] * dim), indexing="ij"), -1).reshape(-1, dim)[:, ::-1]
        local = lambda mi: int((np.asarray(mi) * n ** np.arange(dim)).sum())
        out = np.zeros((nc, n ** dim), dtype=np.int64)
        for c in range(2 ** dim):
            out[:, local([q * bit(c, a) for a in range(dim)])] = cells[:, c]
        for k, (i, j, a) in enumerate(edges):
            for t in range(1, q):
                at = [q * bit(i, x) for x in range(dim)]
                at[a] = t
                out[:, local(at)] = e0 + eid[k] * m + np.where(cells[:, i] < cells[:, j], t, q - t) - 1
        for k, (c, a, b) in enumerate(faces):
            ids = cells[:, fcorner(c, a, b)]                                # corner bits (along a, along b)
            low = ids.argmin(1)
            first = ids[np.arange(nc), low ^ 1] < ids[np.arange(nc), low ^ 2]
            for s in range(1, q):
                for t in range(1, q):
                    sa, tb = np.where(low & 1, q - s, s), np.where(low & 2, q - t, t)
                    at = [q * bit(c, x) for x in range(3)]
                    at[a], at[b] = s, t
                    out[:, local(at)] = (f0 + fid[k] * m * m + np.where(first, sa, tb) - 1
                                         + m * (np.where(first, tb, sa) - 1))
        inner = node[((node > 0) & (node < q)).all(1)]
        for i, mi in enumerate(inner):
            out[:, local(mi)] = c0 + np.arange(nc) * m ** dim + i
        total = c0 + nc * m ** dim
        mask = np.zeros(total, dtype=bool)
        mask[:nv] = bnd != 0
        mask[e0:f0] = np.repeat(ebnd, m)
        mask[f0:c0] = np.repeat(fbnd, m * m)
        return out, total, mask

    around = [[] for _ in range(nv)]
    for c, vs in enumerate(cells.tolist()):
        for v in vs:
            around[v].append(c)
    centre = np.nonzero(bnd == 0)[0]
    patches = np.full((len(centre), max(len(around[v]) for v in centre)), -1, dtype=np.int64)
    for j, v in enumerate(centre):
        patches[j, :len(around[v])] = sorted(around[v])
    colours, used = np.zeros(len(centre), dtype=np.int64), [set() for _ in range(nc)]
    for j in sorted(range(len(centre)), key=lambda j: (_splitmix(int(centre[j])), int(centre[j])), reverse=True):
        taken = set().union(*(used[c] for c in around[centre[j]]))
        colours[j] = next(c for c in range(len(taken) + 1) if c not in taken)
        for c in around[centre[j]]:
            used[c].add(colours[j])
    return _Mesh(coords, cells, kappa, dofs, patches, centre, colours)


def _exact_train(case, seed):
    """Adam on the whole set per step (batch = n: the shuffled order does not matter)."""
    if case["batch"] < case["n"]:
        return None
    x, t = _train_inputs(case, seed)
    mean = lambda a: a.astype(np.float64).mean(0).astype(np.float32)
    std = lambda a: (a.astype(np.float64).std(0) + 1e-6).astype(np.float32)
    x = torch.tensor((x.astype(np.float64) - mean(x)) / std(x))
    t = torch.tensor((t.astype(np.float64) - mean(t)) / std(t))
    rows, cols = (64, 64, 2), (16, 64, 64)
    theta = torch.tensor(pmg.mlp_init(seed).astype(np.float64))          # the start parameters are an input
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    lr, eps = float(np.float32(2e-3)), float(np.float32(1e-8))
    m, v, losses = torch.zeros_like(theta), torch.zeros_like(theta), []
    for step in range(1, case["epochs"] + 1):
        w = theta.clone().requires_grad_(True)
        h, o = x, 0
        for k, (r, c) in enumerate(zip(rows, cols)):
            h = h @ w[o:o + r * c].reshape(r, c).T + w[o + r * c:o + r * c + r]
            o += r * c + r
            h = torch.relu(h) if k < 2 else h
        e = h - t
        weight = torch.ones_like(e)
        weight[:, 0] = torch.where(e[:, 0] < 0, 4.0, 1.0)
        loss = (0.5 * weight.detach() * e * e).sum() / len(x)
        g, = torch.autograd.grad(loss, w)
        losses.append(float(loss))
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        theta = theta - lr * (m / (1 - b1 ** step)) / (torch.sqrt(v / (1 - b2 ** step)) + eps)
    return theta, np.array(losses)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None                                           # several unpreconditioned solves: minutes
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "usmooth":
        coords, cells, bnd, kappa = _unstructured_inputs(case["mesh"], case["size"], case["p"], case["decades"], seed)
        mesh = _unstructured_mesh(coords, cells, bnd, kappa)
        total, free = mesh.dofs(case["p"])[1:]
        b, u0 = _vectors(total, seed)
        u = mesh.sweep(case["p"], b, u0, case["smoother"])
        # Dirichlet entries of the caller's vector stay as they were
        return torch.where(mesh.t(free), mesh.t(u0), u)
    dim, p, n = case["dim"], case["p"], case["n"]
    coords, kappa, b, u, ids, r = _structured_inputs(case, seed)
    if kind == "lanczos":
        out, levels = [None] * _levels(n), _levels(n)
        for level in range(levels - 1, -1, -1):
            mesh = _structured_mesh(dim, n, coords, kappa)
            degrees = [p >> k for k in range(p.bit_length())]
            ritz = torch.zeros(len(mesh.patches), len(degrees), 2, dtype=torch.float64, device=mesh.dev)
            for c in range(2 ** dim):
                chosen = np.nonzero(mesh.colours == c)[0]
                for k, q in enumerate(degrees):
                    if q > 1 and len(chosen):
                        ritz[mesh.t(chosen), k] = torch.stack(mesh.ritz(mesh.view(q, chosen)), 1)
            out[level] = ritz
            if level:
                coords = coords.reshape(*([n + 1] * dim), dim)[(slice(None, None, 2),) * dim].reshape(-1, dim)
                split = sum(([n // 2, 2] for _ in range(dim)), [])
                kappa = kappa.reshape(split).mean(axis=tuple(range(1, 2 * dim, 2))).reshape(-1)
                n //= 2
        return out
    mesh = _structured_mesh(dim, n, coords, kappa)
    if kind == "smooth":
        return mesh.sweep(p, b, u, case["smoother"])
    if kind == "local":
        return mesh.local(p, ids, r, case["smoother"], case["cycles"])
    return mesh.solve(p, b) if case["decades"] == 0.0 else None
