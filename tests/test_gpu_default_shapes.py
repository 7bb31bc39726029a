"""FP32 default launch shapes that give a patch its own warps (2D from degree
3, 3D degree 2) against the FP64 oracle: sweeps, additive sweeps and local
solves with every smoother, and BF16 geometry, with patch counts that leave
the last CTA short (colours of 4, 6 and 9 patches, 7 local solves).  The
launches that keep the one-team form instead: the same bits.

Tolerance: a sweep applies an operator about 20 times, each a handful of
contractions of at most 9 terms, so rounding errors of 6e-8 add up to some 30
of them, times the interval ratio of about 10: 2e-5.  The Cartesian-reinforced
smoother applies a patch inverse, whose condition (some hundreds at degree 8)
takes the place of that ratio: 2e-4.  BF16 geometry: 5e-5, the bound of its
other sweeps."""
import dataclasses

import numpy as np
import pytest

from oracle import fem, lanczos as lz, patch as pt
from paper_2510_17785_gb300 import inputs
from test_gpu_geometry_bf16 import _bf16_element, _bf16_smoother, _dense_level

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LO, HI = 0.25, 2.2
SHAPES = [(2, 6, 3), (2, 6, 4), (2, 6, 5), (2, 6, 6), (2, 6, 7), (2, 6, 8), (3, 4, 2)]
KINDS = ["chebyshev", "jacobi", "fdm"]


def _problem(dim, N, p, kind="chebyshev", **opt):
    from paper_2510_17785_gb300 import pmg
    sm = {"jacobi": pmg.SMOOTHER_JACOBI, "fdm": pmg.SMOOTHER_CARTESIAN}.get(kind, pmg.SMOOTHER_CHEBYSHEV)
    w = inputs.Workload(f"s{dim}_{p}", dim, N, p, 0.2, "uniform", ("loguniform", -1.0, 1.0), "uniform", 50 + p)
    prob = inputs.make_problem(w)
    ctx = pmg.Context(0, precision=pmg.PREC_MIXED, bounds=pmg.BOUNDS_FIXED, fixed_lo=LO, fixed_hi=HI, smoother=sm,
                      **opt)
    ctx.mesh_structured(dim, N, p, 1, prob.coords, prob.kappa)
    ctx.setup()
    return ctx, prob, fem.StructuredMesh(dim, N, prob.coords, prob.kappa)


def _sweep_error(ctx, prob, dim, N, p, smoother, reverse):
    u0 = inputs.random_vector(8, dim, p, N)
    u = torch.tensor(u0, device="cuda")
    ctx.patch_smooth(0, torch.tensor(prob.rhs, device="cuda"), u, 1, reverse)
    ref = smoother.sweep(u0, prob.rhs, reverse=reverse)
    return np.abs(u.cpu().numpy() - ref).max() / np.abs(ref).max()


def _tol(kind):
    return 2e-4 if kind == "fdm" else 2e-5


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("dim,N,p", SHAPES)
def test_sweep(dim, N, p, kind):
    ctx, prob, m = _problem(dim, N, p, kind)
    S = pt.PatchSmoother(m, p, sm=pt.Smoother(kind=kind), bounds_fn=lz.fixed_bounds_fn(LO, HI))
    assert _sweep_error(ctx, prob, dim, N, p, S, p % 2 == 1) < _tol(kind)
    ctx.close()


@pytest.mark.parametrize("dim,N,p", SHAPES)
def test_additive_sweep(dim, N, p):
    ctx, prob, m = _problem(dim, N, p, additive=1, additive_theta=0.7)
    S = pt.PatchSmoother(m, p, bounds_fn=lz.fixed_bounds_fn(LO, HI), additive=True, theta=0.7)
    assert _sweep_error(ctx, prob, dim, N, p, S, False) < _tol("chebyshev")
    ctx.close()


@pytest.mark.parametrize("dim,N,p", [s for s in SHAPES if s[2] != 5])
def test_bf16_geometry_sweep(dim, N, p):
    ctx, prob, m = _problem(dim, N, p, geometry_bf16=1)
    S = _bf16_smoother(m, p, lz.fixed_bounds_fn(LO, HI))
    if _dense_level(dim, p):
        # the level's dense operator is exact, the residual of u is not
        B = pt.PatchSmoother(m, p, bounds_fn=lz.fixed_bounds_fn(LO, HI), element_fn=_bf16_element)
        for v in S.vertices:
            P = S.patch(v)
            P.lv[p] = dataclasses.replace(P.lv[p], A_ic=B.patch(v).lv[p].A_ic)
    assert _sweep_error(ctx, prob, dim, N, p, S, False) < 5e-5
    ctx.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("dim,N,p", SHAPES)
def test_local_solves(dim, N, p, kind):
    ctx, prob, m = _problem(dim, N, p, kind)
    ids = inputs.sample_patches(17, (N - 1) ** dim, 7)
    ni = (2 * p - 1) ** dim
    r = np.random.default_rng(4).uniform(-1, 1, (len(ids), ni))
    d = torch.zeros(r.shape, dtype=torch.float64, device="cuda")
    ctx.local_vcycle(0, torch.tensor(ids, device="cuda"), torch.tensor(r, device="cuda"), d, 2)
    d = d.cpu().numpy()
    byid = {pt.patch_id(dim, N, v): v for v in pt.interior_vertices(dim, N)}
    for i, j in enumerate(ids):
        P = pt.Patch(m, byid[int(j)], pt.levels_halving(p))
        ref = pt.local_solve(P, r[i], pt.Smoother(kind=kind), lz.fixed_bounds_fn(LO, HI)(P, int(j)), 2)
        assert np.abs(d[i] - ref).max() < _tol(kind) * np.abs(ref).max(), j
    ctx.close()


@pytest.mark.parametrize("dim,N,p,precision,kind,together", [
    (2, 52, 8, "mixed", "fdm", False), (2, 24, 7, "mixed", "fdm", True), (2, 44, 5, "mixed", "fdm", True),
    (2, 24, 8, "mixed", "jacobi", False), (3, 11, 2, "fp64", "chebyshev", True), (3, 14, 2, "fp64", "jacobi", True),
    (3, 11, 2, "fp64", "fdm", True)])
def test_local_solves_in_either_form(dim, N, p, precision, kind, together):
    """All patches of a mesh in one launch against launches of at most 60: on
    152 SMs one of the two takes the team (the one launch where `together`)."""
    from paper_2510_17785_gb300 import pmg
    levels = 3 if N % 4 == 0 else 2 if N % 2 == 0 else 1
    sm = {"jacobi": pmg.SMOOTHER_JACOBI, "fdm": pmg.SMOOTHER_CARTESIAN}.get(kind, pmg.SMOOTHER_CHEBYSHEV)
    w = inputs.Workload("e", dim, N, p, 0.2, "uniform", ("loguniform", -1.0, 1.0), "uniform", 50 + p)
    prob = inputs.make_problem(w)
    ctx = pmg.Context(0, precision=pmg.PREC_MIXED if precision == "mixed" else pmg.PREC_FP64, smoother=sm,
                      bounds=pmg.BOUNDS_FIXED, fixed_lo=LO, fixed_hi=HI, autotune=0)
    ctx.mesh_structured(dim, N, p, levels, prob.coords, prob.kappa)
    ctx.setup()
    n, ni = (N - 1) ** dim, (2 * p - 1) ** dim
    ids = torch.arange(n, device="cuda")
    r = torch.rand((n, ni), dtype=torch.float64, generator=torch.Generator().manual_seed(4)).cuda() - 0.5
    one, parts = torch.zeros_like(r), torch.zeros_like(r)
    ctx.local_vcycle(levels - 1, ids, r, one, 2)
    for k in range(0, n, 60):
        ctx.local_vcycle(levels - 1, ids[k:k + 60], r[k:k + 60], parts[k:k + 60], 2)
    assert one.abs().max() > 0 and torch.equal(one, parts)
    ctx.close()


@pytest.mark.parametrize("dim,N,p,precision,kind", [
    (2, 11, 5, "mixed", "chebyshev"), (2, 11, 7, "mixed", "fdm"), (2, 11, 8, "mixed", "jacobi"),
    (2, 72, 3, "mixed", "chebyshev"), (3, 20, 2, "fp64", "chebyshev")])
def test_persistent_sweep_in_team_form(dim, N, p, precision, kind):
    """A persistent sweep that takes the team against one launch per colour that does not."""
    from paper_2510_17785_gb300 import pmg
    sm = {"jacobi": pmg.SMOOTHER_JACOBI, "fdm": pmg.SMOOTHER_CARTESIAN}.get(kind, pmg.SMOOTHER_CHEBYSHEV)
    levels = 3 if N % 4 == 0 else 1
    w = inputs.Workload("e", dim, N, p, 0.2, "uniform", ("loguniform", -1.0, 1.0), "uniform", 50 + p)
    prob = inputs.make_problem(w)
    out = []
    for persistent in (0, 2):
        ctx = pmg.Context(0, precision=pmg.PREC_MIXED if precision == "mixed" else pmg.PREC_FP64, smoother=sm,
                          bounds=pmg.BOUNDS_FIXED, fixed_lo=LO, fixed_hi=HI, autotune=0, dense_local=0,
                          persistent=persistent)
        ctx.mesh_structured(dim, N, p, levels, prob.coords, prob.kappa)
        ctx.setup()
        u = torch.tensor(inputs.random_vector(8, dim, p, N), device="cuda")
        ctx.patch_smooth(levels - 1, torch.tensor(prob.rhs, device="cuda"), u, 2, True)
        out.append(u)
        ctx.close()
    assert torch.equal(*out)
