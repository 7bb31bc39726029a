"""Kernels at the sizes where their tiling changes: ragged tiles of the training
kernel, few Lanczos steps, and unstructured colours of a few to many patches."""
import numpy as np
import pytest

from oracle import fem, lanczos as lz, mlp, patch as pt, unstructured as us
from paper_2510_17785_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(x, dtype=torch.float64):
    return torch.tensor(np.asarray(x), dtype=dtype, device="cuda")


@pytest.mark.parametrize("n", [1, 7, 8, 9, 33, 2432, 2433, 5001])
def test_training_gradient_at_tile_edges(n):
    """Tiles of 8 samples, 304 CTAs: the gradient within 1e-4 (FP32 sums of at
    most a few hundred terms, unit roundoff 6e-8), the loss within 1e-5."""
    from paper_2510_17785_gb300 import pmg
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 16)).astype(np.float32).astype(np.float64)
    T = rng.standard_normal((n, 2)).astype(np.float32).astype(np.float64)
    norm = np.concatenate([np.full(16, 0.25), np.full(16, 2.0), np.full(2, -0.5), np.full(2, 1.5)])
    theta = mlp.init_params(5).astype(np.float32).astype(np.float64)
    f32 = torch.float32
    loss, g = pmg.mlp_grad(dev(theta, f32), dev(norm, f32), dev(X, f32), dev(T, f32), asym=4.0)
    Xs, Ts = (X - 0.25) / 2.0, (T + 0.5) / 1.5
    ref_g, ref_l = mlp.grad(theta, Xs, Ts, 4.0), mlp.loss(theta, Xs, Ts, 4.0)
    assert abs(float(loss.item()) - ref_l) <= 1e-5 * ref_l
    assert np.linalg.norm(g.cpu().numpy() - ref_g) <= 1e-4 * np.linalg.norm(ref_g)


@pytest.mark.parametrize("steps", [1, 2, 9, 40])
def test_lanczos_with_few_and_many_steps(steps):
    """One step (a 1 x 1 tridiagonal matrix) up to more steps than the small
    p-levels have DoFs; 1e-9 of theta_max, as at 16 steps."""
    from paper_2510_17785_gb300 import pmg
    w = inputs.Workload("lz", 2, 4, 4, 0.2, "uniform", ("loguniform", -1, 1), "uniform", 7)
    prob = inputs.make_problem(w)
    ctx = pmg.Context(0, bounds=pmg.BOUNDS_LANCZOS, lanczos_steps=steps, seed=2)
    ctx.mesh_structured(2, 4, 4, 1, prob.coords, prob.kappa)
    ctx.setup()
    ritz = ctx.get_ritz(0)
    m = fem.StructuredMesh(2, 4, prob.coords, prob.kappa)
    for v in pt.interior_vertices(2, 4):
        j = pt.patch_id(2, 4, v)
        P = pt.Patch(m, v, [4, 2, 1])
        for k, q in enumerate((4, 2)):
            _, _, tmin, tmax = lz.patch_bounds(P.lv[q].A, P.lv[q].diag, 2, j, q, k=steps)
            assert abs(ritz[j, k, 0] - tmin) <= 1e-9 * tmax and abs(ritz[j, k, 1] - tmax) <= 1e-9 * tmax, (j, q)
    ctx.close()


@pytest.mark.parametrize("size,p,precision,kind", [(1, 4, "fp64", "chebyshev"), (2, 6, "mixed", "jacobi"),
                                                   (4, 5, "mixed", "chebyshev"), (4, 4, "fp64", "chebyshev")])
def test_shared_patches_equal_local_solves(size, p, precision, kind):
    """With u = 0 a colour's sweep adds every patch's local solve of b: equal up
    to rounding for the largest, the smallest and a middle colour (one CTA per
    patch in both; the same launch size, so the same place of the workspace)."""
    from paper_2510_17785_gb300 import pmg
    P, T = inputs.cube_tetrahedra(size, 13)
    X, C = inputs.tetrahedra_to_hexes(P, T)
    kappa = 10.0 ** np.random.default_rng(1).uniform(-1, 1, len(C))
    ctx = pmg.Context(0, bounds=pmg.BOUNDS_FIXED, fixed_lo=0.25, fixed_hi=2.2,
                      precision=pmg.PREC_MIXED if precision == "mixed" else pmg.PREC_FP64,
                      smoother=pmg.SMOOTHER_JACOBI if kind == "jacobi" else pmg.SMOOTHER_CHEBYSHEV)
    ctx.mesh_upload(3, X, C, p, kappa=kappa)
    ctx.setup()
    m = us.Mesh(3, X, C, kappa)
    verts = m.interior_vertices()
    cd = m.cell_dofs(p)
    bnd = m.boundary_dofs(p)
    count = np.bincount(np.asarray(cd).reshape(-1), minlength=len(bnd))
    b = np.random.default_rng(9).uniform(-1, 1, len(bnd)) * ~bnd
    colours = ctx.get_colours(0)
    sizes = np.bincount(colours)
    ni = ctx.local_size(0)
    for c in sorted({int(sizes.argmax()), int(sizes.argmin()), int(np.argsort(sizes)[len(sizes) // 2])}):
        u = torch.zeros(len(bnd), dtype=torch.float64, device="cuda")
        ctx.patch_smooth_colour(0, c, dev(b), u)
        u = u.cpu().numpy()
        ids = np.nonzero(colours == c)[0].astype(np.int64)
        interior, r = [], np.zeros((len(ids), ni))
        for i, j in enumerate(ids):
            g, k = np.unique(np.asarray([cd[x] for x in m.vertex_cells[verts[int(j)]]]).reshape(-1), return_counts=True)
            g = g[(k == count[g]) & ~bnd[g]]
            interior.append(g)
            r[i, :len(g)] = b[g]
        d = torch.empty(len(ids) * ni, dtype=torch.float64, device="cuda")
        ctx.local_vcycle(0, torch.tensor(ids, device="cuda"), dev(r.reshape(-1)), d, 1)
        d = d.cpu().numpy().reshape(len(ids), ni)
        ref = np.zeros(len(bnd))
        for i, g in enumerate(interior):
            ref[g] += d[i, :len(g)]
        assert np.abs(u - ref).max() <= (1e-12 if precision == "fp64" else 1e-5) * np.abs(ref).max(), c
    ctx.close()
