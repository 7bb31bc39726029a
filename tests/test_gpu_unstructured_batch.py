"""Unstructured patches with their workspace in shared memory and in global
memory (which of the two a launch uses depends on its patch count and on the
other problems of a batch): the same operations in the same order, so the same
bits."""
import numpy as np
import pytest

from paper_2510_17785_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _context(kind, size, p, seed, **opt):
    from paper_2510_17785_gb300 import pmg
    X, cells, bnd = inputs.unstructured_mesh(kind, size, 13)
    kappa = 10.0 ** np.random.default_rng(seed).uniform(-2, 2, len(cells))
    ctx = pmg.Context(0, **opt)
    ctx.mesh_upload(X.shape[1], X, cells, p, bnd, kappa)
    ctx.setup()
    return ctx


@pytest.mark.parametrize("precision,p,kind", [("mixed", 6, "chebyshev"), ("mixed", 6, "jacobi"),
                                              ("fp64", 5, "chebyshev"), ("fp64", 4, "chebyshev")])
def test_local_solves_with_either_workspace(precision, p, kind):
    """Split tetrahedra at these degrees: 126 to 200 KB per patch, one CTA per
    SM.  All patches in one launch (more than the GPU has SMs: global memory)
    against the same patches in launches of at most 100 (shared memory)."""
    from paper_2510_17785_gb300 import pmg
    ctx = _context("tetsplit", 3, p, 1, bounds=pmg.BOUNDS_FIXED, fixed_lo=0.25, fixed_hi=2.2,
                   precision=pmg.PREC_MIXED if precision == "mixed" else pmg.PREC_FP64,
                   smoother=pmg.SMOOTHER_JACOBI if kind == "jacobi" else pmg.SMOOTHER_CHEBYSHEV)
    n, ni = ctx.num_patches(0)[0], ctx.local_size(0)
    assert n > torch.cuda.get_device_properties(0).multi_processor_count > 100
    ids = torch.randperm(n, generator=torch.Generator().manual_seed(3)).cuda()
    r = torch.rand((n, ni), dtype=torch.float64, generator=torch.Generator().manual_seed(4)).cuda() - 0.5
    together, apart = torch.zeros_like(r), torch.zeros_like(r)
    ctx.local_vcycle(0, ids, r, together, 2)
    for k in range(0, n, 100):
        d = torch.zeros_like(r[k:k + 100])
        ctx.local_vcycle(0, ids[k:k + 100].contiguous(), r[k:k + 100].contiguous(), d, 2)
        apart[k:k + 100] = d
    assert together.abs().max() > 0 and torch.equal(together, apart)
    ctx.close()


def test_batches_and_single_solves_in_turn():
    """Six problems, four with patches that want an SM: alone, together, in
    part and alone again, bit for bit."""
    from paper_2510_17785_gb300 import pmg
    specs = [("tetsplit", 2, 6), ("tetsplit", 1, 2), ("tetsplit", 1, 6), ("trisplit2d", 4, 8), ("tetsplit", 2, 6),
             ("extruded", 4, 7)]
    ctxs = [_context(k, s, p, i, bounds=pmg.BOUNDS_LANCZOS, precision=pmg.PREC_MIXED)
            for i, (k, s, p) in enumerate(specs)]
    bs = [torch.tensor(np.random.default_rng(i).uniform(-1, 1, c.num_dofs(0)[0]), device="cuda")
          for i, c in enumerate(ctxs)]

    def alone():
        out = []
        for c, b in zip(ctxs, bs):
            x = torch.zeros_like(b)
            out.append((*c.solve_cg(b, x, 1e-8, 200)[:2], x))
        return out

    def together(n):
        xs = [torch.full_like(b, 7.0) for b in bs[:n]]
        its, rels, _ = pmg.batch_solve_cg(ctxs[:n], bs[:n], xs, 1e-8, 200)
        return list(zip(its, rels, xs))

    ref = alone()
    assert all(rel <= 1e-8 for _, rel, _ in ref)
    for run in (lambda: together(6), lambda: together(3), alone, lambda: together(6)):
        for (it, rel, x), (it0, rel0, x0) in zip(run(), ref):
            assert it == it0 and rel == rel0 and torch.equal(x, x0)
    for c in ctxs:
        c.close()
