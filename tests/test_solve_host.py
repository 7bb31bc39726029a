"""Host side of single and batched CG solves on unstructured meshes, on a
stand-in for the CUDA runtime (fake_cudart.cpp): what a solve captures, which
launches of the unstructured patch kernel take an SM's whole shared memory,
and which form of its default shape the structured one is launched with."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import __graft_entry__ as entry
from paper_2510_17785_gb300 import build as b
from paper_2510_17785_gb300 import inputs, pmg

WARPS, TEAM = 64, 128                  # threads per CTA of the 2D FP32 shapes, degrees 5 to 8

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """The whole library on the stand-in, loaded by the binding."""
    entry.build()
    so = str(tmp_path_factory.mktemp("fake") / "pmg_on_fake.so")
    objs = [os.path.join(b.BUILD, os.path.basename(s) + ".o") for s in b._sources()]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic",
                    "-I/usr/local/cuda/include", os.path.join(HERE, "fake_cudart.cpp"), *objs, "-fopenmp", "-o", so],
                   check=True)
    saved, pmg._lib = pmg._lib, None
    yield pmg.load(so)
    pmg._lib = saved


def _context(kind, size, p, sms=152, **opt):
    X, cells, bnd = inputs.unstructured_mesh(kind, size, 13)
    ctx = pmg.Context(sms % 152, precision=pmg.PREC_MIXED, bounds=pmg.BOUNDS_FIXED, fixed_lo=0.25, fixed_hi=2.2, **opt)
    ctx.mesh_upload(X.shape[1], X, cells, p, bnd)
    ctx.setup()
    return ctx


def _solve(fake, ctxs, vecs):
    """Two iterations of every context, together if there are several."""
    K = len(ctxs)
    ptr = (C.c_void_p * K)(*[v.ctypes.data for v in vecs])
    if K == 1:
        rc = fake.pmg_solve_cg(ctxs[0].h, ptr[0], ptr[0], 1e-8, 2, None, None, None)
    else:
        rc = fake.pmg_batch_solve_cg((C.c_void_p * K)(*[c.h for c in ctxs]), K, ptr, ptr, 1e-8, 2, None, None, None)
    assert rc == pmg.PMG_ERR_NOT_CONVERGED          # the stand-in's residual stays at one


def _captures(fake):
    return fake.fake_calls(b"cudaStreamBeginCapture")


@pytest.mark.parametrize("kind,size,p", [("tetsplit", 1, 2), ("tetsplit", 1, 6), ("trisplit2d", 4, 4)])
def test_alternating_solves_capture_no_graph_again(fake, kind, size, p):
    """Single solves and batches of several sizes in turn: a context captures
    its iteration when a solve first needs it, never again."""
    fake.fake_reset()
    ctxs = [_context(kind, size, p) for _ in range(6)]
    vecs = [np.zeros(c.num_dofs(0)[0]) for c in ctxs]
    rounds = []
    for _ in range(3):
        for n in (1, 6, 2, 5, 1):
            _solve(fake, ctxs[:n], vecs[:n])
        rounds.append(_captures(fake))
    assert rounds[0] > 0 and rounds == [rounds[0]] * 3
    for c in ctxs:
        c.close()


def _launches(fake):
    out = np.zeros(1 << 16, np.int32)
    n = fake.fake_patch_launches(C.c_void_p(out.ctypes.data), out.size)
    assert n <= out.size
    return out[:n].reshape(-1, 3)


@pytest.mark.parametrize("sms", [3, 8, 152])
@pytest.mark.parametrize("degrees", [(6,), (6, 6), (6, 2, 4), (6, 2, 4, 2, 4), (6, 6, 6), (6,) * 5, (6, 2) * 5])
def test_whole_sm_launches_by_patches_in_flight(fake, degrees, sms):
    """Degree 6 of this mesh needs 139 KB a patch (one CTA per SM), degrees 2
    and 4 at most 46 KB (always in shared memory).  A degree-6 launch takes its
    SM where it has at most SMs / share patches: share 1 for one or two such
    problems, 2 for four, 4 for eight, however many other problems there are."""
    fake.fake_reset()
    ctxs = [_context("tetsplit", 1, p, sms) for p in degrees]
    vecs = [np.zeros(c.num_dofs(0)[0]) for c in ctxs]
    colours = np.bincount(ctxs[0].get_colours(0))
    _launches(fake)
    _solve(fake, ctxs, vecs)
    share = {1: 1, 2: 1, 3: 2, 5: 4}[degrees.count(6)]
    got = _launches(fake)
    assert len(got) == 2 * len(colours) * len(degrees)         # pre- and post-sweep, captured once
    whole = got[got[:, 2] > 100 * 1024]
    assert sorted(whole[:, 0]) == sorted([n for n in colours if n <= sms // share] * 2 * degrees.count(6))
    # a sweep outside a batch counts on all SMs
    u = vecs[0].ctypes.data
    assert fake.pmg_patch_smooth(ctxs[0].h, 0, u, u, 1, 0, None) == pmg.PMG_OK
    assert [s > 100 * 1024 for _, _, s in _launches(fake)] == [n <= sms for n in colours]
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("dim,p,precision,smoother,opt,sms,threads", [
    # tabulated solves of every degree and level rule, with few and with many patches per SM
    *[(2, p, 1, 0, dict(dense_local=2, level_rule=r), 152, TEAM) for p in (5, 6, 7, 8) for r in (0, 1)],
    *[(2, p, 1, 0, dict(dense_local=2), 1, TEAM if p > 6 else WARPS) for p in (5, 8)],
    *[(2, p, 1, s, dict(), 152, WARPS) for p in (5, 6, 7) for s in (0, 1, 2)],
    (2, 8, 1, 0, dict(), 152, WARPS), (2, 8, 1, 1, dict(), 152, TEAM), (2, 8, 1, 2, dict(), 152, TEAM),
    (2, 8, 1, 1, dict(), 1, WARPS), (2, 8, 1, 2, dict(), 1, WARPS), (2, 8, 1, 0, dict(level_rule=1), 152, WARPS),
    # 25 patches a colour: 2 to 8 per SM, 8 to 16 per SM
    (2, 7, 1, 2, dict(), 5, TEAM), (2, 7, 1, 2, dict(), 2, WARPS), (2, 5, 1, 2, dict(), 2, TEAM),
    (2, 5, 1, 2, dict(), 1, WARPS),
    # persistent sweeps
    (2, 3, 1, 0, dict(persistent=2), 152, 64), (2, 3, 1, 0, dict(persistent=2), 1, 128),
    *[(2, p, 1, 0, dict(persistent=2), 152, WARPS if p == 6 else TEAM) for p in (5, 6, 7, 8)],
    (2, 8, 1, 0, dict(persistent=2), 5, WARPS),
    # 3D degree 2: FP32 always warps, FP64 by waves (64 patches a colour)
    (3, 2, 1, 0, dict(persistent=2), 152, 64), (3, 2, 1, 0, dict(dense_local=2), 2, 64),
    (3, 2, 0, 0, dict(), 152, 128), (3, 2, 0, 0, dict(), 11, 128), (3, 2, 0, 0, dict(), 9, 256),
    (3, 2, 0, 0, dict(), 6, 128), (3, 2, 0, 2, dict(), 11, 128), (3, 2, 0, 2, dict(), 6, 256),
    (3, 2, 0, 0, dict(persistent=2), 6, 256)])
def test_form_of_the_default_shape(fake, dim, p, precision, smoother, opt, sms, threads):
    """Sweeps of 11^2 cells (25 patches in the first colour) and 9^3 cells (64):
    threads per CTA of that colour's launch."""
    N = 11 if dim == 2 else 9
    x = np.stack(np.meshgrid(*[np.arange(N + 1.0)] * dim, indexing="ij")[::-1], axis=-1).reshape(-1, dim)
    fake.fake_reset()
    ctx = pmg.Context(sms % 152, precision=precision, bounds=pmg.BOUNDS_FIXED, fixed_lo=0.25, fixed_hi=2.2, autotune=0,
                      smoother=smoother, **{"persistent": 0, "dense_local": 0, **opt})
    ctx.mesh_structured(dim, N, p, 1, x, np.ones(N ** dim))
    ctx.setup()
    v = np.zeros(ctx.num_dofs(0)[0])
    _launches(fake)
    assert fake.pmg_patch_smooth(ctx.h, 0, v.ctypes.data, v.ctypes.data, 1, 0, None) == pmg.PMG_OK
    assert _launches(fake)[0][1] == threads
    ctx.close()
