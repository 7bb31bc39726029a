"""Launches of the unstructured patch kernel from several host threads, on a
stand-in for the CUDA runtime (fake_cudart.cpp): contexts may be used by
different threads at once, and the shared memory of a launch varies."""
import ctypes as C
import os
import subprocess
import threading

import pytest

import __graft_entry__ as entry
from paper_2510_17785_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))
SWEEP, LOCAL = 0, 1                    # MODE_SWEEP, MODE_LOCAL


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    entry.build()
    d = tmp_path_factory.mktemp("fake")
    so = str(d / "upatch_on_fake.so")
    subprocess.run([b._nvcc(), *b.ARCH, "-std=c++17", "-O0", "-Xcompiler", "-fPIC", "-c",
                    os.path.join(HERE, "fake_upatch.cu"), "-o", str(d / "fake_upatch.o")], check=True)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic",
                    "-I/usr/local/cuda/include", os.path.join(HERE, "fake_cudart.cpp"), str(d / "fake_upatch.o"),
                    os.path.join(b.BUILD, "umesh_k2.cu.o"), os.path.join(b.BUILD, "basis.cpp.o"), "-fopenmp",
                    "-o", so], check=True)
    lib = C.CDLL(so)
    lib.launch_upatch.argtypes = [C.c_int, C.c_size_t]
    lib.fake_overtake.argtypes = [C.c_size_t]
    return lib


@pytest.mark.parametrize("mode", [SWEEP, LOCAL])
def test_threads_do_not_lower_each_others_limit(fake, mode):
    """Two threads launch with a small and a large workspace slice; the small
    one's limit is set last.  Neither these nor later large launches are refused."""
    fake.fake_reset()
    small, large = 64 * 1024, 160 * 1024
    fake.fake_overtake(128 * 1024)
    got = {}
    ts = [threading.Thread(target=lambda s=s: got.__setitem__(s, fake.launch_upatch(mode, s))) for s in (small, large)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    fake.fake_overtake(0)
    assert got == {small: 0, large: 0}
    assert [fake.launch_upatch(mode, s) for s in (large, 0, large)] == [0, 0, 0]


def test_a_slice_beyond_the_sm_is_refused(fake):
    fake.fake_reset()
    assert fake.launch_upatch(SWEEP, 227 * 1024) == 1          # ST_ARG: CTA and slice exceed 227 KB
    assert fake.launch_upatch(SWEEP, 200 * 1024) == 0
