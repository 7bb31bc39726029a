"""Host side of the interval-network training (pmg_mlp_train, pmg_mlp_grad) on
a stand-in for the CUDA runtime (fake_cudart.cpp) that puts every copy and
launch off to the next synchronisation: what the training asks of the device
must not depend on an asynchronous copy being over when its call returns."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import __graft_entry__ as entry
from paper_2510_17785_gb300 import build as b
from paper_2510_17785_gb300 import pmg

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    entry.build()
    so = str(tmp_path_factory.mktemp("fake") / "mlp_on_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I/usr/local/cuda/include",
                    os.path.join(HERE, "fake_cudart.cpp"), os.path.join(b.BUILD, "mlp.cu.o"), "-o", so], check=True)
    return C.CDLL(so)


def _train(fake, n, batch, epochs, seed, hist=True):
    o = pmg.train_options(epochs=epochs, batch=batch, seed=seed)
    buf = np.zeros(max(pmg.MLP_NPARAM, 18 * n), np.float32)     # the stand-in's kernels read none of it
    loss = np.zeros(epochs, np.float32)
    p = C.c_void_p(buf.ctypes.data)
    return fake.pmg_mlp_train(0, p, p, p, p, C.c_int64(n), C.byref(o), C.c_void_p(loss.ctypes.data if hist else None))


@pytest.mark.parametrize("n,batch,epochs,hist", [(20, 4, 5, True), (20, 4, 5, False), (23, 5, 4, True),
                                                 (9, 16, 3, True), (70000, 1, 3, True), (16, 16, 1, False)])
def test_every_epoch_trains_on_its_own_order(fake, n, batch, epochs, hist):
    """The order of an epoch reaches the device as drawn, however late its copy
    reads the host's memory: with losses read back or not, within one read-back
    of the losses (65,536 steps) and across."""
    fake.fake_reset()
    assert _train(fake, n, batch, epochs, 3, hist) == pmg.PMG_OK
    expect = np.zeros((epochs, n), np.int32)
    fake.fake_expected_orders(C.c_ulonglong(3), n, epochs, C.c_void_p(expect.ctypes.data))
    bb, nb = min(batch, n), n // min(batch, n)
    got = np.zeros(epochs * nb * (bb + 1), np.int32)
    assert fake.fake_orders(C.c_void_p(got.ctypes.data), got.size) == got.size
    got = got.reshape(epochs, nb, bb + 1)
    assert (got[:, :, 0] == bb).all()
    assert np.array_equal(got[:, :, 1:].reshape(epochs, nb * bb), expect[:, :nb * bb])


@pytest.mark.parametrize("function,call", [("cudaMemsetAsync", 1), ("cudaMemcpyAsync", 1), ("cudaMemcpyAsync", 2),
                                           ("launch", 1), ("launch", 2), ("launch", 11)])
def test_training_reports_a_call_that_failed(fake, function, call):
    """Two epochs of five steps: the fill, a copy or a launch that the runtime
    refuses ends the training with PMG_ERR_CUDA, not with PMG_OK."""
    fake.fake_reset()
    fake.fake_fail(function.encode(), call)
    assert _train(fake, 20, 4, 2, 3) == pmg.PMG_ERR_CUDA


@pytest.mark.parametrize("call", [1, 2])
def test_gradient_reports_a_launch_that_failed(fake, call):
    buf = np.zeros(pmg.MLP_NPARAM, np.float32)
    p = C.c_void_p(buf.ctypes.data)
    fake.fake_reset()
    fake.fake_fail(b"launch", call)
    assert fake.pmg_mlp_grad(0, p, p, p, p, 4, C.c_float(4.0), p, p, None) == pmg.PMG_ERR_CUDA
    assert fake.pmg_mlp_grad(0, p, p, p, p, 4, C.c_float(4.0), p, p, None) == pmg.PMG_OK   # a pending error is not its own
